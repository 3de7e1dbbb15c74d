// Completion of the slices from their sampled entries and the factorised render.
//
//  * Omega build: per slice, the observed entries are placed through two occupancy
//    bitmaps (the position of an entry is a popcount of the bits before it, so the
//    layout is deterministic) into a sliced layout per side for the lane-group ALS
//    (lines sorted by entry count, warp tasks of 32 lanes, streams interleaved by
//    chunks of 4) and, for ranks above 16, into CSR / CSC.
//  * Masked ALS (the completion M_s ~= U_s V_s^T at rank r; Sec. 5 uses the factor
//    form M = X Y): up to rank 16 a line (a row of U or of V) belongs to a group of
//    2^g lanes sized by its entry count; each lane accumulates its part of the Gram
//    and right-hand side in registers from the slice's factor rows staged in shared
//    memory, the group reduces with shuffles and its first lane adds the ridge
//    lam_rel tr(G) / r, factors by Cholesky in float32 and solves; lines whose pivots
//    spread beyond 1e6 are solved again in float64.  The half-step kernel is
//    persistent: each CTA takes an equal share of all slices' warp tasks.  Above
//    rank 16 a warp sums the Grams of two lines, a block of the triangle a lane, and half
//    a warp factors and solves each.
//    The rank may differ per slice (factor rows keep the stride of the largest).
//  * Render (Sec. 3 step 5): t_s = V_s^T w, pixel = max(0, u_i . t_s).
#include <math.h>

#include <algorithm>
#include <vector>

#include "lt_internal.cuh"
#include "lt_omega.cuh"
#include "lt_als_common.cuh"
#include "lt_als_tc.cuh"

using namespace ltk;

namespace {



// Group-size classes of a line: class g gives a line of L entries G = 2^g lanes, so
// that a lane takes at most about `lane_entries` of them (g = 0..5; a tuning value).
constexpr int kClasses = 6;

__host__ __device__ inline int line_class(int len, int lane_entries) {
    int g = 0;
    while (g < kClasses - 1 && len > (lane_entries << g)) ++g;
    return g;
}

// Omega build in six passes over the whole GPU (slice = blockIdx.y):
//  1. clear the used words of the row-major bitmap;  2. set the bit of every entry and
//  sum the values (one partial per block, fixed order);  3. the column-major bitmap by
//  32 x 32 bit transposes (a second scattered atomic per entry costs more);  4. one warp
//  per row (column): popcount of each bitmap word, warp scan into the per-word prefix,
//  line count;  5. one block per slice: exclusive scan of the line counts into row /
//  column pointers, mean value;  6. one thread per entry: slot = pointer + bits before.
// A word and its prefix sit side by side, so that an entry finds its index in a line
// with one 8-byte load.
__global__ void k_om_clear(lt_frame F, lt_samples smp, Omega om) {
    const int s = blockIdx.y;
    const int ms = F.slice_off[s + 1] - F.slice_off[s], ns = smp.ncol[s];
    const int64_t nbm = (int64_t)ms * ((ns + 31) >> 5);
    uint2* wr = om.wr + (int64_t)s * om.bm_stride;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nbm; i += (int64_t)gridDim.x * blockDim.x)
        wr[i] = make_uint2(0u, 0u);
}

__global__ void k_om_bits(lt_frame F, lt_samples smp, Omega om, int32_t* status) {
    const int s = blockIdx.y;
    const int ms = F.slice_off[s + 1] - F.slice_off[s], ns = smp.ncol[s], ne = smp.cnt[s];
    const int W = (ns + 31) >> 5;
    uint2* wr = om.wr + (int64_t)s * om.bm_stride;
    const uint32_t* key = smp.key + smp.off[s];
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += gridDim.x * blockDim.x) {
        const uint32_t k = key[e];
        const int r = (int)(k >> 16), c = (int)(k & 0xffffu);
        if (r >= ms || c >= ns) {
            latch(status, LT_EINVAL);
            continue;
        }
        atomicOr(&wr[(int64_t)r * W + (c >> 5)].y, 1u << (c & 31));
    }
}

// Part p of the sum of a slice's values: thread t of kOmParts blocks of 256 adds every
// 256 kOmParts-th value, then the block adds its threads, in a fixed order.  (Entries out
// of range are not in the layout nor in its sum.)
constexpr int kOmParts = 8;

__device__ __forceinline__ void om_sum(const lt_samples& smp, int s, int ms, int ns, int p, float* __restrict__ part) {
    __shared__ float red[32];
    const int ne = smp.cnt[s];
    const uint32_t* key = smp.key + smp.off[s];
    const float* val = smp.val + smp.off[s];
    float sum = 0.f;
    for (int e0 = p * 256 + threadIdx.x; e0 < ne; e0 += 8 * kOmParts * 256) {
        uint32_t k[8];
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {  // the loads of eight steps in flight together
            const int e = min(e0 + u * kOmParts * 256, ne - 1);
            k[u] = __ldg(key + e);
            v[u] = __ldg(val + e);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (e0 + u * kOmParts * 256 < ne && (int)(k[u] >> 16) < ms && (int)(k[u] & 0xffffu) < ns) sum += v[u];
    }
    sum = warp_sum(sum);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[(int64_t)s * kOmParts + p] = t;
    }
}

// one warp per 32 rows: lane i holds a word of row i; bit b of the 32 words is word b's
// transpose, which lane b writes.  The first kOmParts blocks of a slice also sum its values.
__global__ void __launch_bounds__(256) k_om_transpose(lt_frame F, lt_samples smp, Omega om, float* __restrict__ part) {
    const int s = blockIdx.y;
    const int ms = F.slice_off[s + 1] - F.slice_off[s], ns = smp.ncol[s];
    if (blockIdx.x < kOmParts) om_sum(smp, s, ms, ns, blockIdx.x, part);
    const int W = (ns + 31) >> 5, WT = (ms + 31) >> 5;
    const uint2* wr = om.wr + (int64_t)s * om.bm_stride;
    uint2* wc = om.wc + (int64_t)s * om.bt_stride;
    const int lane = threadIdx.x & 31;
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    for (int64_t t = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); t < (int64_t)W * WT; t += nwarps) {
        const int rb = (int)(t / W), cw = (int)(t % W), r = 32 * rb + lane, c = 32 * cw + lane;
        const uint32_t w = r < ms ? wr[(int64_t)r * W + cw].y : 0u;
        uint32_t mine = 0u;
#pragma unroll
        for (int b = 0; b < 32; ++b) {
            const uint32_t x = __ballot_sync(0xffffffffu, (w >> b) & 1u);
            if (lane == b) mine = x;
        }
        if (c < ns) wc[(int64_t)c * WT + rb] = make_uint2(0u, mine);
    }
}

// one warp per line: the word prefixes of one bitmap row, the line's count into cnt_out, and
// the plain words into `bits` where they are wanted
__device__ __forceinline__ void om_line_words(uint2* __restrict__ words, uint32_t* __restrict__ bits, int nw,
                                              int32_t* cnt_out) {
    const int lane = threadIdx.x & 31;
    int carry = 0;
    for (int w0 = 0; w0 < nw; w0 += 32) {
        const int w = w0 + lane;
        const uint32_t b = w < nw ? words[w].y : 0u;
        const int c = __popc(b);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (w < nw) {
            words[w].x = (uint32_t)(carry + incl - c);
            if (bits) bits[w] = b;
        }
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) *cnt_out = carry;
}

__global__ void k_om_lines(lt_frame F, lt_samples smp, Omega om) {
    const int s = blockIdx.y;
    const int row0 = F.slice_off[s], ms = F.slice_off[s + 1] - row0, ns = smp.ncol[s];
    const int W = (ns + 31) >> 5, WT = (ms + 31) >> 5;
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    const int gw = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    for (int l = gw; l < ms + ns; l += nwarps) {
        if (l < ms) {
            const int64_t o = (int64_t)s * om.bm_stride + (int64_t)l * W;
            om_line_words(om.wr + o, om.bm ? om.bm + o : nullptr, W, om.rp + row0 + s + l + 1);
        } else {
            const int c = l - ms;
            const int64_t o = (int64_t)s * om.bt_stride + (int64_t)c * WT;
            om_line_words(om.wc + o, om.bt ? om.bt + o : nullptr, WT, om.cp + (int64_t)s * (F.C + 1) + c + 1);
        }
    }
}

// in place: x[0] = 0, x[1..n] counts -> exclusive prefix x[0..n]
__device__ void om_scan_counts(int32_t* x, int n, int32_t* ws) {
    int carry = 0;
    for (int i0 = 0; i0 < n; i0 += blockDim.x) {
        const int i = i0 + threadIdx.x;
        const int c = i < n ? x[i + 1] : 0;
        int tot;
        const int pre = block_exclusive_scan<int>(c, ws, &tot);
        if (i < n) x[i + 1] = carry + pre + c;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) x[0] = 0;
}

// ord[0..n) = lines by decreasing count (ties by index), from the counts ptr[1..n]
// before they are scanned; a block-wide bitonic sort in shared memory, or the
// identity when n exceeds kOrdMax.
constexpr int kOrdMax = 4096;

// cls[0..7): first sorted line of each class, largest class first (cls[kClasses - 1 - g]
// for class g) and cls[8..15): the first warp task of each, a class-g task covering
// 32 / 2^g lines; cls[6] and cls[14] are the totals.
__device__ void om_classes(const int32_t* __restrict__ cnt1, int n, const int32_t* __restrict__ ord, bool sorted,
                           int lane_entries, int32_t* __restrict__ cls) {
    __shared__ int32_t num[kClasses];
    if (threadIdx.x < kClasses) num[threadIdx.x] = 0;
    __syncthreads();
    if (sorted)
        for (int i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&num[line_class(cnt1[ord[i]], lane_entries)], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!sorted) num[0] = n;  // unsorted: every line on one lane
        int line = 0, task = 0;
        for (int k = 0; k < kClasses; ++k) {  // k-th run in the order = class kClasses - 1 - k
            const int g = kClasses - 1 - k;
            cls[k] = line;
            cls[8 + k] = task;
            line += num[g];
            task += (num[g] + (32 >> g) - 1) / (32 >> g);
        }
        cls[kClasses] = line;
        cls[8 + kClasses] = task;
    }
    __syncthreads();
}

__device__ void om_order(const int32_t* __restrict__ cnt1, int n, int32_t* __restrict__ ord,
                         unsigned long long* key) {
    if (n > kOrdMax) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) ord[i] = i;
        __syncthreads();
        return;
    }
    int N = 1;
    while (N < n) N <<= 1;
    for (int i = threadIdx.x; i < N; i += blockDim.x)
        key[i] = i < n ? ((unsigned long long)(0xffffffffu - (uint32_t)cnt1[i]) << 32) | (uint32_t)i : ~0ull;
    __syncthreads();
    for (int k = 2; k <= N; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < N; i += blockDim.x) {
                const int l = i ^ j;
                if (l > i) {
                    const unsigned long long a = key[i], b = key[l];
                    if ((a > b) == ((i & k) == 0)) {
                        key[i] = b;
                        key[l] = a;
                    }
                }
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < n; i += blockDim.x) ord[i] = (int32_t)(key[i] & 0xffffffffu);
    __syncthreads();
}

// run of the sorted order that holds position li (classes largest first)
__device__ __forceinline__ int om_run(const int32_t* cls, int li) {
    int k = 0;
    while (k + 1 < kClasses && li >= cls[k + 1]) ++k;
    return k;
}

// pos[ord[i]] = i, and the sliced layout of one side: a class-g task covers
// P = 32 / 2^g lines, its lanes hold ceil(count / 2^g) slots at most, so the task
// takes 32 x (that maximum over its lines, rounded up to 4) slots; tb[t] = the
// slots before task t (a multiple of 128).
// The region size goes to *size.
__device__ void om_tasks(const int32_t* __restrict__ cnt1, int n, const int32_t* __restrict__ ord,
                         const int32_t* __restrict__ cls, int32_t* __restrict__ pos, int32_t* __restrict__ tb,
                         int64_t* size, int32_t* ws) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) pos[ord[i]] = i;
    const int T = cls[8 + kClasses];
    int carry = 0;
    for (int t0 = 0; t0 < T; t0 += blockDim.x) {
        const int t = t0 + threadIdx.x;
        int w = 0;
        if (t < T) {
            int k = 0;
            while (k + 1 < kClasses && t >= cls[8 + k + 1]) ++k;
            const int g = kClasses - 1 - k, G = 1 << g, P = 32 >> g;
            const int li0 = cls[k] + (t - cls[8 + k]) * P, li1 = min(li0 + P, cls[k + 1]);
            int kk = 0;
            for (int li = li0; li < li1; ++li) kk = max(kk, (cnt1[ord[li]] + G - 1) >> g);
            w = 32 * ((kk + 3) & ~3);
        }
        int tot;
        const int pre = block_exclusive_scan<int>(w, ws, &tot);
        if (t < T) tb[t] = carry + pre;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *size = carry;
    __syncthreads();
}

__global__ void k_om_scan(lt_frame F, lt_samples smp, Omega om, const float* __restrict__ part, int nparts) {
    __shared__ int32_t ws[32];
    __shared__ unsigned long long key[kOrdMax];
    const int s = blockIdx.x;
    const int row0 = F.slice_off[s], ms = F.slice_off[s + 1] - row0, ns = smp.ncol[s], ne = smp.cnt[s];
    const int32_t* rc1 = om.rp + row0 + s + 1;                // row counts (before the scan)
    const int32_t* cc1 = om.cp + (int64_t)s * (F.C + 1) + 1;  // column counts
    int32_t* rord = om.rord + row0;
    int32_t* cord = om.cord + (int64_t)s * F.C;
    int32_t* rcls = om.rcls + (int64_t)s * 16;
    int32_t* ccls = om.ccls + (int64_t)s * 16;
    if (blockIdx.y == 0) {
        om_order(rc1, ms, rord, key);
        om_classes(rc1, ms, rord, ms <= kOrdMax, om.lane_entries, rcls);
        if (om.sell)
            om_tasks(rc1, ms, rord, rcls, om.rpos + row0, om.rtb + (int64_t)s * om.tcap, om.rbase + s + 1, ws);
        om_scan_counts(om.rp + row0 + s, ms, ws);
        return;
    }
    om_order(cc1, ns, cord, key);
    om_classes(cc1, ns, cord, ns <= kOrdMax, om.lane_entries, ccls);
    if (om.sell)
        om_tasks(cc1, ns, cord, ccls, om.cpos + (int64_t)s * F.C, om.ctb + (int64_t)s * om.tcap, om.cbase + s + 1, ws);
    om_scan_counts(om.cp + (int64_t)s * (F.C + 1), ns, ws);
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int q = 0; q < nparts; ++q) t += part[(int64_t)s * nparts + q];
        om.mu[s] = ne > 0 ? t / (float)ne : 0.f;
    }
}

// region starts of the sliced layouts: in place, x[1..S] sizes -> x[0..S] prefix;
// a total beyond the capacity latches LT_ELIMIT (the scatter then skips slots past it)
// (with the work before each slice: slots and kTaskCost per warp task of the slices whose
// rank the lane-group kernel has)
constexpr int kTaskCost = 512;   // slots worth a task's reduction and Cholesky (32 lanes x 16 entries)

__global__ void k_om_sellpfx(int S, Omega om, const int32_t* __restrict__ rk, int R, int32_t* status) {
    __shared__ int64_t ws[32];
    for (int side = 0; side < 2; ++side) {
        int64_t* x = side == 0 ? om.rbase : om.cbase;
        int64_t carry = 0;
        for (int i0 = 0; i0 < S; i0 += blockDim.x) {
            const int i = i0 + threadIdx.x;
            const int64_t c = i < S ? x[i + 1] : 0;
            int64_t tot;
            const int64_t pre = block_exclusive_scan<int64_t>(c, ws, &tot);
            if (i < S) x[i + 1] = carry + pre + c;
            carry += tot;
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            x[0] = 0;
            if (carry > om.sell_cap) latch(status, LT_ELIMIT);
        }
        __syncthreads();
        int64_t* wk = side == 0 ? om.rwk : om.cwk;
        const int32_t* cls = side == 0 ? om.rcls : om.ccls;
        int64_t work = 0;
        for (int i0 = 0; i0 < S; i0 += blockDim.x) {
            const int i = i0 + threadIdx.x;
            int64_t c = 0;
            if (i < S && slice_rank(rk, i, R) <= 16)
                c = x[i + 1] - x[i] + (int64_t)kTaskCost * cls[16 * i + 8 + kClasses];
            int64_t tot;
            const int64_t pre = block_exclusive_scan<int64_t>(c, ws, &tot);
            if (i < S) wk[i] = work + pre;
            work += tot;
            __syncthreads();
        }
        if (threadIdx.x == 0) wk[S] = work;
        __syncthreads();
    }
}

// slot, within the slice's region, of entry k of the line at sorted position li
__device__ __forceinline__ int64_t sell_slot(const int32_t* __restrict__ cls, const int32_t* __restrict__ tb, int li,
                                             int k) {
    const int run = om_run(cls, li);
    const int g = kClasses - 1 - run, P = 32 >> g;
    const int rel = li - cls[run];
    const int t = cls[8 + run] + rel / P, lane = (rel % P) * (1 << g) + (k & ((1 << g) - 1));
    const int kk = k >> g;
    return (int64_t)tb[t] + 128 * (int64_t)(kk >> 2) + 4 * lane + (kk & 3);
}

__global__ void k_om_scatter(lt_frame F, lt_samples smp, Omega om) {
    const int s = blockIdx.y;
    const int row0 = F.slice_off[s], ms = F.slice_off[s + 1] - row0, ns = smp.ncol[s], ne = smp.cnt[s];
    const int W = (ns + 31) >> 5, WT = (ms + 31) >> 5;
    const uint2* wr = om.wr + (int64_t)s * om.bm_stride;
    const uint2* wc = om.wc + (int64_t)s * om.bt_stride;
    const int32_t* rp = om.rp + row0 + s;
    const int32_t* cp = om.cp + (int64_t)s * (F.C + 1);
    const int64_t o = smp.off[s];
    const uint32_t* key = smp.key + o;
    const float* val = smp.val + o;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += gridDim.x * blockDim.x) {
        const uint32_t k = key[e];
        const int r = (int)(k >> 16), c = (int)(k & 0xffffu);
        if (r >= ms || c >= ns) continue;
        const int64_t iw = (int64_t)r * W + (c >> 5), jw = (int64_t)c * WT + (r >> 5);
        const uint2 a = __ldg(wr + iw), b = __ldg(wc + jw);
        const int kr = (int)a.x + __popc(a.y & ((1u << (c & 31)) - 1u));  // index in its row
        const int kc = (int)b.x + __popc(b.y & ((1u << (r & 31)) - 1u));  // index in its column
        const float v = val[e];
        if (om.csr) {
            om.cidx[o + rp[r] + kr] = (uint16_t)c;
            om.cval[o + rp[r] + kr] = v;
            om.ridx[o + cp[c] + kc] = (uint16_t)r;
            om.rval[o + cp[c] + kc] = v;
            om.r2c[o + rp[r] + kr] = cp[c] + kc;
        }
        if (om.sell) {
            const int64_t pr = sell_slot(om.rcls + (int64_t)s * 16, om.rtb + (int64_t)s * om.tcap,
                                         om.rpos[row0 + r], kr) + om.rbase[s];
            const int64_t pc = sell_slot(om.ccls + (int64_t)s * 16, om.ctb + (int64_t)s * om.tcap,
                                         om.cpos[(int64_t)s * F.C + c], kc) + om.cbase[s];
            if (pr < om.sell_cap) {
                om.sidx_r[pr] = (uint16_t)c;
                om.sval_r[pr] = v;
            }
            if (pc < om.sell_cap) {
                om.sidx_c[pc] = (uint16_t)r;
                om.sval_c[pc] = v;
            }
        }
    }
}

__global__ void k_line_prefix(const lt_samples smp, int S, int64_t* pfx) {
    __shared__ int64_t ws[32];
    int64_t carry = 0;
    for (int c0 = 0; c0 < S; c0 += blockDim.x) {
        const int s = c0 + threadIdx.x;
        const int64_t x = s < S ? (int64_t)smp.ncol[s] : 0;
        int64_t tot;
        const int64_t pre = block_exclusive_scan<int64_t>(x, ws, &tot);
        if (s < S) pfx[s] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) pfx[S] = carry;
}

__global__ void k_als_init(lt_frame F, lt_samples smp, Omega om, int R, const int32_t* __restrict__ rk, SeedRef sr,
                           float* __restrict__ V) {
    const int s = blockIdx.y;
    const uint64_t seed = sr.get();
    const int ns = smp.ncol[s];
    const int r = slice_rank(rk, s, R);  // the slice's rank; components r .. R-1 are 0
    const float amp = sqrtf(fmaxf(om.mu[s], 0.f) / (float)r);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ns * R; i += gridDim.x * blockDim.x) {
        const int j = i / R, k = i % R;
        if (k >= r) {
            V[((int64_t)s * F.C + j) * R + k] = 0.f;
            continue;
        }
        const uint32_t w = philox((uint32_t)k, (uint32_t)j, slice_key(F.slice_id, s), kTagAlsInit, seed).x;
        V[((int64_t)s * F.C + j) * R + k] = amp * (0.5f + (float)w * 2.3283064365386963e-10f);
    }
}

// ---- Two lines by one warp (ranks above 16) -----------------------------------
// For one line (a row of U or of V) with observed entries e and factor rows x_e,
// G = sum_e x_e x_e^T and b = sum_e a_e x_e.  The whole warp sums the Gram of one line after
// the other, then half a warp solves each.  The entries are taken 32 at a time: eight lanes
// copy one factor row (128 contiguous bytes, so a copy instruction touches 4 lines and not
// 32) into the warp's stage with a_e behind it, and the next 32 rows are on their way
// (cp.async) while these are added.  Rows have stride R; components at or beyond the rank
// are zero.  RB = 3 (ranks up to 24) or 4: only the first 8 RB components are copied, added
// and solved for.
constexpr int kWarpRow = 36;               // floats between staged rows: 32 and a_e
constexpr int kWarpStage = 32 * kWarpRow;  // floats of one stage: 32 rows
constexpr int kWarpCol = 36;               // stride of a column of L (16-byte aligned)
constexpr int kWarpGram = 36 * 16 + 32;    // a line's Gram in 4 x 4 blocks, and b

__device__ __forceinline__ void copy16(float* dst, const float* src, bool full) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = full ? 16 : 0;  // 0: the 16 bytes are zeroed and nothing is read
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// starts the copies of rows idx[e0 ..] (at most 32, the rest zero) into st
__device__ __forceinline__ void stage_entries(int len, int e0, int j, const float* __restrict__ src, int R, int rmax,
                                              bool vec, float* st) {
    const int lane = threadIdx.x & 31, c = lane & 7;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int q = 4 * i + (lane >> 3);
        const int jq = __shfl_sync(0xffffffffu, j, q);
        if (4 * c >= rmax) continue;
        const bool live = e0 + q < len && 4 * c < R;
        const float* p = src + (live ? (int64_t)jq * R + 4 * c : 0);
        float* d = st + q * kWarpRow + 4 * c;
        if (vec) {
            copy16(d, p, live);
        } else {  // R not a multiple of 4, or rows not on 16 bytes
#pragma unroll
            for (int k = 0; k < 4; ++k) d[k] = live && 4 * c + k < R ? __ldg(p + k) : 0.f;
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// A line's Gram and b by one warp into `out`.  A lane holds a tile of TR x 4: RB = 3 the 21
// 4 x 4 blocks on or below the diagonal and 6 tiles of b (a tile whose columns are a_e and
// what lies behind it), RB = 4 the 20 tiles of 8 x 4 that reach the diagonal or below and 4
// of b.  A row and all of its partners a lane instead read 33 floats per entry from shared
// memory where a tile reads 8 or 12, and added both triangles.  j, av: index and value of
// the lane's entry among the first 32.
template <int RB>
__device__ __forceinline__ void gram_warp(int len, const uint16_t* __restrict__ idx, const float* __restrict__ val,
                                          int j, float av, const float* __restrict__ src, int R, float* st0, float* out) {
    constexpr int TR = RB == 3 ? 4 : 8, kTiles = RB == 3 ? 21 : 20, kVec = 8 * RB / TR;
    const int lane = threadIdx.x & 31;
    const bool vec = (R & 3) == 0 && ((uintptr_t)src & 15) == 0;
    int tr = 0, tc = 0;  // tile rows TR tr .., columns 4 tc ..
    if (lane < kTiles) {
        if (RB == 3) {
            while ((tr + 1) * (tr + 2) / 2 <= lane) ++tr;
            tc = lane - tr * (tr + 1) / 2;
        } else {
            while ((tr + 1) * (tr + 2) <= lane) ++tr;
            tc = lane - tr * (tr + 1);
        }
    } else if (lane < kTiles + kVec) {
        tr = lane - kTiles;
        tc = 2 * RB;
    }
    F32x2 g2[TR / 2][4];  // two rows of the tile each
#pragma unroll
    for (int u = 0; u < TR / 2; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) g2[u][v] = 0ull;
    __syncwarp();  // the stage is free
    if (len > 0) {
        stage_entries(len, 0, j, src, R, 8 * RB, vec, st0);
        st0[lane * kWarpRow + 8 * RB] = av;
    }
    for (int e0 = 0, h = 0; e0 < len; e0 += 32, h ^= 1) {
        const float* st = st0 + h * kWarpStage;
        if (e0 + 32 < len) {  // warp-uniform
            const int e = e0 + 32 + lane;
            j = e < len ? (int)idx[e] : 0;
            av = e < len ? val[e] : 0.f;
            float* nx = st0 + (h ^ 1) * kWarpStage;
            stage_entries(len, e0 + 32, j, src, R, 8 * RB, vec, nx);
            nx[lane * kWarpRow + 8 * RB] = av;
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        const int n = min(32, len - e0);
        const float* px = st + TR * tr;
        const float* py = st + 4 * tc;
#pragma unroll 4
        for (int q = 0; q < n; ++q) {
            const float4 y = *reinterpret_cast<const float4*>(py + q * kWarpRow);
            const F32x2 y2[4] = {pack2(y.x, y.x), pack2(y.y, y.y), pack2(y.z, y.z), pack2(y.w, y.w)};
#pragma unroll
            for (int u = 0; u < TR / 4; ++u) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(px + q * kWarpRow + 4 * u);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    g2[2 * u][v] = fma2(x.x, y2[v], g2[2 * u][v]);
                    g2[2 * u + 1][v] = fma2(x.y, y2[v], g2[2 * u + 1][v]);
                }
            }
        }
        __syncwarp();  // the stage after next is this one
    }
#pragma unroll
    for (int u = 0; u < TR / 2; ++u) {
        float lo[4], hi[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) unpack2(g2[u][v], lo[v], hi[v]);
        const int row = TR * tr + 2 * u, i = row >> 2;
        if (lane < kTiles) {
            if (tc <= i) {
                float* blk = out + 16 * (i * (i + 1) / 2 + tc) + 4 * (row & 3);
                *reinterpret_cast<float4*>(blk) = make_float4(lo[0], lo[1], lo[2], lo[3]);
                *reinterpret_cast<float4*>(blk + 4) = make_float4(hi[0], hi[1], hi[2], hi[3]);
            }
        } else if (lane < kTiles + kVec) {
            out[36 * 16 + row] = lo[0];
            out[36 * 16 + row + 1] = hi[0];
        }
    }
}

// Eight columns (8 P ..) of the Cholesky of half a warp's line, and the forward
// substitution with them.  Lane l of the half has rows l (columns up to 15) and l + 16.  The
// first register of a row is the current column and the registers move
// down by one per column, so that one loop body serves the eight (all of them unrolled are
// more code than the instruction caches hold: 41% of the stall cycles).  A column of L
// goes through shared memory (then 16-byte broadcast loads, a quarter as many
// instructions as a shuffle per row) and stays there for the backward substitution.
// Entries above the diagonal are not used, so every lane updates its whole row.
template <int P, int RB>
__device__ __forceinline__ void chol_block32(float (&a1)[16], float (&a2)[8 * RB], float& y1, float& y2, int l, int r,
                                             bool& ok, float& dmin, float& dmax, float& inv1, float& inv2, float* Lc) {
    constexpr int W = 8 * (RB - P), W1 = 16 - 8 * P;  // columns left at the start of the block
    const unsigned FULL = 0xffffffffu;
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
        const int J = 8 * P + t;
        const float djj = __shfl_sync(FULL, P < 2 ? a1[0] : a2[0], J & 15, 16);
        if (J < r) {
            ok &= (djj > 0.f);
            dmin = djj < dmin ? djj : dmin;
            dmax = djj > dmax ? djj : dmax;
        }
        const float dpos = djj > 0.f ? djj : 1.f;
        const float ljj = sqrtf(dpos);
        const float inv = 1.f / ljj;
        float* col = Lc + J * kWarpCol;  // row J + c of the column at col[c]
        float l1 = 0.f, l2 = a2[0] * inv;
        if (P < 2) {
            l1 = l > J ? a1[0] * inv : (l == J ? ljj : 0.f);
            if (l >= J) col[l - J] = l1;
            col[l + 16 - J] = l2;
            if (l == J) inv1 = inv;
        } else {
            l2 = l + 16 > J ? l2 : (l + 16 == J ? ljj : 0.f);
            if (l + 16 >= J) col[l + 16 - J] = l2;
            if (l + 16 == J) inv2 = inv;
        }
        const float yj = __shfl_sync(FULL, P < 2 ? y1 * inv1 : y2 * inv2, J & 15, 16);  // L y = b: y_J is final
        if (P < 2) {
            if (l == J) y1 = yj;
            else if (l > J) y1 = fmaf(-l1, yj, y1);
            y2 = fmaf(-l2, yj, y2);
        } else {
            if (l + 16 == J) y2 = yj;
            else if (l + 16 > J) y2 = fmaf(-l2, yj, y2);
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < W / 4; ++q) {  // (columns past the last hold anything and are never read)
            const float4 c = *reinterpret_cast<const float4*>(col + 4 * q);
            if (q > 0) a2[4 * q - 1] = fmaf(-l2, c.x, a2[4 * q]);
            a2[4 * q] = fmaf(-l2, c.y, a2[4 * q + 1]);
            a2[4 * q + 1] = fmaf(-l2, c.z, a2[4 * q + 2]);
            a2[4 * q + 2] = fmaf(-l2, c.w, a2[4 * q + 3]);
            if (4 * q < W1) {
                if (q > 0) a1[4 * q - 1] = fmaf(-l1, c.x, a1[4 * q]);
                a1[4 * q] = fmaf(-l1, c.y, a1[4 * q + 1]);
                a1[4 * q + 1] = fmaf(-l1, c.z, a1[4 * q + 2]);
                a1[4 * q + 2] = fmaf(-l1, c.w, a1[4 * q + 3]);
            }
        }
    }
}

// Solves (G + ridge) u = b of one line in each half of a warp: `gram` is the half's line
// (gram_warp), lane l of the half receives u_l and u_{l+16}.  Returns false (for the half)
// when the float factorisation is not acceptable (a non-positive pivot, or pivots spread
// by more than 1 / kPivotRatio).  Lc: 32 columns of kWarpCol floats a half; it may overlap
// the Grams.
template <int RB>
__device__ __forceinline__ bool pair_solve32(const float* gram, int len, int r, float lam_rel, float* u1, float* u2,
                                             float* Lc) {
    const unsigned FULL = 0xffffffffu;
    const int l = threadIdx.x & 15, k2 = l + 16;
    float a1[16], a2[8 * RB];
    __syncwarp();  // both Grams are written
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int i = l >> 2;
        const float4 t = c <= i ? *reinterpret_cast<const float4*>(gram + 16 * (i * (i + 1) / 2 + c) + 4 * (l & 3))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
        a1[4 * c] = t.x, a1[4 * c + 1] = t.y, a1[4 * c + 2] = t.z, a1[4 * c + 3] = t.w;
    }
#pragma unroll
    for (int c = 0; c < 2 * RB; ++c) {
        const int i = k2 >> 2;
        const float4 t = c <= i && k2 < 8 * RB
                             ? *reinterpret_cast<const float4*>(gram + 16 * (i * (i + 1) / 2 + c) + 4 * (l & 3))
                             : make_float4(0.f, 0.f, 0.f, 0.f);
        a2[4 * c] = t.x, a2[4 * c + 1] = t.y, a2[4 * c + 2] = t.z, a2[4 * c + 3] = t.w;
    }
    float y1 = gram[36 * 16 + l], y2 = k2 < 8 * RB ? gram[36 * 16 + k2] : 0.f;
    __syncwarp();  // Lc is free
    float tr = 0.f, t2 = 0.f;
#pragma unroll
    for (int c = 0; c < 16; ++c)
        if (c == l) tr = a1[c];
#pragma unroll
    for (int c = 16; c < 8 * RB; ++c)
        if (c == k2) t2 = a2[c];
    tr += t2;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) tr += __shfl_xor_sync(FULL, tr, o);
    const bool zero = !(tr > 0.f) || len == 0;
    const float lam = lam_rel * tr / (float)r;
#pragma unroll
    for (int c = 0; c < 16; ++c)
        if (c == l) a1[c] += lam;  // (r > 16: every first row is below the rank)
#pragma unroll
    for (int c = 0; c < 8 * RB; ++c) {
        const float d = k2 < r ? a2[c] + lam : 1.f;
        a2[c] = c == k2 ? d : (k2 >= r ? 0.f : a2[c]);
    }
    if (k2 >= r) y2 = 0.f;
    float dmin = 3.0e38f, dmax = 0.f, inv1 = 1.f, inv2 = 1.f;
    bool ok = true;
    chol_block32<0, RB>(a1, a2, y1, y2, l, r, ok, dmin, dmax, inv1, inv2, Lc);
    chol_block32<1, RB>(a1, a2, y1, y2, l, r, ok, dmin, dmax, inv1, inv2, Lc);
    chol_block32<2, RB>(a1, a2, y1, y2, l, r, ok, dmin, dmax, inv1, inv2, Lc);
    if constexpr (RB > 3) chol_block32<3, RB>(a1, a2, y1, y2, l, r, ok, dmin, dmax, inv1, inv2, Lc);
    // L^T x = y: a lane reads its rows' columns of L (35 k + j: no bank conflicts)
    const float* c1 = Lc + l * (kWarpCol - 1);
    const float* c2 = Lc + k2 * (kWarpCol - 1);
#pragma unroll 4
    for (int j = 8 * RB - 1; j >= 16; --j) {
        const float m1 = c1[j], m2 = c2[j];
        const float xj = __shfl_sync(FULL, y2 * inv2, j - 16, 16);
        if (k2 == j) y2 = xj;
        else if (k2 < j) y2 = fmaf(-m2, xj, y2);
        y1 = fmaf(-m1, xj, y1);
    }
#pragma unroll 4
    for (int j = 15; j >= 0; --j) {
        const float m1 = c1[j];
        const float xj = __shfl_sync(FULL, y1 * inv1, j, 16);
        if (l == j) y1 = xj;
        else if (l < j) y1 = fmaf(-m1, xj, y1);
    }
    *u1 = zero ? 0.f : y1;
    *u2 = zero || k2 >= r ? 0.f : y2;
    return zero || (ok && !(dmin < kPivotRatio * dmax));
}

// ---- Float64 factor and solve of one line in one warp (the retry above rank 16) ----
// Column J of the in-warp Cholesky and the columns after it, unrolled at compile
// time (a loop whose inner bound depends on the outer index is not fully unrolled
// by the compiler, and acc then lives in local memory)
template <int G, typename T, int J>
__device__ __forceinline__ void chol_col(T (&acc)[G], int k, int r, bool& ok, T& dmin, T& dmax) {
    if constexpr (J < G) {
        const unsigned FULL = 0xffffffffu;
        const T djj = __shfl_sync(FULL, acc[J], J, G);
        if (J < r) {
            ok &= (djj > T(0));
            dmin = djj < dmin ? djj : dmin;
            dmax = djj > dmax ? djj : dmax;
        }
        const T dpos = djj > T(0) ? djj : T(1);
        const T ljj = sqrt(dpos);
        const T inv = T(1) / ljj;
        const T lij = (k > J) ? acc[J] * inv : (k == J ? ljj : T(0));
        acc[J] = lij;
#pragma unroll
        for (int c = J + 1; c < G; ++c) {
            const T lcj = __shfl_sync(FULL, lij, c, G);
            if (k > J) acc[c] -= lij * lcj;
        }
        chol_col<G, T, J + 1>(acc, k, r, ok, dmin, dmax);
    }
}

// Step J of the backward substitution L^T x = y and the steps before it
template <int G, typename T, int J>
__device__ __forceinline__ void back_col(const T (&acc)[G], int k, T& x) {
    if constexpr (J >= 0) {
        const unsigned FULL = 0xffffffffu;
        const T xj = __shfl_sync(FULL, x, J, G) / __shfl_sync(FULL, acc[J], J, G);
        if (k == J) x = xj;
#pragma unroll
        for (int c = 0; c < J; ++c) {
            const T ljc = __shfl_sync(FULL, acc[c], J, G);
            if (k == c) x -= ljc * xj;
        }
        back_col<G, T, J - 1>(acc, k, x);
    }
}

// Lane k holds row k of the Gram in acc and b_k in rhs and receives u_k.
template <int G, typename T>
__device__ __forceinline__ void factor_solve_rows(T (&acc)[G], T rhs, int len, int r, float lam_rel, int k,
                                                  T* out_k) {
    const unsigned FULL = 0xffffffffu;
    T tr = T(0);
#pragma unroll
    for (int c = 0; c < G; ++c)
        if (c == k) tr = acc[c];
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) tr += __shfl_xor_sync(FULL, tr, o, G);
    const bool zero = !(tr > T(0)) || len == 0;
    const T lam = (T)lam_rel * tr / (T)r;
#pragma unroll
    for (int c = 0; c < G; ++c)
        if (c == k) acc[c] = (k < r) ? acc[c] + lam : T(1);
    if (k >= r) {
#pragma unroll
        for (int c = 0; c < G; ++c)
            if (c != k) acc[c] = T(0);
        rhs = T(0);
    }
    // right-looking Cholesky: lane i keeps row i; column j of L overwrites acc[j]
    T dmin = T(3.0e38), dmax = T(0);
    bool ok = true;
    chol_col<G, T, 0>(acc, k, r, ok, dmin, dmax);
    // forward L y = b: lane k holds L[k][0..k] in acc[0..k]
    T y = rhs;
#pragma unroll
    for (int j = 0; j < G; ++j) {
        const T yj = __shfl_sync(FULL, y, j, G) / __shfl_sync(FULL, acc[j], j, G);
        if (k == j) y = yj;
        else if (k > j) y -= acc[j] * yj;
    }
    // backward L^T x = y: x_j is final at step j; L[j][c] (c < j) comes from lane j
    T x = y;
    back_col<G, T, G - 1>(acc, k, x);
    *out_k = (zero || k >= r) ? T(0) : x;
}

// One half-step for ranks above 16: rows of U (rows_side) or columns of V, two lines a
// warp.  A persistent grid: warps take the frame's lines in order, two at a time, from
// a counter (lines of one slice run side by side and share its factor rows in L1), so
// that no CTA waits for another's share.  A line whose pivots fail the check goes to
// the float64 pass (k_als_retry).
// What bounds it: issue and the latency of shared memory at 16 warps per SM (each scheduler
// issues in 51% of its cycles; the 24 warps that stages of 16 rows leave room for gain
// nothing), then the dependent columns of the solve.  Completion of the 200-box scene (5.7 M
// entries, ranks 8 to 32 per slice, 10 sweeps; the lane-group kernel has the slices up to
// rank 16): 23.9 ms with a lane per factor row in the copies, a shuffle per element in the
// Cholesky and 32-way bank conflicts in the solves; 12.6 ms with a row of the Gram a lane
// and a warp per solve; 7.85 ms so.
constexpr int kHalfWarps = 8;
// a warp's floats: two stages and the first line's Gram; the second line's Gram and then the
// columns of L of both take the same place
constexpr int kHalfFloats = 2 * kWarpStage + kWarpGram;
constexpr int kHalfSmem = kHalfWarps * kHalfFloats * 4;
constexpr int kHalfCols = 32 * kWarpCol + 16;  // from the first half's columns of L to the second's: other banks
static_assert(kHalfCols + 32 * kWarpCol <= kHalfFloats, "the columns of L fit");
static_assert(kHalfFloats % 4 == 0 && kWarpGram % 4 == 0 && kHalfCols % 4 == 0, "16-byte accesses");

__global__ void __launch_bounds__(32 * kHalfWarps, 2) k_als_half(lt_frame F, lt_samples smp, Omega om, int R,
                                                                const int32_t* __restrict__ rk, float lam_rel,
                                                                bool rows_side, const float* __restrict__ Fin,
                                                                float* __restrict__ Fout, AlsQueue<32> aq,
                                                                int32_t* __restrict__ next) {
    extern __shared__ __align__(16) float wst[];
    const int lane = threadIdx.x & 31, half = lane >> 4, l = lane & 15;
    float* st = wst + (threadIdx.x >> 5) * kHalfFloats;
    const int S = F.S;
    const int64_t total = rows_side ? (int64_t)F.slice_off[S] : om.line_pfx[S];
    int s = -1;
    int64_t s_lo = 0, s_hi = 0;  // lines of slice s
    for (;;) {
        int64_t L0 = 0;
        if (lane == 0) L0 = 2 * (int64_t)atomicAdd(next, 1);
        L0 = __shfl_sync(0xffffffffu, L0, 0);
        if (L0 >= total) break;
        // the two lines (uniform in the warp; rank 0: none, or the lane-group kernel has it)
        int rr[2], len[2], jj[2];
        int64_t ent[2], dst[2], srow[2];
        float vv[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t L = L0 + h;
            rr[h] = len[h] = jj[h] = 0;
            ent[h] = dst[h] = srow[h] = 0;
            vv[h] = 0.f;
            if (L >= total) continue;
            if (L >= s_hi) {  // the slice with s_lo <= L < s_hi, at or after the last one's
                int x = s < 0 ? 0 : s + 1, y = S - 1;
                while (x < y) {
                    const int m = (x + y) >> 1;
                    if (L >= (rows_side ? (int64_t)F.slice_off[m + 1] : om.line_pfx[m + 1])) x = m + 1;
                    else y = m;
                }
                s = x;
                s_lo = rows_side ? (int64_t)F.slice_off[s] : om.line_pfx[s];
                s_hi = rows_side ? (int64_t)F.slice_off[s + 1] : om.line_pfx[s + 1];
            }
            const int r = slice_rank(rk, s, R);  // the slice's rank (factor rows have stride R)
            if (rk && r <= 16) continue;         // per-slice ranks: the lane-group kernel has these slices
            rr[h] = r;
            const int line = (int)(L - s_lo);
            const int row0 = F.slice_off[s];
            srow[h] = rows_side ? (int64_t)s * F.C * R : (int64_t)row0 * R;
            const int32_t* ptr = rows_side ? om.rp + row0 + s : om.cp + (int64_t)s * (F.C + 1);
            const int b0 = ptr[line];
            len[h] = ptr[line + 1] - b0;
            dst[h] = rows_side ? (int64_t)(row0 + line) * R : ((int64_t)s * F.C + line) * R;
            ent[h] = smp.off[s] + b0;
            if (lane < len[h]) {
                jj[h] = (int)(rows_side ? om.cidx : om.ridx)[ent[h] + lane];
                vv[h] = (rows_side ? om.cval : om.rval)[ent[h] + lane];
            }
        }
        if (rr[0] + rr[1] == 0) continue;
        const bool three = max(rr[0], rr[1]) <= 24;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            if ((h ? rr[1] : rr[0]) == 0) continue;
            const int n = h ? len[1] : len[0], j = h ? jj[1] : jj[0];
            const float av = h ? vv[1] : vv[0];
            const uint16_t* idx = (rows_side ? om.cidx : om.ridx) + (h ? ent[1] : ent[0]);
            const float* val = (rows_side ? om.cval : om.rval) + (h ? ent[1] : ent[0]);
            const float* src = Fin + (h ? srow[1] : srow[0]);
            float* out = h ? st : st + 2 * kWarpStage;
            if (three) gram_warp<3>(n, idx, val, j, av, src, R, st, out);
            else gram_warp<4>(n, idx, val, j, av, src, R, st, out);
        }
        const float* gram = half ? st : st + 2 * kWarpStage;
        float* Lc = st + half * kHalfCols;
        const int r = half ? rr[1] : rr[0], n = half ? len[1] : len[0];
        float x1, x2;
        const bool ok = three ? pair_solve32<3>(gram, n, max(r, 17), lam_rel, &x1, &x2, Lc)
                              : pair_solve32<4>(gram, n, max(r, 17), lam_rel, &x1, &x2, Lc);
        if (r > 0) {
            const int64_t d = half ? dst[1] : dst[0];
            Fout[d + l] = ok ? x1 : 0.f;
            if (l + 16 < R) Fout[d + l + 16] = ok ? x2 : 0.f;
            if (!ok && l == 0) {
                // rare: the float pivots were not acceptable; k_als_retry forms the line's
                // Gram again in float64 from the factor rows (a Gram summed in float32 would
                // carry its rounding into the solve)
                const int qs = atomicAdd(aq.count, 1);
                if (qs < aq.cap) {
                    aq.dst[qs] = d;
                    aq.slot[qs] = half ? ent[1] : ent[0];
                    aq.src[qs] = half ? srow[1] : srow[0];
                    aq.len[qs] = n;
                    aq.grp[qs] = 0;  // contiguous in CSR / CSC
                    aq.rank[qs] = r;
                } else {
                    latch(aq.status, LT_ELIMIT);
                }
            }
        }
        __syncwarp();
    }
}

// ---- Masked ALS, a group of lanes per line (r <= 16) ---------------------------
// A line is a row of U_s (U-step) or a column of V_s (V-step); its 2^g lanes have its
// entries in turn, each as a stream of the sliced layout.  A lane gathers the factor row
// x_j of each of its entries from the slice's factor rows staged in shared memory and
// accumulates the lower triangle of G = sum x_j x_j^T and b = sum a_j x_j in registers
// (RP(RP+1)/2 + RP values); the group's sums go to its first lane, which adds the ridge
// lam_rel tr(G)/r, factors G by Cholesky in float32 and solves.
// Lines whose pivots fail the check go to a queue; a second kernel forms their
// Gram again in float64 (products of the float32 factors are exact in float64) and
// solves it in float64, so an ill-conditioned line carries no float32 rounding.
// A staged factor row is RP floats (RP/4 16-byte slots).  Slot q of row j is stored
// at slot q ^ h(j) so that the rows read by one quarter-warp (random j) spread over
// all eight 16-byte bank groups of a 128-byte shared-memory wavefront.
template <int RP>
__device__ __forceinline__ int stage_slot(int j, int q) {
    constexpr int NQ = RP / 4, RPB = 8 / NQ;  // slots per row, rows per wavefront
    return j * NQ + (q ^ ((j / RPB) % NQ));
}

// A factor row, from the staged rows or, for a slice of more rows than the stage holds,
// from memory (row -1: zeros).
template <int RP>
__device__ __forceinline__ void load_row(float (&x)[RP], int j, int r, int R, const float* __restrict__ src,
                                         bool staged, bool vec, const float4* stage4) {
    if (staged) {
#pragma unroll
        for (int q = 0; q < RP / 4; ++q) {
            const float4 t = stage4[stage_slot<RP>(j, q)];
            x[4 * q] = t.x;
            x[4 * q + 1] = t.y;
            x[4 * q + 2] = t.z;
            x[4 * q + 3] = t.w;
        }
    } else if (vec) {  // R and r multiples of 4, rows on 16 bytes
#pragma unroll
        for (int q = 0; q < RP / 4; ++q) {
            float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j >= 0 && 4 * q < r) t = __ldg(reinterpret_cast<const float4*>(src + (int64_t)j * R) + q);
            x[4 * q] = t.x;
            x[4 * q + 1] = t.y;
            x[4 * q + 2] = t.z;
            x[4 * q + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int c = 0; c < RP; ++c) x[c] = j >= 0 && c < r ? __ldg(src + (int64_t)j * R + c) : 0.f;
    }
}

template <int RP>
__device__ __forceinline__ void add_entry(const float (&x)[RP], float av, float (&a)[RP * (RP + 1) / 2],
                                          float (&bb)[RP]) {
#pragma unroll
    for (int i = 0; i < RP; ++i) {
        bb[i] = fmaf(av, x[i], bb[i]);
#pragma unroll
        for (int k = 0; k <= i; ++k) a[i * (i + 1) / 2 + k] = fmaf(x[i], x[k], a[i * (i + 1) / 2 + k]);
    }
}

// The entry streams of a warp's lanes on their way: a ring of kRing chunks of 4 entries
// (8 bytes of indices, 16 of values a lane), filled by cp.async so that no register
// holds them.  Every lane reads what it copied itself.
constexpr int kRing = 4;
constexpr int kRingBytes = kRing * 32 * 24;  // of a warp

__device__ __forceinline__ void ring_copy(unsigned char* ring, int slot, const uint2* idx, const float4* val) {
    const int lane = threadIdx.x & 31;
    const unsigned di = (unsigned)__cvta_generic_to_shared(ring + slot * 256 + lane * 8);
    const unsigned dv = (unsigned)__cvta_generic_to_shared(ring + kRing * 256 + slot * 512 + lane * 16);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(di), "l"(idx) : "memory");
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dv), "l"(val) : "memory");
}

// Adds x_e x_e^T (lower triangle) and a_e x_e for the nk entries of one lane's
// stream (chunks of 4 at idx4[32 c], vv4[32 c]) to a and bb, in stream order.
// The row of the next entry is loaded before this one is added, so that the
// shared-memory reads (bank conflicts of random rows) run under the arithmetic, and the
// stream is three chunks ahead.  Every lane runs to the longest stream of the warp; past
// its own end it adds zeros (row zrow), which leave the sums as they are.  Two entries per
// round of the inner loop: the whole chunk unrolled is more code than the instruction
// caches hold.
template <int RP>
__device__ __forceinline__ void stream_gram(int nk, const uint2* __restrict__ idx4, const float4* __restrict__ vv4,
                                            int r, int R, const float* __restrict__ src, bool staged, bool vec,
                                            int zrow, const float4* stage4, unsigned char* ring,
                                            float (&a)[RP * (RP + 1) / 2], float (&bb)[RP]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < RP * (RP + 1) / 2; ++i) a[i] = 0.f;
#pragma unroll
    for (int i = 0; i < RP; ++i) bb[i] = 0.f;
    const int nc = (__reduce_max_sync(0xffffffffu, nk) + 3) >> 2;
    if (nc == 0) return;
    auto ring_idx = [&](int c) { return *reinterpret_cast<const uint2*>(ring + (c & (kRing - 1)) * 256 + lane * 8); };
    auto fill = [&](int c) {
        if (c < nc) ring_copy(ring, c & (kRing - 1), idx4 + 32 * c, vv4 + 32 * c);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int c = 0; c < kRing - 1; ++c) fill(c);
    asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");  // chunk 0
    float x[RP], y[RP];
    uint2 ic = ring_idx(0);
    load_row<RP>(x, nk > 0 ? (int)(ic.x & 0xffffu) : zrow, r, R, src, staged, vec, stage4);
    for (int c = 0; c < nc; ++c) {
        fill(c + kRing - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");  // chunks up to c + 1
        const float4 vc = *reinterpret_cast<const float4*>(ring + kRing * 256 + (c & (kRing - 1)) * 512 + lane * 16);
        const uint2 in = ring_idx(c + 1);  // (past the last chunk: not used)
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const int e = 4 * c + 2 * h;
            const uint32_t w0 = h ? ic.y : ic.x, w1 = h ? in.x : ic.y;
            const float v0 = h ? vc.z : vc.x, v1 = h ? vc.w : vc.y;
            load_row<RP>(y, e + 1 < nk ? (int)(w0 >> 16) : zrow, r, R, src, staged, vec, stage4);
            add_entry<RP>(x, e < nk ? v0 : 0.f, a, bb);
            load_row<RP>(x, e + 2 < nk ? (int)(w1 & 0xffffu) : zrow, r, R, src, staged, vec, stage4);
            add_entry<RP>(y, e + 1 < nk ? v1 : 0.f, a, bb);
        }
        ic = in;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// One lane of a warp task: `line` (or -1) is its line, `sub` its rank among the G
// lanes of the line, `slot` the first slot of its stream (task base + 4 lane).
template <int RP>
__device__ __forceinline__ void als_line(const lt_frame& F, const Omega& om, int r, int R, bool rows_side,
                                         const float* __restrict__ src_base, const float* __restrict__ src,
                                         bool staged, bool vec, int zrow, const float4* stage4,
                                         unsigned char* ring, float* __restrict__ Fout, float lam_rel, const AlsQueue<RP>& q, int s,
                                         int line, int sub, int G, int64_t slot) {
    constexpr int NA = RP * (RP + 1) / 2;
    const int row0 = F.slice_off[s];
    int len = 0;
    if (line >= 0) {
        if (rows_side) {
            const int32_t* rp = om.rp + row0 + s;
            len = rp[line + 1] - rp[line];
        } else {
            const int32_t* cp = om.cp + (int64_t)s * (F.C + 1);
            len = cp[line + 1] - cp[line];
        }
    }
    const uint16_t* sidx = rows_side ? om.sidx_r : om.sidx_c;
    const float* sval = rows_side ? om.sval_r : om.sval_c;
    float a[NA], bb[RP];
    const int nk = sub < len ? (len - sub + G - 1) / G : 0;
    stream_gram<RP>(nk, reinterpret_cast<const uint2*>(sidx + slot), reinterpret_cast<const float4*>(sval + slot), r,
                    R, src, staged, vec, zrow, stage4, ring, a, bb);
    if (G > 1) {  // the group's partial sums into its first lane (G is warp-uniform)
        for (int m = G >> 1; m > 0; m >>= 1) {
#pragma unroll
            for (int i = 0; i < NA; ++i) a[i] += __shfl_down_sync(0xffffffffu, a[i], m, G);
#pragma unroll
            for (int i = 0; i < RP; ++i) bb[i] += __shfl_down_sync(0xffffffffu, bb[i], m, G);
        }
    }
    if (line < 0 || sub != 0) return;
    const int64_t dst = rows_side ? (int64_t)(row0 + line) * R : ((int64_t)s * F.C + line) * R;
    for (int i = r; i < R; ++i) Fout[dst + i] = 0.f;  // components beyond the slice's rank
    if (chol_solve<RP, float>(a, bb, r, lam_rel, true)) {
#pragma unroll
        for (int i = 0; i < RP; ++i)
            if (i < r) Fout[dst + i] = bb[i];
        return;
    }
    // rare: queue the line for the float64 pass (k_als_retry)
    const int qs = atomicAdd(q.count, 1);
    if (qs >= q.cap) {
        latch(q.status, LT_ELIMIT);
        return;
    }
    q.dst[qs] = dst;
    q.slot[qs] = slot;
    q.src[qs] = src - src_base;
    q.len[qs] = len;
    q.grp[qs] = G;
    q.rank[qs] = r;
}

// stage the slice's source factor rows (nsrc rows of stride R, the first r values,
// zero-padded to RP) in shared memory, and a row of zeros after them
template <int RP>
__device__ __forceinline__ void stage_factors(const float* __restrict__ src, int nsrc, int r, int R, bool vec,
                                              float4* stage4) {
    constexpr int NQ = RP / 4;
    for (int i = threadIdx.x; i < (nsrc + 1) * NQ; i += blockDim.x) {
        const int row = i / NQ, q4 = i % NQ;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < nsrc) {
            const float* p = src + (int64_t)row * R + 4 * q4;
            if (vec) {
                if (4 * q4 < r) v = __ldg(reinterpret_cast<const float4*>(p));
            } else {
                v.x = 4 * q4 < r ? __ldg(p) : 0.f;
                v.y = 4 * q4 + 1 < r ? __ldg(p + 1) : 0.f;
                v.z = 4 * q4 + 2 < r ? __ldg(p + 2) : 0.f;
                v.w = 4 * q4 + 3 < r ? __ldg(p + 3) : 0.f;
            }
        }
        stage4[stage_slot<RP>(row, q4)] = v;
    }
}

// Persistent half-step: one CTA per SM.  CTA c owns the warp tasks (all slices, in
// slice order) whose start lies in its equal share [lo, hi) of the side's work, a task
// counting its slots and kTaskCost for its solve.  It stages the source factor rows of
// the slices it touches, as many at once as fit (most shares lie in two or three
// slices), and its warps take all their tasks from one shared counter.
// What bounds it: latency at two warps per scheduler (the registers of a lane's Gram) and
// the bank conflicts of random factor rows.  Completion of 7.2 M entries in 64 slices,
// rank 16, 10 sweeps: 4.24 ms with 110 KB of stage, one slice staged at a time, shares
// that count slots only, no row loaded ahead and the stream one chunk ahead; 2.83 ms so
// (with the Omega build below it).  With three times the rows (slices over the old
// stage, read from memory by scalar loads): 11.57 to 6.53 ms.
// Packed multiply-adds (two elements an instruction) run at the rate of single ones
// here and cost register moves: 4.58 ms.
constexpr int kSegs = 8;

struct AlsSeg {
    int s, t0, t1;      // tasks [t0, t1) of slice s
    int row;            // first staged row, or -1: not staged
    int end;            // tasks of the batch up to and with this segment
};

template <int RP>
__global__ void __launch_bounds__(256, RP == 8 ? 2 : 1) k_als_line(lt_frame F, lt_samples smp, Omega om, int R,
                                                    const int32_t* __restrict__ rk, bool rows_side,
                                                    const float* __restrict__ Fin, float* __restrict__ Fout,
                                                    float lam_rel, AlsQueue<RP> q, int stage_rows) {
    extern __shared__ float4 stage4[];
    __shared__ int s_next, s_n;
    __shared__ AlsSeg seg[kSegs];
    unsigned char* ring = reinterpret_cast<unsigned char*>(stage4 + (int64_t)stage_rows * (RP / 4)) +
                          (threadIdx.x >> 5) * kRingBytes;
    const int S = F.S;
    const int64_t* base = rows_side ? om.rbase : om.cbase;
    const int64_t* wk = rows_side ? om.rwk : om.cwk;
    const int32_t* cls_all = rows_side ? om.rcls : om.ccls;
    const int32_t* tb_all = rows_side ? om.rtb : om.ctb;
    // a layout over its capacity was latched as LT_ELIMIT and not written: read nothing
    if (base[S] > om.sell_cap) return;
    const int64_t total = wk[S];
    const int64_t lo = total * blockIdx.x / gridDim.x;
    const int64_t hi = blockIdx.x + 1 == gridDim.x ? INT64_MAX : total * (blockIdx.x + 1) / gridDim.x;
    // tasks of slice x (none where its rank is k_als_half's) and the work before task t
    auto tasks_of = [&](int x) {
        return slice_rank(rk, x, R) <= RP ? cls_all[(int64_t)x * 16 + 8 + kClasses] : 0;
    };
    auto before = [&](int x, int t) {
        return wk[x] + tb_all[(int64_t)x * om.tcap + t] + (int64_t)kTaskCost * t;
    };
    // first task in [t, T) of slice x that starts at or after `at`
    auto first_task = [&](int x, int t, int T, int64_t at) {
        while (t < T) {
            const int m = (t + T) >> 1;
            if (before(x, m) < at) t = m + 1; else T = m;
        }
        return t;
    };
    const int lane = threadIdx.x & 31;
    int s = -1, t = 0;  // next task to consider (thread 0's view, shared through seg)
    if (threadIdx.x == 0) {
        // Task starts are non-decreasing in (slice, task) order and every task of slice
        // s starts at or before the end of slice s: the first slice that ends at or after
        // lo holds the first task at or after lo, if it has one, else a later slice does.
        int x = 0, y = S;
        while (x < y) {
            const int m = (x + y) >> 1;
            if (wk[m + 1] < lo) x = m + 1; else y = m;
        }
        s = x;
        t = s < S ? first_task(s, 0, tasks_of(s), lo) : 0;
    }
    for (;;) {
        if (threadIdx.x == 0) {
            // the next slice segments of this CTA (tasks starting before hi), while their rows fit
            int n = 0, used = 0, tasks = 0;
            while (s < S && n < kSegs) {
                const int T = tasks_of(s);
                if (t < T && before(s, t) >= hi) s = S;  // the share ends here
                if (s >= S) break;
                const int t1 = first_task(s, t, T, hi);
                if (t < t1) {
                    const int need = (rows_side ? smp.ncol[s] : F.slice_off[s + 1] - F.slice_off[s]) + 1;
                    const bool fits = need <= stage_rows;
                    if (fits && used + need > stage_rows) break;  // in the next batch
                    tasks += t1 - t;
                    seg[n++] = AlsSeg{s, t, t1, fits ? used : -1, tasks};
                    if (fits) used += need;
                }
                if (t1 < T) {
                    s = S;  // the share ends inside this slice
                } else {
                    ++s;
                    t = 0;
                }
            }
            s_n = n;
            s_next = 0;
        }
        __syncthreads();
        const int n = s_n;
        if (n == 0) break;
        for (int k = 0; k < n; ++k) {
            if (seg[k].row < 0) continue;
            const int sl = seg[k].s, row0 = F.slice_off[sl], r = slice_rank(rk, sl, R);
            const float* src = rows_side ? Fin + (int64_t)sl * F.C * R : Fin + (int64_t)row0 * R;
            const bool vec = (R & 3) == 0 && (r & 3) == 0 && ((uintptr_t)src & 15) == 0;
            stage_factors<RP>(src, rows_side ? smp.ncol[sl] : F.slice_off[sl + 1] - row0, r, R, vec,
                              stage4 + seg[k].row * (RP / 4));
        }
        __syncthreads();
        for (;;) {
            int tk = 0;
            if (lane == 0) tk = atomicAdd(&s_next, 1);
            tk = __shfl_sync(0xffffffffu, tk, 0);
            if (tk >= seg[n - 1].end) break;
            int k = 0;
            while (tk >= seg[k].end) ++k;
            tk = seg[k].t1 - (seg[k].end - tk);
            const int sl = seg[k].s, row0 = F.slice_off[sl], r = slice_rank(rk, sl, R);
            const bool staged = seg[k].row >= 0;
            const int nsrc = rows_side ? smp.ncol[sl] : F.slice_off[sl + 1] - row0;
            const float* src = rows_side ? Fin + (int64_t)sl * F.C * R : Fin + (int64_t)row0 * R;
            const bool vec = (R & 3) == 0 && (r & 3) == 0 && ((uintptr_t)src & 15) == 0;
            const int32_t* ord = rows_side ? om.rord + row0 : om.cord + (int64_t)sl * F.C;
            const int32_t* cls = cls_all + (int64_t)sl * 16;
            int c = 0;
            while (c + 1 < kClasses && tk >= cls[8 + c + 1]) ++c;
            const int g = kClasses - 1 - c, G = 1 << g;
            const int li = cls[c] + (tk - cls[8 + c]) * (32 >> g) + (lane >> g);
            const bool live = li < cls[c + 1];
            als_line<RP>(F, om, r, R, rows_side, Fin, src, staged, vec, staged ? nsrc : -1,
                         stage4 + (staged ? seg[k].row * (RP / 4) : 0), ring, Fout, lam_rel, q, sl, live ? ord[li] : -1,
                         lane & (G - 1), G, base[sl] + tb_all[(int64_t)sl * om.tcap + tk] + 4 * lane);
        }
        __syncthreads();  // the stage and the segments are reused by the next batch
    }
}

// float64 solve of the queued lines: one warp per line.  The warp walks the line's
// entries in chunks of 32 (lane l gathers entry e0 + l: its factor row and value into
// shared memory), and each lane accumulates its share of the Gram lower triangle and
// right-hand side elements (element lane + 32 p) in float64 over the chunk; the
// first lane then factors and solves in float64.
template <int RP>
__global__ void __launch_bounds__(128) k_als_retry(AlsQueue<RP> q, Omega om, bool rows_side,
                                                   const float* __restrict__ Fin, int R, float lam_rel,
                                                   float* __restrict__ Fout, int32_t* __restrict__ n_fp64) {
    constexpr int NA = RP * (RP + 1) / 2, NV = NA + RP, PER = (NV + 31) / 32;
    __shared__ float xs[4][32][RP + 1];
    __shared__ float av[4][32];
    __shared__ double gs[4][NV];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int ei[PER], ek[PER];  // owned element: Gram (ei, ek) with ek <= ei, or b_ei (ek = -1); ei = -1 for none
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int e = lane + 32 * p;
        ei[p] = -1;
        ek[p] = -1;
        if (e < NA) {
            int i = 0;
            while ((i + 1) * (i + 2) / 2 <= e) ++i;
            ei[p] = i;
            ek[p] = e - i * (i + 1) / 2;
        } else if (e < NV) {
            ei[p] = e - NA;
        }
    }
    const uint16_t* sidx = rows_side ? om.sidx_r : om.sidx_c;
    const float* sval = rows_side ? om.sval_r : om.sval_c;
    const int n = (int)min((int64_t)*q.count, q.cap);
    for (int t = blockIdx.x * 4 + w; t < n; t += gridDim.x * 4) {
        const int len = q.len[t], G = q.grp[t], r = q.rank[t];
        const int64_t slot = q.slot[t];
        const float* src = Fin + q.src[t];
        double acc[PER];
#pragma unroll
        for (int p = 0; p < PER; ++p) acc[p] = 0.0;
        for (int e0 = 0; e0 < len; e0 += 32) {
            const int e = e0 + lane;
            if (e < len) {
                int j;
                if (G > 0) {  // sliced layout
                    const int u = e % G, kk = e / G;
                    const int64_t pos = slot + 4 * u + 128 * (kk >> 2) + (kk & 3);
                    j = sidx[pos];
                    av[w][lane] = sval[pos];
                } else {      // CSR / CSC
                    j = (rows_side ? om.cidx : om.ridx)[slot + e];
                    av[w][lane] = (rows_side ? om.cval : om.rval)[slot + e];
                }
#pragma unroll
                for (int c = 0; c < RP; ++c) xs[w][lane][c] = c < r ? src[(int64_t)j * R + c] : 0.f;
            }
            __syncwarp();
            const int ne = min(32, len - e0);
            for (int k2 = 0; k2 < ne; ++k2) {
#pragma unroll
                for (int p = 0; p < PER; ++p) {
                    if (ei[p] >= 0) {
                        const double xi = (double)xs[w][k2][ei[p]];
                        const double xk = ek[p] >= 0 ? (double)xs[w][k2][ek[p]] : (double)av[w][k2];
                        acc[p] = fma(xi, xk, acc[p]);
                    }
                }
            }
            __syncwarp();
        }
#pragma unroll
        for (int p = 0; p < PER; ++p)
            if (lane + 32 * p < NV) gs[w][lane + 32 * p] = acc[p];
        __syncwarp();
        if constexpr (RP == 32) {
            // rank above 16: the warp factors and solves (lane k holds row k), the
            // Cholesky of one lane would not fit its registers
            double row[32];
#pragma unroll
            for (int c = 0; c < 32; ++c)
                row[c] = c <= lane ? gs[w][lane * (lane + 1) / 2 + c] : gs[w][c * (c + 1) / 2 + lane];
            double xd = 0.0;
            factor_solve_rows<32, double>(row, gs[w][NA + lane], len, r, lam_rel, lane, &xd);
            if (lane < r) Fout[q.dst[t] + lane] = (float)xd;
            if (lane == 0) atomicAdd(n_fp64, 1);
        } else if (lane == 0) {
            double a[NA], b[RP];
            for (int i = 0; i < NA; ++i) a[i] = gs[w][i];
            for (int i = 0; i < RP; ++i) b[i] = gs[w][NA + i];
            chol_solve<RP, double>(a, b, r, lam_rel, false);
            float* d = Fout + q.dst[t];
            for (int i = 0; i < RP; ++i)
                if (i < r) d[i] = (float)b[i];
            atomicAdd(n_fp64, 1);
        }
        __syncwarp();
    }
}

// Image of slice s (Sec. 3): t_s = V_s^T w, then img[perm[i]] = max(0, u_i . t_s).
// blockIdx.y is the slice; each CTA forms t_s itself (the slice's V rows are read once
// from DRAM and then from L2): thread x owns component x % r of the columns
// x / r + c (blockDim / r), c = 0, 1, ... (consecutive threads read consecutive floats),
// and the partial sums are added in a fixed order.  The CTAs of a slice then split
// its rows, a thread per row (16-byte loads of u_i when r is a multiple of 4 and U
// 16-byte aligned).
__global__ void __launch_bounds__(512) k_render(lt_frame F, lt_samples smp, const float* __restrict__ U,
                                                const float* __restrict__ V, int r, const float* __restrict__ w,
                                                const int32_t* __restrict__ perm, float* __restrict__ img) {
    __shared__ float part[512];
    __shared__ float t[32];
    const int s = blockIdx.y;
    const int ns = smp.ncol[s];
    const int cpp = (int)blockDim.x / r;  // columns per pass
    const int col = (int)threadIdx.x / r, k = (int)threadIdx.x - col * r;
    float acc = 0.f;
    if (col < cpp) {
        const float* Vs = V + (int64_t)s * F.C * r;
        const float* ws = w ? w + (int64_t)s * F.C : nullptr;
        for (int j = col; j < ns; j += cpp) acc = fmaf(Vs[(int64_t)j * r + k], ws ? ws[j] : 1.f, acc);
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    if ((int)threadIdx.x < r) {
        float a = 0.f;
        for (int c = 0; c < cpp; ++c) a += part[c * r + threadIdx.x];
        t[threadIdx.x] = a;
    }
    __syncthreads();
    const int row0 = F.slice_off[s], ms = F.slice_off[s + 1] - row0;
    const bool vec = (r & 3) == 0 && ((uintptr_t)U & 15) == 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ms; i += gridDim.x * blockDim.x) {
        const float* u = U + (int64_t)(row0 + i) * r;
        float v = 0.f;
        if (vec) {
            const float4* u4 = reinterpret_cast<const float4*>(u);
            for (int q = 0; q < (r >> 2); ++q) {
                const float4 x = __ldg(u4 + q);
                v = fmaf(x.x, t[4 * q], v);
                v = fmaf(x.y, t[4 * q + 1], v);
                v = fmaf(x.z, t[4 * q + 2], v);
                v = fmaf(x.w, t[4 * q + 3], v);
            }
        } else {
            for (int q = 0; q < r; ++q) v = fmaf(__ldg(u + q), t[q], v);
        }
        img[perm[row0 + i]] = fmaxf(v, 0.f);
    }
}

// r_s = min(R, max(8, 8 ceil(n'_s / cols))): a multiple of 8 growing with the coarsened cut
__global__ void k_slice_ranks(lt_samples smp, int S, int R, int cols, int32_t* __restrict__ rank) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) {
        const int n = smp.ncol[s];
        rank[s] = min(R, max(8, 8 * ((n + cols - 1) / cols)));
    }
}

}  // namespace

namespace ltk {

lt_status omega_build(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, int64_t E, bool sell, bool csr, bool bits,
                      const int32_t* rk, int R, Omega* omp) {
    const int S = f->S, C = f->C;
    const int64_t mr = std::max(f->max_rows, 1);
    Omega& om = *omp;
    om.bm_stride = mr * ((C + 31) / 32);
    om.bt_stride = (int64_t)C * ((mr + 31) / 32);
    om.sell = sell;
    om.csr = csr;
    // Sliced layout capacity, le = lane_entries.  Per slice and side, for lines sorted
    // by count, the padding of a task is at most the entries of the task before it
    // (the first task of class g < 5 adds at most 32 le slots, of class 5 at most
    // L_max), rounding to a multiple of 4 adds at most 128 slots per task, and there
    // are at most n / 32 + 2 E_s / (32 le) + 6 tasks (a class g > 0 line has more than
    // le 2^(g-1) entries): at most E_s (1 + 8 / le) + 4 n + L_max + 160 le + 768 slots.
    // Beyond the capacity the scatter latches LT_ELIMIT.
    const int64_t nmax = std::max<int64_t>(mr, C);
    om.lane_entries = ctx->tune.als_lane_entries;
    const int64_t le = om.lane_entries;
    om.sell_cap = om.sell ? E + (8 * E + le - 1) / le + E / 32 + (int64_t)S * (5 * nmax + 160 * le + 1024) : 0;
    om.tcap = (int)nmax + 8;
    const size_t e_csr = om.csr ? (size_t)E : 0, e_sell = (size_t)om.sell_cap;
    const size_t t_sell = om.sell ? (size_t)S * om.tcap : 0;
    lt_status st;
    char* p = (char*)lt_scratch(ctx, SCR_OMEGA,
                                (size_t)(f->m + S) * 4 + (size_t)S * (C + 1) * 4 + e_csr * 16 + e_sell * 12 + S * 8 +
                                    (size_t)S * (om.bm_stride + om.bt_stride) * (bits ? 12 : 8) + (S + 1) * 8 + (size_t)f->m * 8 +
                                    (size_t)S * C * 8 + (size_t)S * 128 + (size_t)(S + 1) * 16 + t_sell * 8 + (size_t)(S + 1) * 16 +
                                    (size_t)S * kOmParts * 4 + 36 * 256,
                                &st);
    if (!p) return st;
    auto take = [&](size_t nbytes) {
        char* q = p;
        p += (nbytes + 255) & ~(size_t)255;
        return q;
    };
    om.rp = (int32_t*)take((f->m + S) * 4);
    om.cp = (int32_t*)take((size_t)S * (C + 1) * 4);
    om.cidx = (uint16_t*)take(e_csr * 2);
    om.cval = (float*)take(e_csr * 4);
    om.ridx = (uint16_t*)take(e_csr * 2);
    om.rval = (float*)take(e_csr * 4);
    om.r2c = (int32_t*)take(e_csr * 4);
    om.mu = (float*)take(S * 4);
    om.bm = bits ? (uint32_t*)take((size_t)S * om.bm_stride * 4) : nullptr;
    om.bt = bits ? (uint32_t*)take((size_t)S * om.bt_stride * 4) : nullptr;
    om.wr = (uint2*)take((size_t)S * om.bm_stride * 8);
    om.wc = (uint2*)take((size_t)S * om.bt_stride * 8);
    om.line_pfx = (int64_t*)take((S + 1) * 8);
    om.rord = (int32_t*)take((size_t)f->m * 4);
    om.cord = (int32_t*)take((size_t)S * C * 4);
    om.rcls = (int32_t*)take((size_t)S * 16 * 4);
    om.ccls = (int32_t*)take((size_t)S * 16 * 4);
    om.rpos = (int32_t*)take((size_t)f->m * 4);
    om.cpos = (int32_t*)take((size_t)S * C * 4);
    om.rtb = (int32_t*)take(t_sell * 4);
    om.ctb = (int32_t*)take(t_sell * 4);
    om.rbase = (int64_t*)take((size_t)(S + 1) * 8);
    om.cbase = (int64_t*)take((size_t)(S + 1) * 8);
    om.rwk = (int64_t*)take((size_t)(S + 1) * 8);
    om.cwk = (int64_t*)take((size_t)(S + 1) * 8);
    om.sidx_r = (uint16_t*)take(e_sell * 2);
    om.sval_r = (float*)take(e_sell * 4);
    om.sidx_c = (uint16_t*)take(e_sell * 2);
    om.sval_c = (float*)take(e_sell * 4);
    float* part = (float*)take((size_t)S * kOmParts * 4);  // partial sums of the observed values
    if ((size_t)(p - (char*)ctx->scr[SCR_OMEGA]) > ctx->scr_size[SCR_OMEGA])
        return lt_fail(ctx, LT_ENOMEM, "omega_build: layout overflow");
    const int nsm = ctx->num_sms;
    // (a thread's chain of dependent loads is what these passes wait for: grids of up to 16
    // CTAs per SM; 4 took 0.31 ms for the scatter of 7.2 M entries)
    const unsigned wide = (unsigned)std::max(1, 16 * nsm / S);
    k_om_clear<<<dim3(std::max(1, 2 * nsm / S), S), 256, 0, ctx->stream>>>(*f, *smp, om);
    LT_LAUNCH_CHECK(ctx, "k_om_clear");
    k_om_bits<<<dim3(wide, S), 256, 0, ctx->stream>>>(*f, *smp, om, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_om_bits");
    k_om_transpose<<<dim3(std::max(kOmParts, 8 * nsm / S), S), 256, 0, ctx->stream>>>(*f, *smp, om, part);
    LT_LAUNCH_CHECK(ctx, "k_om_transpose");
    k_om_lines<<<dim3(wide, S), 256, 0, ctx->stream>>>(*f, *smp, om);
    LT_LAUNCH_CHECK(ctx, "k_om_lines");
    k_om_scan<<<dim3(S, 2), 1024, 0, ctx->stream>>>(*f, *smp, om, part, kOmParts);
    LT_LAUNCH_CHECK(ctx, "k_om_scan");
    if (om.sell) {
        k_om_sellpfx<<<1, 1024, 0, ctx->stream>>>(S, om, rk, R, ctx->d_status);
        LT_LAUNCH_CHECK(ctx, "k_om_sellpfx");
    }
    k_om_scatter<<<dim3(wide, S), 256, 0, ctx->stream>>>(*f, *smp, om);
    LT_LAUNCH_CHECK(ctx, "k_om_scatter");
    k_line_prefix<<<1, 1024, 0, ctx->stream>>>(*smp, S, om.line_pfx);
    LT_LAUNCH_CHECK(ctx, "k_line_prefix");
    return LT_OK;
}

}  // namespace ltk

namespace {

// The previous frame's columns and factors that start a frame's completion
struct WarmStart {
    const int32_t* col_node;   // [S][C] tree node of each previous column
    const int32_t* ncol;       // [S]    previous columns per slice
    const float* V;            // [S][C][R] previous V rows
};

// Temporal coherence: column c of slice s whose node was a column i of the previous
// frame's slice s starts from the previous V row i (components below the slice's
// rank; the previous rows are zero beyond their own rank), the others keep the
// seeded start.  One CTA per slice; the previous node list is staged in shared memory
// and searched linearly (the cut is not sorted by node id).
__global__ void __launch_bounds__(256) k_als_warm(lt_frame F, lt_samples smp, int R, const int32_t* __restrict__ rk,
                                                  WarmStart w, float* __restrict__ V) {
    extern __shared__ int32_t pn[];
    const int s = blockIdx.x;
    const int np = min(w.ncol[s], F.C), ns = smp.ncol[s];
    for (int i = threadIdx.x; i < np; i += blockDim.x) pn[i] = w.col_node[(int64_t)s * F.C + i];
    __syncthreads();
    const int r = slice_rank(rk, s, R);
    for (int c = threadIdx.x; c < ns; c += blockDim.x) {
        const int node = smp.col_node[(int64_t)s * F.C + c];
        int hit = -1;
        for (int i = 0; i < np; ++i)
            if (pn[i] == node) {
                hit = i;
                break;
            }
        if (hit < 0) continue;
        const float* src = w.V + ((int64_t)s * F.C + hit) * R;
        float* dst = V + ((int64_t)s * F.C + c) * R;
        for (int k = 0; k < R; ++k) dst[k] = k < r ? src[k] : 0.f;
    }
}

lt_status complete_impl(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, int32_t iters, float lam_rel,
                        uint64_t seed, lt_factors* uv, const WarmStart* warm) {
    if (!ctx || !frame_ok2(f) || !smp || !smp->key || !smp->val || !smp->off || !smp->cnt || !smp->ncol || !uv ||
        !uv->U || !uv->V || uv->r < 1 || uv->r > 32 || iters < 0 || !(lam_rel >= 0.f))
        return lt_fail(ctx, LT_EINVAL, "lt_complete: bad arguments");
    cudaSetDevice(ctx->device);
    const int S = f->S, C = f->C;
    // The sampling capacity sizes the scratch; a captured frame reuses the recorded value.
    int64_t E = 0;
    if (ctx->use_plan) {
        E = ctx->plan.entries;
    } else {
        LT_CUDA(ctx, cudaMemcpyAsync(&E, smp->off + S, sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
        LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        ctx->plan.entries = E;
    }
    const int64_t mr = std::max(f->max_rows, 1);
    const int R = uv->r;            // stride of the factor rows, the largest rank
    const int32_t* rk = uv->rank;   // per-slice ranks (NULL: R for every slice)
    // Slices of rank <= 16 go to the tensor-core form (CSR / CSC) or the lane-group
    // SIMT kernel (sliced layout), as tuned; the two-lines-a-warp ALS takes the others
    // (CSR / CSC); with per-slice ranks above 16 two of them run.
    const bool low = R <= 16 || rk != nullptr;
    const bool tc = low && ctx->tune.als_form == 1;
    Omega om;
    lt_status st = omega_build(ctx, f, smp, E, low && !tc, R > 16 || tc, tc, rk, R, &om);
    if (st != LT_OK) return st;
    const int RP = R <= 8 ? 8 : 16;  // the low-rank kernels cover ranks up to RP
    // per half-step retry counters (one set for ranks <= 16, one above) and the
    // float64 count
    const bool high = R > 16;
    const int nq = std::max(1, 2 * iters);
    char* sp = (char*)lt_scratch(ctx, SCR_ALS, (size_t)(3 * nq + 64) * 4 + 256, &st);
    if (!sp) return st;
    int32_t* n64 = (int32_t*)sp;
    int32_t* qcount = n64 + 64;
    int32_t* qcount_hi = qcount + nq;
    int32_t* next_hi = qcount + 2 * nq;  // line counters of k_als_half
    LT_CUDA(ctx, cudaMemsetAsync(n64, 0, (size_t)(3 * nq + 64) * 4, ctx->stream));
    const int nsm = ctx->num_sms;
    k_als_init<<<dim3(8, S), 256, 0, ctx->stream>>>(*f, *smp, om, R, rk, seed_ref(ctx, seed), uv->V);
    LT_LAUNCH_CHECK(ctx, "k_als_init");
    if (warm) {
        const size_t shm = (size_t)C * 4;
        if (shm > 48 * 1024)
            LT_CUDA(ctx, cudaFuncSetAttribute(k_als_warm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
        k_als_warm<<<S, 256, shm, ctx->stream>>>(*f, *smp, R, rk, *warm, uv->V);
        LT_LAUNCH_CHECK(ctx, "k_als_warm");
    }
    // lane-group kernel: one thread (group) per line; one 256-thread CTA per SM (its
    // registers fill the SM) stages the factor rows of its slices, each with a row of
    // zeros, and the streams' rings: up to 216 KB (3072 rows at rank 16)
    const size_t row_bytes = (size_t)RP * 4;
    const int per_sm = RP == 8 ? 2 : 1;  // rank 8 needs half the registers: two CTAs of 108 KB
    const size_t ring_bytes = 8 * kRingBytes;
    const int stage_rows = (int)((216 * 1024 / per_sm - ring_bytes) / row_bytes);
    const size_t dyn = (size_t)stage_rows * row_bytes + ring_bytes;
    const int64_t cap = std::min<int64_t>(std::max<int64_t>(f->m, (int64_t)S * C), 1 << 18);
    int64_t *qdst = nullptr, *qslot = nullptr, *qsrc = nullptr;
    int32_t *qlen = nullptr, *qgrp = nullptr, *qrank = nullptr;
    AlsQueue<32> qhi{};
    if (low || high) {
        const size_t a8 = ((size_t)cap * 8 + 255) & ~(size_t)255, a4 = ((size_t)cap * 4 + 255) & ~(size_t)255;
        const size_t set = 3 * a8 + 3 * a4;
        char* qp = (char*)lt_scratch(ctx, SCR_GRAM, 2 * set, &st);
        if (!qp) return st;
        char* hp = qp + set;  // the queue of the lines above rank 16
        qhi = AlsQueue<32>{nullptr, (int64_t*)hp, (int64_t*)(hp + a8), (int64_t*)(hp + 2 * a8),
                           (int32_t*)(hp + 3 * a8), (int32_t*)(hp + 3 * a8 + a4), (int32_t*)(hp + 3 * a8 + 2 * a4),
                           cap, ctx->d_status};
        qdst = (int64_t*)qp;
        qslot = (int64_t*)(qp + a8);
        qsrc = (int64_t*)(qp + 2 * a8);
        qlen = (int32_t*)(qp + 3 * a8);
        qgrp = (int32_t*)(qp + 3 * a8 + a4);
        qrank = (int32_t*)(qp + 3 * a8 + 2 * a4);
    }
    if (om.sell) {
        if (RP == 8)
            LT_CUDA(ctx, cudaFuncSetAttribute(k_als_line<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
        else
            LT_CUDA(ctx, cudaFuncSetAttribute(k_als_line<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
    }
    if (high) LT_CUDA(ctx, cudaFuncSetAttribute(k_als_half, cudaFuncAttributeMaxDynamicSharedMemorySize, kHalfSmem));
    TcPlan tcp{};
    if (tc) {
        st = als_tc_plan(ctx, f, smp, om, E, R, rk, RP, 2 * iters, &tcp);
        if (st != LT_OK) return st;
    }
    for (int it = 0; it < iters; ++it) {
        for (int side = 0; side < 2; ++side) {
            const bool rows = side == 0;
            const float* fin = rows ? uv->V : uv->U;
            float* fout = rows ? uv->U : uv->V;
            int32_t* cnt = qcount + 2 * it + side;
            if (tc) {
                TcQueue tq{cnt, qdst, qslot, qsrc, qlen, qgrp, qrank, cap, ctx->d_status};
                st = als_tc_half(ctx, f, smp, om, R, rk, rows, fin, fout, lam_rel, tcp, 2 * it + side, tq, nullptr);
                if (st != LT_OK) return st;
                if (RP == 8) {
                    AlsQueue<8> q{cnt, qdst, qslot, qsrc, qlen, qgrp, qrank, cap, ctx->d_status};
                    k_als_retry<8><<<nsm, 128, 0, ctx->stream>>>(q, om, rows, fin, R, lam_rel, fout, n64);
                } else {
                    AlsQueue<16> q{cnt, qdst, qslot, qsrc, qlen, qgrp, qrank, cap, ctx->d_status};
                    k_als_retry<16><<<nsm, 128, 0, ctx->stream>>>(q, om, rows, fin, R, lam_rel, fout, n64);
                }
                LT_LAUNCH_CHECK(ctx, "k_als_retry");
            } else if (om.sell && RP == 8) {
                AlsQueue<8> q{cnt, qdst, qslot, qsrc, qlen, qgrp, qrank, cap, ctx->d_status};
                k_als_line<8><<<per_sm * nsm, 256, dyn, ctx->stream>>>(*f, *smp, om, R, rk, rows, fin, fout, lam_rel, q,
                                                              stage_rows);
                LT_LAUNCH_CHECK(ctx, "k_als_line");
                k_als_retry<8><<<nsm, 128, 0, ctx->stream>>>(q, om, rows, fin, R, lam_rel, fout, n64);
                LT_LAUNCH_CHECK(ctx, "k_als_retry");
            } else if (om.sell) {
                AlsQueue<16> q{cnt, qdst, qslot, qsrc, qlen, qgrp, qrank, cap, ctx->d_status};
                k_als_line<16><<<nsm, 256, dyn, ctx->stream>>>(*f, *smp, om, R, rk, rows, fin, fout, lam_rel, q,
                                                               stage_rows);
                LT_LAUNCH_CHECK(ctx, "k_als_line");
                k_als_retry<16><<<nsm, 128, 0, ctx->stream>>>(q, om, rows, fin, R, lam_rel, fout, n64);
                LT_LAUNCH_CHECK(ctx, "k_als_retry");
            }
            if (high) {
                AlsQueue<32> q = qhi;
                q.count = qcount_hi + 2 * it + side;
                k_als_half<<<2 * nsm, 32 * kHalfWarps, kHalfSmem, ctx->stream>>>(*f, *smp, om, R, rk, lam_rel, rows, fin, fout,
                                                                            q, next_hi + 2 * it + side);
                LT_LAUNCH_CHECK(ctx, "k_als_half");
                k_als_retry<32><<<nsm, 128, 0, ctx->stream>>>(q, om, rows, fin, R, lam_rel, fout, n64);
                LT_LAUNCH_CHECK(ctx, "k_als_retry");
            }
        }
    }
    return LT_OK;
}

}  // namespace

extern "C" lt_status lt_complete(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, int32_t iters,
                                 float lam_rel, uint64_t seed, lt_factors* uv) {
    return complete_impl(ctx, f, smp, iters, lam_rel, seed, uv, nullptr);
}

extern "C" lt_status lt_complete_warm(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, int32_t iters,
                                      float lam_rel, uint64_t seed, const int32_t* prev_col_node,
                                      const int32_t* prev_ncol, const float* prev_V, lt_factors* uv) {
    if (!prev_col_node || !prev_ncol || !prev_V || (uv && prev_V == uv->V))
        return lt_fail(ctx, LT_EINVAL, "lt_complete_warm: bad arguments");
    const WarmStart w{prev_col_node, prev_ncol, prev_V};
    return complete_impl(ctx, f, smp, iters, lam_rel, seed, uv, &w);
}

extern "C" lt_status lt_als_gram(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, const lt_factors* uv,
                                 int32_t side, float* gram) {
    if (!ctx || !frame_ok2(f) || !smp || !smp->key || !smp->val || !smp->off || !smp->cnt || !smp->ncol || !uv ||
        !uv->U || !uv->V || uv->r < 1 || uv->r > 16 || uv->rank || (side != 0 && side != 1) || !gram)
        return lt_fail(ctx, LT_EINVAL, "lt_als_gram: bad arguments");
    cudaSetDevice(ctx->device);
    int64_t E = 0;
    LT_CUDA(ctx, cudaMemcpyAsync(&E, smp->off + f->S, sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
    LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    Omega om;
    lt_status st = omega_build(ctx, f, smp, E, false, true, true, nullptr, uv->r, &om);
    if (st != LT_OK) return st;
    const int R = uv->r, RP = R <= 8 ? 8 : 16;
    TcPlan tcp{};
    st = als_tc_plan(ctx, f, smp, om, E, R, nullptr, RP, 1, &tcp);
    if (st != LT_OK) return st;
    const TcQueue none{};
    return als_tc_half(ctx, f, smp, om, R, nullptr, side == 0, side == 0 ? uv->V : uv->U, nullptr, 0.f, tcp, 0, none,
                       gram);
}

extern "C" lt_status lt_complete_fp64_lines(lt_ctx* ctx, int64_t* count_host) {
    if (!ctx || !count_host) return lt_fail(ctx, LT_EINVAL, "lt_complete_fp64_lines: bad arguments");
    *count_host = 0;
    if (!ctx->scr[SCR_ALS]) return LT_OK;  // no lt_complete ran on this context yet
    cudaSetDevice(ctx->device);
    int32_t v = 0;  // word 0 of the ALS scratch: the float64 count of the last lt_complete
    LT_CUDA(ctx, cudaMemcpyAsync(&v, ctx->scr[SCR_ALS], sizeof(v), cudaMemcpyDeviceToHost, ctx->stream));
    LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    *count_host = v;
    return LT_OK;
}

extern "C" lt_status lt_slice_ranks(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, int32_t R, int32_t cols,
                                    int32_t* rank) {
    if (!ctx || !frame_ok2(f) || !smp || !smp->ncol || !rank || R < 1 || R > 32 || cols < 1)
        return lt_fail(ctx, LT_EINVAL, "lt_slice_ranks: bad arguments");
    cudaSetDevice(ctx->device);
    k_slice_ranks<<<(f->S + 255) / 256, 256, 0, ctx->stream>>>(*smp, f->S, R, cols, rank);
    LT_LAUNCH_CHECK(ctx, "k_slice_ranks");
    return LT_OK;
}

extern "C" lt_status lt_render(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, const lt_factors* uv,
                               const float* w, const int32_t* row_perm, float* img) {
    if (!ctx || !frame_ok2(f) || !smp || !smp->ncol || !uv || !uv->U || !uv->V || uv->r < 1 || uv->r > 32 ||
        !row_perm || !img)
        return lt_fail(ctx, LT_EINVAL, "lt_render: bad arguments");
    cudaSetDevice(ctx->device);
    const int per = std::max(1, std::min(64, (int)((f->max_rows + 511) / 512)));
    k_render<<<dim3(per, f->S), 512, 0, ctx->stream>>>(*f, *smp, uv->U, uv->V, uv->r, w, row_perm, img);
    LT_LAUNCH_CHECK(ctx, "k_render");
    return LT_OK;
}
