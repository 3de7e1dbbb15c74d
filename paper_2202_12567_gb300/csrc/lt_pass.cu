// Sampling passes of the sparse renderer.
//
//  * Pass 1 and light coarsening (Sec. 4, Eq. 2): the cut nodes of every slice draw
//    their k_c rows and evaluate them (one kernel over all slices), then the cut's
//    ancestor forest is walked level by level with two kernels per level over all
//    slices.  One group of lanes (8, a warp or a CTA by the pair's rows) handles a
//    sibling pair from end to end: the union zeta_f = zeta_a U zeta_b, the entries
//    missing from either child, and the merge when cost = eps + cost(q) < tau * S_hat,
//    eps = max |V_q - V_p I_q / I_p| (in a dark slice, S_hat = 0, when the cost is
//    exactly zero).
//  * Pass 2 (Sec. 5, Eq. 3): per slice one cluster of eight CTAs draws (column from
//    the integer CDF of g or of given weights, row uniform) in rounds, keeps the
//    first occurrence of every new entry in draw order, and stops at
//    ceil(rate m' n') entries.
//  * Entry evaluation: one thread per pass-2 entry (one shadow ray), the column side
//    read from per-frame column records (k_col_records).
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include "lt_internal.cuh"

using namespace ltk;

namespace {

constexpr int kP1Threads = 1024;
constexpr int kMaxRowsPerNode = 64;
constexpr int kMaxDraws = 1 << 16;
constexpr int kMaxCut = 16384;
constexpr int kStNot = 0, kStAlive = 1, kStDead = 2, kStRejected = 3;

struct P1Plan {
    int32_t* k;        // [S][C]   rows per cut node
    int32_t* cap;      // [S][NF]  storage capacity per forest node
    int32_t* off;      // [S][NF]  storage offset inside the slice's region
    int32_t* cnt;      // [S][NF]  current |zeta|
    int32_t* state;    // [S][NF]
    float* cost;       // [S][NF]
    int32_t* pfx;      // [S][C+1] prefix of k
    int32_t* colx;     // [S][C]   forest node of each output column
    int32_t* eoff;     // [S][C]   output offset of each column
    int64_t* total;    // [S]      storage slots of the slice
    int64_t* base;     // [S]      start of the slice's storage
};

__device__ __forceinline__ float node_scale(const lt_tree& T, const float4* __restrict__ vpls, int64_t n, int node) {
    const int r = T.rep[node];
    const float flux = __ldg(&vpls[2 * n + r].w);
    const float alb = __ldg(&vpls[r].w);
    return __fdiv_rn(T.I[node], __fmul_rn(flux, alb));
}

// ------------------------------------------------------------------ pass 1: plan
// Each thread has a run of the cut's nodes, then of the forest's: one scan each (chunks of
// 512 with a scan per chunk: 53 us on 64 slices of a cut of 4600 nodes; 40 us so).
__global__ void __launch_bounds__(kP1Threads) k_pass1_plan(lt_frame F, float rate1, P1Plan pl) {
    __shared__ int32_t ws[32];
    const int s = blockIdx.x;
    const int C = F.C, NF = 2 * C - 1;
    const int ms = F.slice_off[s + 1] - F.slice_off[s];
    int32_t* k = pl.k + (int64_t)s * C;
    int32_t* cap = pl.cap + (int64_t)s * NF;
    int32_t* off = pl.off + (int64_t)s * NF;
    int32_t* pfx = pl.pfx + (int64_t)s * (C + 1);
    const float kappa = fmaxf(2.0f, __fmul_rn(rate1, (float)ms));
    const float Iroot = F.tree.I[0];
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        const int node = F.forest[8 * c];
        const float x = __fmul_rn(__fmul_rn(kappa, (float)C), __fdiv_rn(F.tree.I[node], Iroot));
        int kc = (int)floorf(__fadd_rn(x, 0.5f));
        kc = min(max(kc, 2), kMaxRowsPerNode);
        kc = min(kc, ms);
        k[c] = kc;
    }
    __syncthreads();
    {
        const int run = (C + blockDim.x - 1) / blockDim.x, lo = min(C, (int)threadIdx.x * run), hi = min(C, lo + run);
        int sum = 0, K;
        for (int c = lo; c < hi; ++c) sum += k[c];
        int at = block_exclusive_scan<int>(sum, ws, &K);
        for (int c = lo; c < hi; ++c) {
            pfx[c] = at;
            at += k[c];
        }
        if (threadIdx.x == 0) pfx[C] = K;
    }
    __syncthreads();
    for (int x = threadIdx.x; x < NF; x += blockDim.x) {
        const int* fx = F.forest + 8 * x;
        cap[x] = x < C ? k[x] : min(ms, pfx[fx[5] + 1] - pfx[fx[4]]);
    }
    __syncthreads();
    const int run = (NF + blockDim.x - 1) / blockDim.x, lo = min(NF, (int)threadIdx.x * run), hi = min(NF, lo + run);
    int sum = 0, tot;
    for (int x = lo; x < hi; ++x) sum += cap[x];
    int at = block_exclusive_scan<int>(sum, ws, &tot);
    for (int x = lo; x < hi; ++x) {
        off[x] = at;
        at += cap[x];
    }
    if (threadIdx.x == 0) pl.total[s] = tot;
}

// ------------------------------------------------------------------ pass 1: flat kernels
// Every step below runs over all slices at once.  Per forest level a testable sibling
// pair is handled from end to end by one group of lanes: the union of the two sorted
// row lists (the slot of a row is its rank in its own list plus its rank in the other
// less the rows in both), one shadow ray per row that only one child holds, eps over
// the union, Eq. 2, and the merge.  Pairs of up to kSmallPair rows take 8 lanes, of up
// to kMidPair a warp, bigger ones a CTA.  A level is two launches (small pairs, which
// also list the others; then the others), or two steps of one persistent cooperative
// launch with grid-wide barriers (k_p1_walk).  What bounds it: latency (dependent loads,
// then the rays of a pair).  Against five launches a level with the missing entries in a
// queue and a serial merge per small pair: the 64x64 frame 1.71 to 1.19 ms (1.01 ms with
// a CTA per listed pair where they are few, 0.95 ms with one record per forest node), the
// sampling of the 512x512 scene with 1000 boxes 7.1 to 5.1, then 4.7 ms.

struct P1Store {
    int32_t* rows;     // [total] row of each storage slot
    float* v0;         // [total]  (V_a, or V_f after a merge)
    float* v1;         // [total]  (V_b), == v0 + total
    float* v2;         // [total]  V_a kept at a merge (coarsening to a target size), else null
    int64_t total;
};

struct P1Work {
    int64_t* kpfx;     // [S+1] prefix over slices of the initial entry counts
    float* leafmean;   // [S][C] mean of each cut node's initial entries
    float* thr;        // [S] tau * S_hat (-1 in a dark slice, S_hat = 0)
    float4* nrec;      // [NF][4] per forest node: its representative's planes, then (scale, I, 0, 0)
    int64_t* mcount;   // [Hmax] pairs of a warp per level
    int64_t* bcount;   // [Hmax] pairs of a CTA per level
    int64_t* mnext;    // [Hmax] the next pair of a warp to take
    int64_t* mid;      // [bcap] flat pair index of a warp's pair
    int64_t* big;      // [bcap] flat pair index of a CTA's pair
    unsigned* bar;     // arrival counter of the persistent walk's grid barriers
    int64_t bcap;
};

// -- what an entry or a pair reads of a forest node, in one 64-byte record
__global__ void k_p1_nodes(lt_frame F, float4* __restrict__ nrec) {
    const float4* vpls = reinterpret_cast<const float4*>(F.vpls);
    const int NF = 2 * F.C - 1;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < NF; x += gridDim.x * blockDim.x) {
        const int node = F.forest[8 * x];
        const PointRec L = load_rec(vpls, F.n, F.tree.rep[node]);
        nrec[4 * x] = L.a;
        nrec[4 * x + 1] = L.b;
        nrec[4 * x + 2] = L.c;
        nrec[4 * x + 3] = make_float4(node_scale(F.tree, vpls, F.n, node), F.tree.I[node], 0.f, 0.f);
    }
}

// -- draws of the cut nodes and state of every forest node.  A node's rows are the first
// k distinct draws, ascending.  Up to kSerialDraws rows a thread draws for its node; for
// more the warp does it, 32 draws at a time (a serial search and an insertion sort of
// up to 64 rows cost 0.65 ms on the 512x512 scene with about 30 rows a node).
constexpr int kSerialDraws = 4;

__global__ void __launch_bounds__(256) k_p1_draws(lt_frame F, SeedRef sr, P1Plan pl, P1Store st, int32_t* status) {
    __shared__ int32_t got_rows[8][kMaxRowsPerNode];
    const unsigned FULL = 0xffffffffu;
    const int C = F.C, NF = 2 * C - 1;
    const uint64_t seed = sr.get();
    const int lane = threadIdx.x & 31;
    int32_t* mine = got_rows[threadIdx.x >> 5];
    const int64_t total = (int64_t)F.S * NF;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x; i0 < total; i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t idx = i0 + threadIdx.x;
        const bool in = idx < total;
        const int s = in ? (int)(idx / NF) : 0, x = in ? (int)(idx % NF) : 0;
        const int ms = F.slice_off[s + 1] - F.slice_off[s];
        const int k = in && x < C ? pl.k[(int64_t)s * C + x] : 0;
        int32_t* r = st.rows;
        if (in) {
            pl.cost[(int64_t)s * NF + x] = 0.f;
            pl.state[(int64_t)s * NF + x] = x < C && ms > 0 ? kStAlive : kStNot;
            if (x < C) r += pl.base[s] + pl.off[(int64_t)s * NF + x];
            else pl.cnt[(int64_t)s * NF + x] = 0;
        }
        const bool node = in && x < C;
        const bool wide = node && k < ms && k > kSerialDraws;
        if (node && !wide) {
            int got = 0;
            if (k >= ms) {
                for (int t = 0; t < ms; ++t) r[t] = t;
                got = ms;
            } else {
                int v[kSerialDraws];  // ascending
                for (int t = 0; got < k && t < kMaxDraws; ++t) {
                    int u = (int)uniform_index(
                        philox((uint32_t)t, (uint32_t)x, slice_key(F.slice_id, s), kTagPass1, seed).x, (uint32_t)ms);
                    bool dup = false;
#pragma unroll
                    for (int q = 0; q < kSerialDraws; ++q) dup |= q < got && v[q] == u;
                    if (dup) continue;
                    ++got;
#pragma unroll
                    for (int q = 0; q < kSerialDraws; ++q) {
                        if (q >= got) continue;
                        if (q == got - 1 || u < v[q]) {  // insert u, carry what it displaces
                            const int w = q == got - 1 ? u : v[q];
                            v[q] = u;
                            u = w;
                        }
                    }
                }
                if (got < k) latch(status, LT_ELIMIT);
#pragma unroll
                for (int q = 0; q < kSerialDraws; ++q)
                    if (q < got) r[q] = v[q];
            }
            pl.cnt[(int64_t)s * NF + x] = got;
        }
        for (unsigned left = __ballot_sync(FULL, wide); left; left &= left - 1) {
            const int src = __ffs(left) - 1;
            const int ws = __shfl_sync(FULL, s, src), wx = __shfl_sync(FULL, x, src), wk = __shfl_sync(FULL, k, src);
            const uint32_t wm = (uint32_t)__shfl_sync(FULL, ms, src);
            int got = 0;
            for (int t0 = 0; got < wk && t0 < kMaxDraws; t0 += 32) {
                const int v = (int)uniform_index(
                    philox((uint32_t)(t0 + lane), (uint32_t)wx, slice_key(F.slice_id, ws), kTagPass1, seed).x, wm);
                bool fresh = __ffs(__match_any_sync(FULL, v)) - 1 == lane;  // the first of its value in the batch
                for (int q = 0; q < got; ++q) fresh &= mine[q] != v;
                const unsigned b = __ballot_sync(FULL, fresh);
                const int pos = got + __popc(b & ((1u << lane) - 1u));
                __syncwarp();  // every lane has read the list
                if (fresh && pos < wk) mine[pos] = v;
                got = min(wk, got + __popc(b));
                __syncwarp();
            }
            if (got < wk && lane == 0) latch(status, LT_ELIMIT);
            int32_t* wr = st.rows + pl.base[ws] + pl.off[(int64_t)ws * NF + wx];
            for (int e = lane; e < got; e += 32) {  // a row's place is the number of smaller ones
                const int v = mine[e];
                int rank = 0;
                for (int q = 0; q < got; ++q) rank += mine[q] < v;
                wr[rank] = v;
            }
            if (lane == 0) pl.cnt[(int64_t)ws * NF + wx] = got;
            __syncwarp();
        }
    }
}

// -- first row slot of every slice: exclusive prefix of the per-slice totals
__global__ void k_p1_base(int S, P1Plan pl) {
    __shared__ int64_t ws[32];
    int64_t carry = 0;
    for (int c0 = 0; c0 < S; c0 += blockDim.x) {
        const int s = c0 + threadIdx.x;
        const int64_t x = s < S ? pl.total[s] : 0;
        int64_t tot;
        const int64_t pre = block_exclusive_scan<int64_t>(x, ws, &tot);
        if (s < S) pl.base[s] = carry + pre;
        carry += tot;
    }
}

__global__ void k_p1_kpfx(lt_frame F, P1Plan pl, int64_t* kpfx) {
    __shared__ int64_t ws[32];
    int64_t carry = 0;
    for (int c0 = 0; c0 < F.S; c0 += blockDim.x) {
        const int s = c0 + threadIdx.x;
        const int64_t x = s < F.S ? (int64_t)pl.pfx[(int64_t)s * (F.C + 1) + F.C] : 0;
        int64_t tot;
        const int64_t pre = block_exclusive_scan<int64_t>(x, ws, &tot);
        if (s < F.S) kpfx[s] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) kpfx[F.S] = carry;
}

// -- initial entries of every cut node of every slice (one shadow ray per thread)
__global__ void __launch_bounds__(128) k_p1_initial(lt_frame F, Grid g, float dmin2, P1Plan pl, P1Store st,
                                                    const int64_t* __restrict__ kpfx,
                                                    const float4* __restrict__ nrec, int32_t* status) {
    const float4* pts = reinterpret_cast<const float4*>(F.pts);
    const int C = F.C, NF = 2 * C - 1;
    const int64_t total = kpfx[F.S];
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = F.S;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (kpfx[mid] <= idx) lo = mid;
            else hi = mid;
        }
        const int s = lo;
        const int e = (int)(idx - kpfx[s]);
        const int32_t* pf = pl.pfx + (int64_t)s * (C + 1);
        int a = 0, b = C;  // largest c with pf[c] <= e
        while (b - a > 1) {
            const int mid = (a + b) >> 1;
            if (pf[mid] <= e) a = mid;
            else b = mid;
        }
        const int c = a, t = e - pf[c];
        const int64_t slot = pl.base[s] + pl.off[(int64_t)s * NF + c] + t;
        const PointRec P = load_rec(pts, F.m, F.slice_off[s] + st.rows[slot]);
        const PointRec L = {nrec[4 * c], nrec[4 * c + 1], nrec[4 * c + 2]};
        const float v = entry_value(P, L, nrec[4 * c + 3].x, dmin2, g);
        if (!isfinite(v)) latch(status, LT_ENUMERIC);  // a non-finite input (flux, albedo, position)
        st.v0[slot] = v;
    }
}

__global__ void k_p1_leafmean(lt_frame F, P1Plan pl, P1Store st, float* leafmean) {
    const int C = F.C, NF = 2 * C - 1;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)F.S * C;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int s = (int)(idx / C), c = (int)(idx % C);
        const int n = pl.cnt[(int64_t)s * NF + c];
        const float* v = st.v0 + pl.base[s] + pl.off[(int64_t)s * NF + c];
        float sum = 0.f;
        for (int t = 0; t < n; ++t) sum += v[t];
        leafmean[idx] = n > 0 ? sum / (float)n : 0.f;
    }
}

// tau * S_hat per slice, S_hat = sum_c mean(V_c) (fixed reduction order).  A dark
// slice (S_hat = 0: every pass-1 entry is zero) gets -1: its relative bound is zero,
// and it is read as met by a pair whose cost is exactly zero (the samples cannot
// tell the two lights apart), so such a slice coarsens as far as its entries agree.
__global__ void k_p1_thr(lt_frame F, const float* __restrict__ leafmean, float tau, float* thr) {
    __shared__ float red[32];
    const int s = blockIdx.x;
    float sum = 0.f;
    for (int c = threadIdx.x; c < F.C; c += blockDim.x) sum += leafmean[(int64_t)s * F.C + c];
    sum = warp_sum(sum);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        thr[s] = t > 0.f ? tau * t : -1.f;
    }
}

// -- coarsening to a target cut size (Sec. 4): every pair is tested (threshold +inf,
// so all merge and every internal node gets its cost); then per slice the C - target
// pairs of smallest effective cost eff(f) = max(cost(f), eff(a), eff(b)) (ties: lower
// height, lower id) are the merged ones.  Merging by least cost among the testable
// pairs, one at a time, merges exactly those: a pair becomes testable only after its
// children merged, and the effective cost is the cost at which the greedy order
// reaches it.
__global__ void k_p1_thr_inf(int S, float* thr) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) thr[s] = INFINITY;
}

__device__ __forceinline__ unsigned long long eff_key(const lt_frame& F, const float* eff, int f) {
    return (unsigned long long)__float_as_uint(eff[f]) << 32 | (unsigned long long)F.forest[8 * f + 6] << 20 |
           (unsigned long long)(f - F.C);
}

__global__ void __launch_bounds__(1024) k_p1_target(lt_frame F, P1Plan pl, float* __restrict__ effs, int target) {
    __shared__ int32_t hist[256];
    __shared__ unsigned long long sel[2];
    __shared__ int32_t krem;
    const int s = blockIdx.x;
    const int C = F.C, NF = 2 * C - 1;
    const int ms = F.slice_off[s + 1] - F.slice_off[s];
    if (ms == 0) return;
    const float* cost = pl.cost + (int64_t)s * NF;
    int32_t* state = pl.state + (int64_t)s * NF;
    float* eff = effs + (int64_t)s * NF;
    for (int x = threadIdx.x; x < C; x += blockDim.x) eff[x] = 0.f;
    __syncthreads();
    for (int h = 1; h <= F.H; ++h) {
        for (int i = F.level_off[h] + threadIdx.x; i < F.level_off[h + 1]; i += blockDim.x) {
            const int f = F.level_nodes[i];
            eff[f] = fmaxf(cost[f], fmaxf(eff[F.forest[8 * f + 1]], eff[F.forest[8 * f + 2]]));
        }
        __syncthreads();
    }
    const int K = max(0, min(C - target, C - 1));
    if (threadIdx.x == 0) {
        sel[0] = sel[1] = 0ull;
        krem = K - 1;
    }
    __syncthreads();
    for (int pass = 7; pass >= 0 && K > 0; --pass) {  // radix select of the K-th smallest key
        for (int b = threadIdx.x; b < 256; b += blockDim.x) hist[b] = 0;
        __syncthreads();
        const unsigned long long prefix = sel[0], mask = sel[1];
        for (int f = C + threadIdx.x; f < NF; f += blockDim.x) {
            const unsigned long long key = eff_key(F, eff, f);
            if ((key & mask) == prefix) atomicAdd(&hist[(key >> (8 * pass)) & 255], 1);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int k = krem, digit = 255;
            for (int b = 0; b < 256; ++b) {
                if (k < hist[b]) {
                    digit = b;
                    break;
                }
                k -= hist[b];
            }
            krem = k;
            sel[0] = prefix | ((unsigned long long)digit << (8 * pass));
            sel[1] = mask | (255ull << (8 * pass));
        }
        __syncthreads();
    }
    const unsigned long long pivot = sel[0];
    auto merged = [&](int x) { return x >= C && K > 0 && eff_key(F, eff, x) <= pivot; };
    for (int x = threadIdx.x; x < NF; x += blockDim.x) {
        const bool chosen = x < C || merged(x);
        const int par = F.forest[8 * x + 3];
        int stt;
        if (chosen) {
            stt = (par >= 0 && merged(par)) ? kStDead : kStAlive;
        } else {
            const int a = F.forest[8 * x + 1], b = F.forest[8 * x + 2];
            const bool ca = a < C || merged(a), cb = b < C || merged(b);
            stt = (ca && cb) ? kStRejected : kStNot;
        }
        state[x] = stt;
    }
}

struct PairCtx {
    int s, f, a, b, na, nb, row0;
    int64_t base;
    const int32_t* ra;
    const int32_t* rb;
    int64_t ia, ib, iff;   // storage offsets of a, b, f inside the slice's region
};

__device__ __forceinline__ bool load_pair(const lt_frame& F, const P1Plan& pl, const P1Store& st, int h, int64_t t,
                                          PairCtx& pc) {
    const int l0 = F.level_off[h], np = F.level_off[h + 1] - l0;
    const int NF = 2 * F.C - 1;
    // (a frame has fewer than 2^32 pairs a level: S <= 1024 where the completions take it, C <= 16384;
    // larger S goes the long way)
    if (t <= 0xffffffffll) {
        const uint32_t q = (uint32_t)t / (uint32_t)np;
        pc.s = (int)q;
        pc.f = F.level_nodes[l0 + (int)((uint32_t)t - q * (uint32_t)np)];
    } else {
        pc.s = (int)(t / np);
        pc.f = F.level_nodes[l0 + (int)(t % np)];
    }
    pc.a = F.forest[8 * pc.f + 1];
    pc.b = F.forest[8 * pc.f + 2];
    const int32_t* state = pl.state + (int64_t)pc.s * NF;
    if (state[pc.a] != kStAlive || state[pc.b] != kStAlive) return false;
    const int32_t* cnt = pl.cnt + (int64_t)pc.s * NF;
    const int32_t* off = pl.off + (int64_t)pc.s * NF;
    pc.na = cnt[pc.a];
    pc.nb = cnt[pc.b];
    pc.base = pl.base[pc.s];
    pc.ia = pc.base + off[pc.a];
    pc.ib = pc.base + off[pc.b];
    pc.iff = pc.base + off[pc.f];
    pc.ra = st.rows + pc.ia;
    pc.rb = st.rows + pc.ib;
    pc.row0 = F.slice_off[pc.s];
    return true;
}

// -- one level: pairs of a group of lanes
// (64x64 frame / sampling of the 512x512 scene, ms: small pairs up to 8 rows 0.95 / 4.64,
// 16: 0.96 / 4.64, 32: 1.00 / 4.77, 64: 1.02 / 5.0; warp pairs up to 128 rows 5% slower on the
// latter than 256, 512 2%)
constexpr int kSmallPair = 16;   // rows of both children: 8 lanes, at most 2 rows a lane
constexpr int kMidPair = 256;    // a warp, at most 8 rows a lane
constexpr int kGroup = 8;

__device__ __forceinline__ float pair_entry(const lt_frame& F, const Grid& g, float dmin2, int row, const float4* rec,
                                            int32_t* status) {
    const PointRec P = load_rec(reinterpret_cast<const float4*>(F.pts), F.m, row);
    const PointRec L = {rec[0], rec[1], rec[2]};
    const float v = entry_value(P, L, rec[3].x, dmin2, g);
    if (!isfinite(v)) latch(status, LT_ENUMERIC);
    return v;
}

// The ratios of a pair (Sec. 4): q is estimated from p, the child whose representative
// the parent takes.
struct PairRatio {
    bool p_is_a;
    float rq;   // I_q / I_p
    float rfp;  // I_f / I_p
};

__device__ __forceinline__ PairRatio pair_ratio(const float4* __restrict__ nrec, const PairCtx& pc) {
    PairRatio r;
    const float Ia = nrec[4 * pc.a + 3].y, Ib = nrec[4 * pc.b + 3].y, If = nrec[4 * pc.f + 3].y;
    r.p_is_a = Ia >= Ib;
    r.rq = r.p_is_a ? __fdiv_rn(Ib, Ia) : __fdiv_rn(Ia, Ib);
    r.rfp = __fdiv_rn(If, r.p_is_a ? Ia : Ib);
    return r;
}

// One row of the union: element t of the concatenated lists (t < na: row t of a, else row
// t - na of b), its place p in the other list and whether the other holds it too.
struct PairRow {
    int x, p;
    bool in_a, in_b, both;
};

__device__ __forceinline__ PairRow pair_row(const int32_t* A, int na, const int32_t* B, int nb, int t) {
    PairRow r;
    r.in_a = t < na;
    r.in_b = !r.in_a && t < na + nb;
    r.x = 0;
    r.p = 0;
    r.both = false;
    if (r.in_a || r.in_b) {
        const int32_t* O = r.in_a ? B : A;
        const int no = r.in_a ? nb : na;
        r.x = r.in_a ? A[t] : B[t - na];
        r.p = lower_bound<int32_t>(O, no, r.x);
        r.both = r.p < no && O[r.p] == r.x;
    }
    return r;
}

// Values of a row for both children (the missing one evaluated), stored at `slot`;
// returns |V_q - V_p I_q / I_p|.
__device__ __forceinline__ float pair_put(const lt_frame& F, const Grid& g, float dmin2, const P1Store& st,
                                          const PairCtx& pc, const PairRatio& pr, const float4* rec_a,
                                          const float4* rec_b, const PairRow& r, int t, int slot, int32_t* status) {
    const float own = st.v0[r.in_a ? pc.ia + t : pc.ib + (t - pc.na)];
    const float oth = r.both ? st.v0[pc.ib + r.p]
                             : pair_entry(F, g, dmin2, pc.row0 + r.x, r.in_a ? rec_b : rec_a, status);
    const float va = r.in_a ? own : oth, vb = r.in_a ? oth : own;
    st.rows[pc.iff + slot] = r.x;
    st.v0[pc.iff + slot] = va;
    st.v1[pc.iff + slot] = vb;
    const float vp = pr.p_is_a ? va : vb, vq = pr.p_is_a ? vb : va;
    return fabsf(vq - vp * pr.rq);
}

// Cost (Eq. 2), merge or reject; `first`, `step`: this thread's slots of the union.
__device__ __forceinline__ void decide_pair(const lt_frame& F, const P1Plan& pl, const P1Store& st, const float* thr,
                                            const PairCtx& pc, const PairRatio& pr, int nf, float e_max, int first,
                                            int step, bool writer) {
    const int NF = 2 * F.C - 1;
    float* cost = pl.cost + (int64_t)pc.s * NF;
    int32_t* state = pl.state + (int64_t)pc.s * NF;
    const float cf = e_max + cost[pr.p_is_a ? pc.b : pc.a];
    const float th = thr[pc.s];
    const bool merge = th < 0.f ? cf == 0.f : cf < th;  // th < 0: a dark slice
    if (merge) {
        float* fa = st.v0 + pc.iff;
        const float* fb = st.v1 + pc.iff;
        float* keep = st.v2 ? st.v2 + pc.iff : nullptr;
        for (int t = first; t < nf; t += step) {
            if (keep) keep[t] = fa[t];
            fa[t] = (pr.p_is_a ? fa[t] : fb[t]) * pr.rfp;
        }
    }
    if (writer) {
        pl.cnt[(int64_t)pc.s * NF + pc.f] = nf;
        cost[pc.f] = cf;
        state[pc.f] = merge ? kStAlive : kStRejected;
        if (merge) {
            state[pc.a] = kStDead;
            state[pc.b] = kStDead;
        }
    }
}

// One pair by each group of G lanes of the warp (every lane of the warp calls it; `live`
// is uniform in a group).  The trip count is the warp's largest, so that the groups'
// shadow rays run side by side.
template <int G>
__device__ __forceinline__ void group_pair(const lt_frame& F, const Grid& g, float dmin2, const P1Plan& pl,
                                           const P1Store& st, const P1Work& w, const PairCtx& pc, const int32_t* A,
                                           const int32_t* B, bool live, int32_t* status) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, gl = lane & (G - 1), sh = lane & ~(G - 1);
    const unsigned gm = G == 32 ? FULL : (1u << G) - 1u, lt = (1u << gl) - 1u;
    const int na = live ? pc.na : 0, nb = live ? pc.nb : 0;
    PairRatio pr{};
    if (live) pr = pair_ratio(w.nrec, pc);
    const int trips = (__reduce_max_sync(FULL, na + nb) + G - 1) / G;
    int ca = 0, cb = 0;  // rows of a (of b) so far that both children hold
    float e = 0.f;
    for (int it = 0; it < trips; ++it) {
        const int t = it * G + gl;
        const PairRow r = pair_row(A, na, B, nb, t);
        const unsigned ma = (__ballot_sync(FULL, r.in_a && r.both) >> sh) & gm;
        const unsigned mb = (__ballot_sync(FULL, r.in_b && r.both) >> sh) & gm;
        if (r.in_a || (r.in_b && !r.both)) {
            const int slot = r.in_a ? t + r.p - (ca + __popc(ma & lt)) : t - na + r.p - (cb + __popc(mb & lt));
            e = fmaxf(e, pair_put(F, g, dmin2, st, pc, pr, w.nrec + 4 * pc.a, w.nrec + 4 * pc.b, r, t, slot, status));
        }
        ca += __popc(ma);
        cb += __popc(mb);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) e = fmaxf(e, __shfl_xor_sync(FULL, e, o));
    __syncwarp();  // the group's stores are visible to the group
    if (live) decide_pair(F, pl, st, w.thr, pc, pr, na + nb - ca, e, gl, G, gl == 0);
}

// step 1: the pairs of at most kSmallPair rows, 8 lanes each; the others are listed
__device__ __forceinline__ void p1_small_body(const lt_frame& F, const Grid& g, float dmin2, const P1Plan& pl,
                                              const P1Store& st, const P1Work& w, int h, int32_t* status) {
    const int np = F.level_off[h + 1] - F.level_off[h];
    const int64_t npairs = (int64_t)F.S * np;
    const int lane = threadIdx.x & 31;
    const int per = blockDim.x / kGroup;
    for (int64_t t0 = blockIdx.x * (int64_t)per; t0 < npairs; t0 += (int64_t)gridDim.x * per) {  // block-uniform
        const int64_t t = t0 + threadIdx.x / kGroup;
        PairCtx pc{};
        const bool active = t < npairs && load_pair(F, pl, st, h, t, pc);
        const int rows = pc.na + pc.nb;
        const bool mid = active && rows > kSmallPair && rows <= kMidPair, big = active && rows > kMidPair;
        const bool head = (lane & (kGroup - 1)) == 0;
        const unsigned bm = __ballot_sync(0xffffffffu, mid && head), bb = __ballot_sync(0xffffffffu, big && head);
        for (int kind = 0; kind < 2; ++kind) {
            const unsigned b = kind ? bb : bm;
            if (b == 0) continue;  // warp-uniform
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd((unsigned long long*)(kind ? w.bcount : w.mcount) + h,
                                            (unsigned long long)__popc(b));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (head && (kind ? big : mid)) {
                const int64_t q = (int64_t)base + __popc(b & ((1u << lane) - 1u));
                if (q < w.bcap) (kind ? w.big : w.mid)[q] = t;
                else latch(status, LT_ELIMIT);
            }
        }
        group_pair<kGroup>(F, g, dmin2, pl, st, w, pc, pc.ra, pc.rb, active && rows <= kSmallPair, status);
    }
}

// step 2: the listed pairs.  A CTA per pair of more than kMidPair rows (both row lists
// staged in shared memory when they fit), then a warp per pair; where a level has few
// pairs (at most kFewPairs per CTA), a CTA each for those too: with a warp, a level waits
// for eight shadow rays one after the other.  (64x64 frame 1.08 ms with kFewPairs 0, 1.01
// with 4, 1.02 with 16.)  Pairs differ in their rows and rays: the warps take theirs from a
// counter and stage both row lists before they search them (sampling of the 512x512 scene
// 4.64 ms with fixed shares and searches in memory, 4.16 so; the CTAs' pairs from a counter
// cost the 64x64 frame 1%).
constexpr int kBigStage = 4096;
constexpr int kFewPairs = 4;

__device__ __forceinline__ void p1_rest_body(const lt_frame& F, const Grid& g, float dmin2, const P1Plan& pl,
                                             const P1Store& st, const P1Work& w, int h, int32_t* status) {
    __shared__ int32_t stage[2 * kBigStage];
    int32_t *sa = stage, *sb = stage + kBigStage;
    __shared__ int32_t ws[32];
    __shared__ float red[32];
    // the CTA's pair: in shared memory, the registers are for the rays
    __shared__ PairCtx pc;
    __shared__ PairRatio pr;
    __shared__ float4 rec[8];
    __shared__ int s_live;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t nbig = min(w.bcount[h], w.bcap), nmid = min(w.mcount[h], w.bcap);
    const bool few = nmid <= (int64_t)kFewPairs * gridDim.x;
    for (int64_t q = blockIdx.x; q < nbig + (few ? nmid : 0); q += gridDim.x) {
        __syncthreads();  // the previous pair is done with the shared state
        if (threadIdx.x == 0) {
            s_live = load_pair(F, pl, st, h, q < nbig ? w.big[q] : w.mid[q - nbig], pc);
            if (s_live) pr = pair_ratio(w.nrec, pc);
        }
        __syncthreads();
        if (!s_live) continue;
        const bool staged = pc.na <= kBigStage && pc.nb <= kBigStage;
        if (threadIdx.x < 8) rec[threadIdx.x] = w.nrec[4 * (threadIdx.x < 4 ? pc.a : pc.b) + (threadIdx.x & 3)];
        if (staged) {
            for (int i = threadIdx.x; i < pc.na; i += blockDim.x) sa[i] = pc.ra[i];
            for (int j = threadIdx.x; j < pc.nb; j += blockDim.x) sb[j] = pc.rb[j];
        }
        __syncthreads();
        const int32_t* A = staged ? sa : pc.ra;
        const int32_t* B = staged ? sb : pc.rb;
        int ca = 0, cb = 0;
        float e = 0.f;
        for (int t0 = 0; t0 < pc.na + pc.nb; t0 += blockDim.x) {
            const int t = t0 + threadIdx.x;
            const PairRow r = pair_row(A, pc.na, B, pc.nb, t);
            int tot;  // rows of a in the low half, of b in the high half (a block is at most 1024)
            const int pre = block_exclusive_scan<int>(r.both ? (r.in_a ? 1 : 1 << 16) : 0, ws, &tot);
            if (r.in_a || (r.in_b && !r.both)) {
                const int slot = r.in_a ? t + r.p - (ca + (pre & 0xffff)) : t - pc.na + r.p - (cb + (pre >> 16));
                e = fmaxf(e, pair_put(F, g, dmin2, st, pc, pr, rec, rec + 4, r, t, slot, status));
            }
            ca += tot & 0xffff;
            cb += tot >> 16;
        }
        e = warp_max(e);
        if (lane == 0) red[wid] = e;
        __syncthreads();  // also the block's stores before decide_pair reads them
        float em = 0.f;
        for (int k = 0; k < nw; ++k) em = fmaxf(em, red[k]);
        decide_pair(F, pl, st, w.thr, pc, pr, pc.na + pc.nb - ca, em, threadIdx.x, blockDim.x, threadIdx.x == 0);
    }
    if (few) return;
    __syncthreads();  // the stage is free
    int32_t* mine = stage + wid * kMidPair;  // both lists of the warp's pair
    for (;;) {
        unsigned long long q = 0;
        if (lane == 0) q = atomicAdd((unsigned long long*)w.mnext + h, 1ull);
        q = __shfl_sync(0xffffffffu, q, 0);
        if ((int64_t)q >= nmid) break;
        PairCtx wpc;
        if (!load_pair(F, pl, st, h, w.mid[q], wpc)) continue;  // uniform in the warp
        __syncwarp();
        for (int i = lane; i < wpc.na; i += 32) mine[i] = wpc.ra[i];
        for (int i = lane; i < wpc.nb; i += 32) mine[wpc.na + i] = wpc.rb[i];
        __syncwarp();
        group_pair<32>(F, g, dmin2, pl, st, w, wpc, mine, mine + wpc.na, true, status);
    }
}

// Per-level form: each step of each level is its own launch.
constexpr int kRestThreads = 512;

__global__ void __launch_bounds__(128, 6) k_p1_small(lt_frame F, Grid g, float dmin2, P1Plan pl, P1Store st, P1Work w,
                                                  int h, int32_t* status) {
    p1_small_body(F, g, dmin2, pl, st, w, h, status);
}
__global__ void __launch_bounds__(kRestThreads, 2) k_p1_rest(lt_frame F, Grid g, float dmin2, P1Plan pl, P1Store st, P1Work w,
                                                 int h, int32_t* status) {
    p1_rest_body(F, g, dmin2, pl, st, w, h, status);
}

// Persistent form: one cooperative launch walks every level, the two steps of a level
// separated by grid-wide barriers.  `bar` counts block arrivals (zeroed before the
// launch); barrier k is passed when it reaches k * gridDim.x.  Every wait is bounded:
// past the limit the block latches LT_ELIMIT and leaves the walk (so do the others at
// their next barrier, also bounded).
constexpr unsigned kBarSpins = 1u << 21;

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned& k, int32_t* status, int* s_ok) {
    __syncthreads();
    ++k;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        const unsigned target = k * gridDim.x;
        int ok = 1;
        for (unsigned it = 0; ld_acquire_gpu(bar) < target; ++it) {
            if (it >= kBarSpins) {
                ok = 0;
                latch(status, LT_ELIMIT);
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

__global__ void __launch_bounds__(256, 3) k_p1_walk(lt_frame F, Grid g, float dmin2, P1Plan pl, P1Store st, P1Work w,
                                                 int32_t* status) {
    __shared__ int s_ok;
    unsigned k = 0;
    for (int h = 1; h <= F.H; ++h) {
        if (F.level_off[h + 1] == F.level_off[h]) continue;  // uniform over the grid
        p1_small_body(F, g, dmin2, pl, st, w, h, status);
        if (!grid_barrier(w.bar, k, status, &s_ok)) return;
        p1_rest_body(F, g, dmin2, pl, st, w, h, status);
        if (!grid_barrier(w.bar, k, status, &s_ok)) return;
    }
}

// -- the coarsened cut of every slice in leaf order, and where each column's entries go
constexpr int kOutThreads = 1024;

__global__ void __launch_bounds__(kOutThreads) k_p1_output(lt_frame F, P1Plan pl, lt_samples smp, int32_t* status) {
    extern __shared__ int32_t mark[];  // [C] forest node whose first leaf is c, else -1
    __shared__ long long ws[32];
    const int s = blockIdx.x;
    const int C = F.C, NF = 2 * C - 1;
    const int ms = F.slice_off[s + 1] - F.slice_off[s];
    const int32_t* cnt = pl.cnt + (int64_t)s * NF;
    const int32_t* state = pl.state + (int64_t)s * NF;
    if (ms == 0) {
        if (threadIdx.x == 0) {
            smp.ncol[s] = 0;
            smp.n1[s] = 0;
            smp.cnt[s] = 0;
        }
        return;
    }
    for (int c = threadIdx.x; c < C; c += blockDim.x) mark[c] = -1;
    __syncthreads();
    for (int x = threadIdx.x; x < NF; x += blockDim.x)
        if (state[x] == kStAlive) mark[F.forest[8 * x + 4]] = x;
    __syncthreads();
    int32_t* colx = pl.colx + (int64_t)s * C;
    int32_t* eoff = pl.eoff + (int64_t)s * C;
    // each thread has a run of cut nodes: one scan for the columns and their entry counts
    const int run = (C + blockDim.x - 1) / blockDim.x, c_lo = min(C, (int)threadIdx.x * run), c_hi = min(C, c_lo + run);
    auto entries = [&](int x) {
        const int par = F.forest[8 * x + 3];
        return par >= 0 && state[par] == kStRejected ? cnt[par] : cnt[x];
    };
    long long cols = 0;  // columns in the high half, entries in the low half
    for (int c = c_lo; c < c_hi; ++c)
        if (mark[c] >= 0) cols += (1ll << 40) + entries(mark[c]);
    long long tot;
    long long at = block_exclusive_scan<long long>(cols, ws, &tot);
    for (int c = c_lo; c < c_hi; ++c) {
        const int x = mark[c];
        if (x < 0) continue;
        const int j = (int)(at >> 40);
        colx[j] = x;
        eoff[j] = (int)(at & ((1ll << 40) - 1));
        smp.col_node[(int64_t)s * C + j] = F.forest[8 * x];
        at += (1ll << 40) + entries(x);
    }
    const int ncol = (int)(tot >> 40), n1 = (int)(tot & ((1ll << 40) - 1));
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool over = (int64_t)n1 > smp.off[s + 1] - smp.off[s];
        if (over) latch(status, LT_ELIMIT);
        smp.ncol[s] = ncol;
        smp.n1[s] = over ? 0 : n1;
        smp.cnt[s] = over ? 0 : n1;
        pl.total[s] = over ? -1 : 0;  // (the plan's totals are not needed any more) -1: no room for the entries
    }
}

// the entries and the importance g of every column, a warp per column (by the slice's one
// CTA after its scan, as this was, copying 5 M entries kept 64 of the SMs busy for 0.11 ms:
// a frame of 65536 points took 4.14 ms, 4.07 so, with the loads of the Omega build's
// sums in flight together)
__global__ void __launch_bounds__(256) k_p1_entries(lt_frame F, P1Plan pl, P1Store st, lt_samples smp) {
    const int s = blockIdx.x;  // (grid.y ends at 65535)
    const int C = F.C, NF = 2 * C - 1;
    const int lane = threadIdx.x & 31;
    const int32_t* cnt = pl.cnt + (int64_t)s * NF;
    const int32_t* off = pl.off + (int64_t)s * NF;
    const int32_t* state = pl.state + (int64_t)s * NF;
    const int64_t base = pl.base[s];
    const int32_t* rows = st.rows + base;
    const float* v0 = st.v0 + base;
    const float* v1 = st.v1 + base;
    const bool over = pl.total[s] < 0;
    const int ncol = smp.ncol[s];
    uint32_t* key = smp.key + smp.off[s];
    float* val = smp.val + smp.off[s];
    float* gs = smp.g + (int64_t)s * C;
    for (int j = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5); j < ncol; j += gridDim.y * (blockDim.x >> 5)) {
        const int x = pl.colx[(int64_t)s * C + j];
        const int par = F.forest[8 * x + 3];
        const bool from_par = par >= 0 && state[par] == kStRejected;
        const int src = from_par ? par : x;
        const int n = cnt[src];
        const int32_t* rr = rows + off[src];
        const float* vv = (from_par && F.forest[8 * par + 2] == x) ? v1 + off[src]
                          : (from_par && st.v2)                   ? st.v2 + base + off[src]
                                                                  : v0 + off[src];
        float mx = -3.0e38f, mn = 3.0e38f;
        const int dst = pl.eoff[(int64_t)s * C + j];
        for (int t = lane; t < n; t += 32) {
            const float v = vv[t];
            mx = fmaxf(mx, v);
            mn = fminf(mn, v);
            if (!over) {
                key[dst + t] = ((uint32_t)rr[t] << 16) | (uint32_t)j;
                val[dst + t] = v;
            }
        }
        mx = warp_max(mx);
        mn = warp_min(mn);
        if (lane == 0) gs[j] = n >= 2 ? mx - mn : -1.f;
    }
}

// a column of fewer than two entries takes the slice's largest g
__global__ void __launch_bounds__(256) k_p1_gfill(lt_frame F, lt_samples smp) {
    __shared__ float red[8];
    const int s = blockIdx.x, ncol = smp.ncol[s];
    float* gs = smp.g + (int64_t)s * F.C;
    float gm = -1.f;
    bool fill = false;
    for (int j = threadIdx.x; j < ncol; j += blockDim.x) {
        gm = fmaxf(gm, gs[j]);
        fill |= gs[j] < 0.f;
    }
    gm = warp_max(gm);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = gm;
    if (!__syncthreads_or(fill)) return;
    float m = -1.f;
    for (int w = 0; w < 8; ++w) m = fmaxf(m, red[w]);
    const float gfill = m >= 0.f ? m : 0.f;
    for (int j = threadIdx.x; j < ncol; j += blockDim.x)
        if (gs[j] < 0.f) gs[j] = gfill;
}

// ------------------------------------------------------------------ pass 2
__device__ __forceinline__ uint32_t hash32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352dU;
    x ^= x >> 15;
    x *= 0x846ca68bU;
    x ^= x >> 16;
    return x;
}

constexpr uint32_t kEmpty = 0xffffffffu;
constexpr int kP2Cluster = 8;    // CTAs per slice (one thread-block cluster)
constexpr int kP2Block = 512;    // threads per CTA
constexpr int kP2Draws = 4;      // draws per thread per round
constexpr int kGuide = 2048;     // buckets of the CDF guide table

// Per slice (one CTA each): the inclusive integer CDF of the quantised column
// weights (q = max(1, floor(w / w_max * 2^24)), 0 for w <= 0) and the bitmap of the
// pass-1 entries.
__global__ void __launch_bounds__(1024) k_p2_prep(lt_frame F, const float* __restrict__ weights, lt_samples smp,
                                                  unsigned long long* __restrict__ cdf_all,
                                                  unsigned long long* __restrict__ total_all, uint32_t* bitmap_all,
                                                  int64_t bitmap_stride) {
    __shared__ unsigned long long wsum[32];
    __shared__ float red[32];
    const int s = blockIdx.x;
    const int C = F.C;
    const int ms = F.slice_off[s + 1] - F.slice_off[s];
    const int ns = smp.ncol[s];
    const int n1 = smp.n1[s];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const float* w = (weights ? weights : smp.g) + (int64_t)s * C;
    float wm = 0.f;
    for (int j = threadIdx.x; j < ns; j += blockDim.x) wm = fmaxf(wm, w[j]);
    wm = warp_max(wm);
    if (lane == 0) red[wid] = wm;
    __syncthreads();
    float wmax = 0.f;
    for (int i = 0; i < nw; ++i) wmax = fmaxf(wmax, red[i]);
    unsigned long long* cdf = cdf_all + (int64_t)s * C;
    unsigned long long carry = 0;
    for (int c0 = 0; c0 < ns; c0 += blockDim.x) {
        const int j = c0 + threadIdx.x;
        unsigned long long q = 0;
        if (j < ns) {
            if (!(wmax > 0.f)) {
                q = 1;
            } else {
                const float wj = w[j];
                if (wj > 0.f) {
                    const float r = __fmul_rn(__fdiv_rn(wj, wmax), 16777216.0f);
                    q = (unsigned long long)floorf(r);
                    if (q < 1) q = 1;
                }
            }
        }
        unsigned long long tot;
        const unsigned long long pre = block_exclusive_scan<unsigned long long>(q, wsum, &tot);
        if (j < ns) cdf[j] = carry + pre + q;
        carry += tot;
    }
    if (threadIdx.x == 0) total_all[s] = carry;
    const int W = (ns + 31) >> 5;
    uint32_t* bm = bitmap_all + (int64_t)s * bitmap_stride;
    for (int64_t i = threadIdx.x; i < (int64_t)ms * W; i += blockDim.x) bm[i] = 0u;
    __syncthreads();
    const uint32_t* key1 = smp.key + smp.off[s];
    for (int i = threadIdx.x; i < n1; i += blockDim.x) {
        const uint32_t k = key1[i];
        const int r = (int)(k >> 16), c = (int)(k & 0xffffu);
        if (r < ms && c < ns) atomicOr(bm + (int64_t)r * W + (c >> 5), 1u << (c & 31));
    }
}

// One cluster of kP2Cluster CTAs per slice.  A round takes the next
// kP2Cluster x kP2Block x kP2Draws draws in order (CTA k the k-th block of them,
// thread i of a CTA kP2Draws consecutive ones), keeps those whose (row, col) is
// not observed yet (bitmap) and is the first of its key in the round, and accepts them in
// draw order (a prefix over the CTAs' counts) up to the target.  Every CTA of the
// cluster computes the same accepted count, so all take the same cluster barriers.
// The first draw of a key: the new draws set their bit (atomicOr); a draw that finds it
// set since the round began shares its key with another (about one in a hundred does),
// enters the key with its index in a hash table spread over the cluster's shared memory
// (home CTA hash & 7) and marks the key in a filter that every CTA has; the draws that set
// their bit look the key up only where the filter says so, and the smallest index of the
// key is kept.  What bounds a round is the latency of its L2 atomics and five cluster
// barriers.  5.4 M entries in 64 slices: 0.37 ms (cold caches), 0.80 ms when every draw
// went through the table with two remote atomics and found its CDF bucket by a 64-bit
// division.
constexpr int kP2Filter = 512;   // words of the filter

__global__ void __cluster_dims__(kP2Cluster, 1, 1) __launch_bounds__(kP2Block, 2)
    k_pass2(lt_frame F, float rate, SeedRef sr, lt_samples smp, const unsigned long long* __restrict__ cdf_all,
            const unsigned long long* __restrict__ total_all, uint32_t* bitmap_all, int64_t bitmap_stride, int hpart,
            int32_t* status) {
    namespace cg = cooperative_groups;
    // dynamic shared memory: cdf[C] (u64), hkey[hpart] (u32), htid[hpart] (int32: the
    // smallest draw index of the key in the round), guide[kGuide + 1] (int32), filter
    extern __shared__ unsigned long long p2sm[];
    unsigned long long* scdf = p2sm;
    uint32_t* hkey = reinterpret_cast<uint32_t*>(p2sm + F.C);
    int32_t* htid = reinterpret_cast<int32_t*>(hkey + hpart);
    int32_t* guide = htid + hpart;
    uint32_t* filter = reinterpret_cast<uint32_t*>(guide + kGuide + 1);
    __shared__ int32_t ws[32];
    __shared__ int32_t s_cnt;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int s = blockIdx.x / kP2Cluster;
    const int C = F.C;
    const int ms = F.slice_off[s + 1] - F.slice_off[s];
    const int ns = smp.ncol[s];
    const int n1 = smp.n1[s];
    const uint64_t seed = sr.get();
    if (ms == 0 || ns == 0) {
        if (rank == 0 && threadIdx.x == 0) smp.cnt[s] = n1;
        return;
    }
    const int64_t T = (int64_t)ceil((double)rate * (double)ms * (double)ns);
    int64_t need = T - n1;
    if (need <= 0) {
        if (rank == 0 && threadIdx.x == 0) smp.cnt[s] = n1;
        return;
    }
    const int64_t capacity = smp.off[s + 1] - smp.off[s];
    if (n1 + need > capacity) {
        if (rank == 0 && threadIdx.x == 0) latch(status, LT_ELIMIT);
        need = capacity - n1;
    }
    const unsigned long long total = total_all[s];
    const uint32_t th = (uint32_t)(total >> 32), tl = (uint32_t)total;
    const int W = (ns + 31) >> 5;
    uint32_t* bm = bitmap_all + (int64_t)s * bitmap_stride;
    for (int j = threadIdx.x; j < ns; j += blockDim.x) scdf[j] = cdf_all[(int64_t)s * C + j];
    for (int i = threadIdx.x; i < hpart; i += blockDim.x) {
        hkey[i] = kEmpty;
        htid[i] = 0x7fffffff;
    }
    for (int i = threadIdx.x; i < kP2Filter; i += blockDim.x) filter[i] = 0u;
    __syncthreads();
    // guide table: guide[k] = first c with cdf[c] > floor(k total / kGuide); a draw u in
    // bucket k = floor(u kGuide / total) has its column in [guide[k], guide[k + 1]]
    for (int k = threadIdx.x; k <= kGuide; k += blockDim.x) {
        const unsigned long long v = (unsigned long long)k * total / kGuide;
        int a = 0, b = ns - 1;  // cdf[ns - 1] = total > v for k < kGuide
        while (a < b) {
            const int m = (a + b) >> 1;
            if (scdf[m] > v) b = m;
            else a = m + 1;
        }
        guide[k] = a;
    }
    cl.sync();
    const int64_t cap_draws = 64 * T + 64;
    uint32_t* keyout = smp.key + smp.off[s] + n1;
    const int64_t per_cta = (int64_t)blockDim.x * kP2Draws, per_round = per_cta * kP2Cluster;
    int64_t accepted = 0;
    for (int64_t t0 = 0; accepted < need && t0 < cap_draws; t0 += per_round) {
        uint32_t rc[kP2Draws];
        int home[kP2Draws], slot[kP2Draws], tr[kP2Draws];
        int64_t tt[kP2Draws];
        unsigned long long u[kP2Draws];
        uint32_t wrow[kP2Draws], wcol[kP2Draws];
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d) {  // draw and column search, all draws at once
            tt[d] = t0 + rank * per_cta + (int64_t)threadIdx.x * kP2Draws + d;
            const U4 x = philox((uint32_t)tt[d], 0u, slice_key(F.slice_id, s), kTagPass2, seed);
            u[d] = (unsigned long long)x.x * th + (((unsigned long long)x.x * tl) >> 32);
            wrow[d] = x.y;
            wcol[d] = x.x;
            home[d] = -1;
        }
        int lo[kP2Draws];
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d) {  // first c with cdf[c] > u, from its guide bucket
            // u = floor(x total / 2^32), so its bucket floor(u kGuide / total) is
            // floor(x kGuide / 2^32) or the one before
            static_assert(kGuide == 2048, "bucket shift");
            const int k = (int)(wcol[d] >> 21);
            int a = guide[max(k - 1, 0)], b = guide[k + 1];
            while (a < b) {
                const int m = (a + b) >> 1;
                if (scdf[m] > u[d]) b = m;
                else a = m + 1;
            }
            lo[d] = a;
        }
        uint32_t word[kP2Draws];
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d) {
            const int c = lo[d], r = (int)uniform_index(wrow[d], (uint32_t)ms);
            rc[d] = ((uint32_t)r << 16) | (uint32_t)c;
            // L2 reads: other CTAs of the cluster set bits in earlier rounds (L1 is not coherent)
            word[d] = tt[d] < cap_draws ? __ldcg(bm + (int64_t)r * W + (c >> 5)) : 0xffffffffu;
        }
        cl.sync();  // every CTA has read its words: from here on a bit is set by this round or was seen
        uint32_t newmask = 0, lost = 0;
        uint32_t old[kP2Draws];
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d) {
            const int r = (int)(rc[d] >> 16), c = (int)(rc[d] & 0xffffu);
            tr[d] = (int)(tt[d] - t0);
            old[d] = 0u;
            if ((word[d] >> (c & 31)) & 1u) continue;  // observed (or past the draw cap)
            newmask |= 1u << d;
            old[d] = atomicOr(bm + (int64_t)r * W + (c >> 5), 1u << (c & 31));
        }
        uint32_t hash[kP2Draws], key[kP2Draws];
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d) {
            const int r = (int)(rc[d] >> 16), c = (int)(rc[d] & 0xffffu);
            key[d] = (uint32_t)r * (uint32_t)ns + (uint32_t)c;
            hash[d] = hash32(key[d]);
            if (!((newmask >> d) & 1u) || !((old[d] >> (c & 31)) & 1u)) continue;
            lost |= 1u << d;  // another draw of the round has this key
            const int k = (int)(hash[d] & (kP2Cluster - 1));
            uint32_t* rk = cl.map_shared_rank(hkey, k);
            int32_t* rt = cl.map_shared_rank(htid, k);
            uint32_t p = (hash[d] >> 3) & (uint32_t)(hpart - 1);
            bool entered = false;
            for (int probe = 0; probe < hpart; ++probe) {
                const uint32_t prev = atomicCAS(&rk[p], kEmpty, key[d]);
                if (prev == kEmpty || prev == key[d]) {
                    atomicMin(&rt[p], tr[d]);
                    home[d] = k;
                    slot[d] = (int)p;
                    entered = prev == kEmpty;
                    break;
                }
                p = (p + 1) & (uint32_t)(hpart - 1);
            }
            // a full table part: not expected, a round has at most half as many shared keys as draws
            if (home[d] < 0) latch(status, LT_ELIMIT);
            if (!entered) continue;  // the key is in the filters, or its first draw is putting it there
            const uint32_t fb = (hash[d] >> 3) & (uint32_t)(32 * kP2Filter - 1);
            for (int q = 0; q < kP2Cluster; ++q) atomicOr(cl.map_shared_rank(filter, q) + (fb >> 5), 1u << (fb & 31));
        }
        cl.sync();
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d) {  // the draws that set their bit, where the key may have others
            if (!(((newmask & ~lost) >> d) & 1u)) continue;
            const uint32_t fb = (hash[d] >> 3) & (uint32_t)(32 * kP2Filter - 1);
            if (!((filter[fb >> 5] >> (fb & 31)) & 1u)) continue;
            const int k = (int)(hash[d] & (kP2Cluster - 1));
            const uint32_t* rk = cl.map_shared_rank(hkey, k);
            uint32_t p = (hash[d] >> 3) & (uint32_t)(hpart - 1);
            for (int probe = 0; probe < hpart; ++probe) {
                const uint32_t at = rk[p];
                if (at == kEmpty) break;
                if (at == key[d]) {
                    atomicMin(cl.map_shared_rank(htid, k) + p, tr[d]);
                    home[d] = k;
                    slot[d] = (int)p;
                    break;
                }
                p = (p + 1) & (uint32_t)(hpart - 1);
            }
        }
        cl.sync();
        int mine = 0;
        uint32_t firstmask = 0;
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d) {
            if (!((newmask >> d) & 1u)) continue;
            const bool first = home[d] >= 0 ? cl.map_shared_rank(htid, home[d])[slot[d]] == tr[d] : !((lost >> d) & 1u);
            if (first) {
                firstmask |= 1u << d;
                ++mine;
            }
        }
        int tot;
        int pos = block_exclusive_scan<int>(mine, ws, &tot);
        if (threadIdx.x == 0) s_cnt = tot;
        cl.sync();
        int before = 0, round_total = 0;
        for (int k = 0; k < kP2Cluster; ++k) {
            const int ck = *cl.map_shared_rank(&s_cnt, k);
            if (k < rank) before += ck;
            round_total += ck;
        }
#pragma unroll
        for (int d = 0; d < kP2Draws; ++d)
            if (firstmask & (1u << d)) {
                const int64_t g = accepted + before + pos;
                if (g < need) keyout[g] = rc[d];
                ++pos;
            }
        accepted += min((int64_t)round_total, need - accepted);
        // every CTA is past its look-ups (the barrier before the counts): the table is free
        for (int i = threadIdx.x; i < hpart; i += blockDim.x) {
            hkey[i] = kEmpty;
            htid[i] = 0x7fffffff;
        }
        for (int i = threadIdx.x; i < kP2Filter; i += blockDim.x) filter[i] = 0u;
        __threadfence();
        cl.sync();
    }
    if (rank == 0 && threadIdx.x == 0) smp.cnt[s] = n1 + (int)accepted;
}

// ------------------------------------------------------------------ entry evaluation
__global__ void k_count_prefix(const lt_samples smp, int S, int64_t* pfx) {
    __shared__ int64_t ws[32];
    int64_t carry = 0;
    for (int c0 = 0; c0 < S; c0 += blockDim.x) {
        const int s = c0 + threadIdx.x;
        const int64_t x = s < S ? (int64_t)(smp.cnt[s] - smp.n1[s]) : 0;
        int64_t tot;
        const int64_t pre = block_exclusive_scan<int64_t>(x, ws, &tot);
        if (s < S) pfx[s] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) pfx[S] = carry;
}

// Column records of a frame: for every (slice, coarsened column) the representative
// VPL's three record planes and the node's scale I_c / (flux albedo) of its
// representative, 64 B each ([S][C][4] float4), so that an entry gathers its column
// with one contiguous load (a slice's few hundred columns stay in L1) instead of the
// node, its representative, the three VPL planes and three scale terms.
__global__ void k_col_records(lt_frame F, lt_samples smp, float4* __restrict__ tab) {
    const int s = blockIdx.y;
    const int ns = smp.ncol[s];
    const float4* vpls = reinterpret_cast<const float4*>(F.vpls);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ns; c += gridDim.x * blockDim.x) {
        const int node = smp.col_node[(int64_t)s * F.C + c];
        const PointRec L = load_rec(vpls, F.n, F.tree.rep[node]);
        float4* t = tab + ((int64_t)s * F.C + c) * 4;
        t[0] = L.a;
        t[1] = L.b;
        t[2] = L.c;
        t[3] = make_float4(node_scale(F.tree, vpls, F.n, node), 0.f, 0.f, 0.f);
    }
}

template <bool COUNT>
__global__ void __launch_bounds__(128) k_eval_entries(lt_frame F, Grid g, float dmin2, lt_samples smp,
                                                      const int64_t* __restrict__ pfx,
                                                      const float4* __restrict__ coltab,
                                                      unsigned long long* __restrict__ stats, int32_t* status) {
    extern __shared__ int64_t spfx[];
    const int S = F.S;
    for (int i = threadIdx.x; i <= S; i += blockDim.x) spfx[i] = pfx[i];
    __syncthreads();
    const int64_t total = spfx[S];
    const float4* pts = reinterpret_cast<const float4*>(F.pts);
    const float4* vpls = reinterpret_cast<const float4*>(F.vpls);
    WorkCount wc;
    int rays = 0, entries = 0;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = S;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (spfx[mid] <= idx) lo = mid;
            else hi = mid;
        }
        const int s = lo;
        const int64_t e = smp.off[s] + smp.n1[s] + (idx - spfx[s]);
        const uint32_t k = smp.key[e];
        const int r = (int)(k >> 16), c = (int)(k & 0xffffu);
        const PointRec P = load_rec(pts, F.m, F.slice_off[s] + r);
        PointRec L;
        float scale;
        if (coltab) {  // the frame's column records
            const float4* t = coltab + ((int64_t)s * F.C + c) * 4;
            L.a = __ldg(t);
            L.b = __ldg(t + 1);
            L.c = __ldg(t + 2);
            scale = __ldg(t + 3).x;
        } else {
            const int node = smp.col_node[(int64_t)s * F.C + c];
            L = load_rec(vpls, F.n, F.tree.rep[node]);
            scale = node_scale(F.tree, vpls, F.n, node);
        }
        const float v = entry_value<COUNT>(P, L, scale, dmin2, g, &wc, &rays);
        if (COUNT) {
            ++entries;
        } else {
            if (!isfinite(v)) latch(status, LT_ENUMERIC);
            smp.val[e] = v;
        }
    }
    if (COUNT) {
        atomicAdd(stats + 0, (unsigned long long)entries);
        atomicAdd(stats + 1, (unsigned long long)rays);
        atomicAdd(stats + 2, (unsigned long long)wc.cells);
        atomicAdd(stats + 3, (unsigned long long)wc.boxes);
    }
}

bool frame_ok(const lt_frame* f) {
    return f && f->pts && f->vpls && f->slice_off && f->S > 0 && f->m > 0 && f->n > 0 && f->C >= 1 &&
           f->C <= kMaxCut && f->forest && f->max_rows >= 0 && f->max_rows <= 65535 && f->tree.I &&
           f->tree.rep && (((uintptr_t)f->pts & 15) == 0) && (((uintptr_t)f->vpls & 15) == 0) &&
           (f->C == 1 || (f->level_off && f->level_nodes)) && f->H >= 0;
}

bool samples_ok(const lt_samples* s) {
    return s && s->ncol && s->col_node && s->g && s->off && s->key && s->val && s->n1 && s->cnt;
}

}  // namespace

namespace {

lt_status sample_pass1(lt_ctx* ctx, const lt_frame* f, float rate1, float tau, int32_t target, float d_min,
                       uint64_t seed, lt_samples* smp) {
    if (!ctx->d_cell_off) return lt_fail(ctx, LT_EINVAL, "lt_sample_pass1: no scene uploaded");
    cudaSetDevice(ctx->device);
    const int S = f->S, C = f->C, NF = 2 * C - 1;
    lt_status st;
    const size_t n_k = (size_t)S * C, n_f = (size_t)S * NF, n_p = (size_t)S * (C + 1);
    const size_t bytes = (n_k * 3 + n_f * 5 + n_p) * sizeof(int32_t) + 2 * S * sizeof(int64_t) + 16 * 256;
    char* p = (char*)lt_scratch(ctx, SCR_P1_PLAN, bytes, &st);
    if (!p) return st;
    P1Plan pl;
    auto take = [&](size_t nbytes) {
        char* q = p;
        p += (nbytes + 255) & ~(size_t)255;
        return q;
    };
    pl.total = (int64_t*)take(S * sizeof(int64_t));
    pl.base = (int64_t*)take(S * sizeof(int64_t));
    pl.k = (int32_t*)take(n_k * 4);
    pl.colx = (int32_t*)take(n_k * 4);
    pl.eoff = (int32_t*)take(n_k * 4);
    pl.cap = (int32_t*)take(n_f * 4);
    pl.off = (int32_t*)take(n_f * 4);
    pl.cnt = (int32_t*)take(n_f * 4);
    pl.state = (int32_t*)take(n_f * 4);
    pl.cost = (float*)take(n_f * 4);
    pl.pfx = (int32_t*)take(n_p * 4);
    if ((size_t)(p - (char*)ctx->scr[SCR_P1_PLAN]) > ctx->scr_size[SCR_P1_PLAN])
        return lt_fail(ctx, LT_ENOMEM, "lt_sample_pass1: plan layout overflow");
    k_pass1_plan<<<S, kP1Threads, 0, ctx->stream>>>(*f, rate1, pl);
    LT_LAUNCH_CHECK(ctx, "k_pass1_plan");
    k_p1_base<<<1, 1024, 0, ctx->stream>>>(S, pl);
    LT_LAUNCH_CHECK(ctx, "k_p1_base");
    // The row-slot total sizes the scratch below; it follows from the setup alone
    // (cut, forest, slices, rate1), so a captured frame reuses the recorded value.
    int64_t acc = 0;
    if (ctx->use_plan) {
        acc = ctx->plan.p1_total;
    } else {
        std::vector<int64_t> tot(S);
        LT_CUDA(ctx, cudaMemcpyAsync(tot.data(), pl.total, S * sizeof(int64_t), cudaMemcpyDeviceToHost, ctx->stream));
        LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        for (int s = 0; s < S; ++s) acc += tot[s];
        ctx->plan.p1_total = acc;
    }
    // storage: rows, then v0 and v1 back to back (a flat value index addresses both);
    // then the work arrays of the flat kernels
    const int Hn = f->H + 2;
    const int64_t bcap = std::max<int64_t>((int64_t)S * C, 1024);
    const size_t store_bytes = (size_t)std::max<int64_t>(acc, 1) * (target > 0 ? 16 : 12) + 1024;
    const size_t eff_bytes = target > 0 ? (size_t)S * NF * 4 : 0;
    const size_t work_bytes = (size_t)(S + 1) * 8 + (size_t)S * C * 4 + (size_t)S * 4 + (size_t)Hn * 24 +
                              (size_t)bcap * 16 + (size_t)NF * 64 + eff_bytes + 18 * 256;
    char* q = (char*)lt_scratch(ctx, SCR_P1_STORE, store_bytes + work_bytes, &st);
    if (!q) return st;
    P1Store store;
    store.total = acc;
    store.rows = (int32_t*)q;
    store.v0 = (float*)(q + ((acc * 4 + 255) & ~255LL));
    store.v1 = store.v0 + acc;
    store.v2 = target > 0 ? store.v1 + acc : nullptr;
    char* wp = q + ((store_bytes + 255) & ~(size_t)255);
    auto wtake = [&](size_t nbytes) {
        char* r = wp;
        wp += (nbytes + 255) & ~(size_t)255;
        return r;
    };
    P1Work w;
    w.kpfx = (int64_t*)wtake((size_t)(S + 1) * 8);
    w.leafmean = (float*)wtake((size_t)S * C * 4);
    w.thr = (float*)wtake((size_t)S * 4);
    w.mcount = (int64_t*)wtake((size_t)Hn * 24 + 8);  // the counters, zeroed together
    w.bcount = w.mcount + Hn;
    w.mnext = w.bcount + Hn;
    w.nrec = (float4*)wtake((size_t)NF * 64);
    w.mid = (int64_t*)wtake((size_t)bcap * 8);
    w.big = (int64_t*)wtake((size_t)bcap * 8);
    w.bar = (unsigned*)(w.mnext + Hn);
    w.bcap = bcap;
    float* effs = target > 0 ? (float*)wtake(eff_bytes) : nullptr;
    if ((size_t)(wp - q) > ctx->scr_size[SCR_P1_STORE])
        return lt_fail(ctx, LT_ENOMEM, "lt_sample_pass1: work layout overflow");
    LT_CUDA(ctx, cudaMemsetAsync(w.mcount, 0, (size_t)Hn * 24 + 8, ctx->stream));
    const int nsm = ctx->num_sms;
    const float dmin2 = d_min * d_min;
    auto grid_for = [&](int64_t items, int threads) {
        return (unsigned)std::max<int64_t>(1, std::min<int64_t>((items + threads - 1) / threads, 32 * (int64_t)nsm));
    };
    k_p1_draws<<<grid_for((int64_t)S * NF, 256), 256, 0, ctx->stream>>>(*f, seed_ref(ctx, seed), pl, store,
                                                                        ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_p1_draws");
    k_p1_nodes<<<(NF + 255) / 256, 256, 0, ctx->stream>>>(*f, w.nrec);
    LT_LAUNCH_CHECK(ctx, "k_p1_nodes");
    k_p1_kpfx<<<1, 1024, 0, ctx->stream>>>(*f, pl, w.kpfx);
    LT_LAUNCH_CHECK(ctx, "k_p1_kpfx");
    const int ray_grid = ctx->tune.ray_ctas_per_sm * nsm;
    k_p1_initial<<<ray_grid, 128, 0, ctx->stream>>>(*f, ctx->grid, dmin2, pl, store, w.kpfx, w.nrec, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_p1_initial");
    k_p1_leafmean<<<grid_for((int64_t)S * C, 256), 256, 0, ctx->stream>>>(*f, pl, store, w.leafmean);
    LT_LAUNCH_CHECK(ctx, "k_p1_leafmean");
    if (target > 0) {
        k_p1_thr_inf<<<(S + 255) / 256, 256, 0, ctx->stream>>>(S, w.thr);
        LT_LAUNCH_CHECK(ctx, "k_p1_thr_inf");
    } else {
        k_p1_thr<<<S, 256, 0, ctx->stream>>>(*f, w.leafmean, tau, w.thr);
        LT_LAUNCH_CHECK(ctx, "k_p1_thr");
    }
    std::vector<int32_t> loff(f->H + 2, 0);
    if (ctx->use_plan) {
        if ((int)ctx->plan.level_off.size() != f->H + 2)
            return lt_fail(ctx, LT_EINVAL, "lt_sample_pass1: recorded frame plan does not match the forest");
        loff = ctx->plan.level_off;
    } else {
        if (f->H > 0)
            LT_CUDA(ctx, cudaMemcpyAsync(loff.data(), f->level_off, (f->H + 2) * 4, cudaMemcpyDeviceToHost,
                                         ctx->stream));
        LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        ctx->plan.level_off = loff;
    }
    const bool walk = ctx->tune.p1_form == 1 && f->H > 0;
    if (walk) {
        if (ctx->p1_walk_blocks == 0) {
            int nb = 0;
            LT_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_p1_walk, 256, 0));
            ctx->p1_walk_blocks = std::max(1, std::min(nb, 8));
        }
        // every block resident at once (the cooperative launch checks it)
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3((unsigned)(ctx->p1_walk_blocks * nsm));
        lc.blockDim = dim3(256);
        lc.dynamicSmemBytes = 0;
        lc.stream = ctx->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        lc.attrs = at;
        lc.numAttrs = 1;
        LT_CUDA(ctx, cudaLaunchKernelEx(&lc, k_p1_walk, *f, ctx->grid, dmin2, pl, store, w, ctx->d_status));
        LT_LAUNCH_CHECK(ctx, "k_p1_walk");
    }
    for (int h = 1; h <= f->H && !walk; ++h) {
        const int64_t npairs = (int64_t)S * (loff[h + 1] - loff[h]);
        if (npairs == 0) continue;
        k_p1_small<<<grid_for(npairs * kGroup, 128), 128, 0, ctx->stream>>>(*f, ctx->grid, dmin2, pl, store, w, h,
                                                                           ctx->d_status);
        LT_LAUNCH_CHECK(ctx, "k_p1_small");
        k_p1_rest<<<2 * nsm, kRestThreads, 0, ctx->stream>>>(*f, ctx->grid, dmin2, pl, store, w, h, ctx->d_status);
        LT_LAUNCH_CHECK(ctx, "k_p1_rest");
    }
    if (target > 0) {
        k_p1_target<<<S, 1024, 0, ctx->stream>>>(*f, pl, effs, target);
        LT_LAUNCH_CHECK(ctx, "k_p1_target");
    }
    const size_t shm = (size_t)C * 4;
    if (shm > 16 * 1024)
        LT_CUDA(ctx, cudaFuncSetAttribute(k_p1_output, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    k_p1_output<<<S, kOutThreads, shm, ctx->stream>>>(*f, pl, *smp, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_p1_output");
    k_p1_entries<<<dim3(S, (unsigned)std::max(1, std::min((C + 7) / 8, 8 * nsm / S))), 256, 0, ctx->stream>>>(
        *f, pl, store, *smp);
    LT_LAUNCH_CHECK(ctx, "k_p1_entries");
    k_p1_gfill<<<S, 256, 0, ctx->stream>>>(*f, *smp);
    LT_LAUNCH_CHECK(ctx, "k_p1_gfill");
    return LT_OK;
}

}  // namespace

extern "C" lt_status lt_sample_pass1(lt_ctx* ctx, const lt_frame* f, float rate1, float tau, float d_min,
                                     uint64_t seed, lt_samples* smp) {
    if (!ctx || !frame_ok(f) || !samples_ok(smp) || !(rate1 >= 0.f) || !(tau >= 0.f))
        return lt_fail(ctx, LT_EINVAL, "lt_sample_pass1: bad arguments");
    return sample_pass1(ctx, f, rate1, tau, 0, d_min, seed, smp);
}

extern "C" lt_status lt_sample_pass1_target(lt_ctx* ctx, const lt_frame* f, float rate1, int32_t target,
                                            float d_min, uint64_t seed, lt_samples* smp) {
    if (!ctx || !frame_ok(f) || !samples_ok(smp) || !(rate1 >= 0.f) || target < 1)
        return lt_fail(ctx, LT_EINVAL, "lt_sample_pass1_target: bad arguments");
    return sample_pass1(ctx, f, rate1, 0.f, target, d_min, seed, smp);
}

extern "C" lt_status lt_sample_pass2(lt_ctx* ctx, const lt_frame* f, const float* weights, float rate,
                                     uint64_t seed, lt_samples* smp) {
    if (!ctx || !frame_ok(f) || !samples_ok(smp) || !(rate >= 0.f))
        return lt_fail(ctx, LT_EINVAL, "lt_sample_pass2: bad arguments");
    cudaSetDevice(ctx->device);
    const int S = f->S, C = f->C;
    const int64_t stride = (int64_t)std::max(f->max_rows, 1) * ((C + 31) / 32);
    lt_status st;
    uint32_t* bm = (uint32_t*)lt_scratch(ctx, SCR_BITMAP, (size_t)S * stride * 4, &st);
    if (!bm) return st;
    unsigned long long* cdf_all = (unsigned long long*)lt_scratch(ctx, SCR_P2_CDF, ((size_t)S * C + S + 64) * 8, &st);
    if (!cdf_all) return st;
    unsigned long long* total_all = cdf_all + (size_t)S * C;
    k_p2_prep<<<S, 1024, 0, ctx->stream>>>(*f, weights, *smp, cdf_all, total_all, bm, stride);
    LT_LAUNCH_CHECK(ctx, "k_p2_prep");
    // each CTA's part of the round's hash table: a slot per draw of the CTA (only keys drawn
    // more than once enter it)
    const int hpart = kP2Block * kP2Draws;
    const size_t shm = (size_t)C * 8 + (size_t)hpart * 8 + (size_t)(kGuide + 2 + kP2Filter) * 4;
    if (shm > (size_t)220 * 1024)
        return lt_fail(ctx, LT_EINVAL, "lt_sample_pass2: global cut too large for the pass-2 CDF in shared memory");
    LT_CUDA(ctx, cudaFuncSetAttribute(k_pass2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    k_pass2<<<S * kP2Cluster, kP2Block, shm, ctx->stream>>>(*f, rate, seed_ref(ctx, seed), *smp, cdf_all, total_all, bm,
                                                            stride, hpart, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_pass2");
    return LT_OK;
}

extern "C" lt_status lt_eval_entries(lt_ctx* ctx, const lt_frame* f, float d_min, lt_samples* smp) {
    if (!ctx || !frame_ok(f) || !samples_ok(smp)) return lt_fail(ctx, LT_EINVAL, "lt_eval_entries: bad arguments");
    if (!ctx->d_cell_off) return lt_fail(ctx, LT_EINVAL, "lt_eval_entries: no scene uploaded");
    cudaSetDevice(ctx->device);
    lt_status st;
    const size_t apfx = ((size_t)(f->S + 1) * 8 + 255) & ~(size_t)255;
    char* p = (char*)lt_scratch(ctx, SCR_MISC, apfx + (size_t)f->S * f->C * 64, &st);
    if (!p) return st;
    int64_t* pfx = (int64_t*)p;
    float4* tab = (float4*)(p + apfx);
    k_count_prefix<<<1, 1024, 0, ctx->stream>>>(*smp, f->S, pfx);
    LT_LAUNCH_CHECK(ctx, "k_count_prefix");
    k_col_records<<<dim3((unsigned)std::min(16, (f->C + 255) / 256), f->S), 256, 0, ctx->stream>>>(*f, *smp, tab);
    LT_LAUNCH_CHECK(ctx, "k_col_records");
    const size_t shm = (size_t)(f->S + 1) * 8;
    if (shm > 16 * 1024)
        LT_CUDA(ctx, cudaFuncSetAttribute(k_eval_entries<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)shm));
    k_eval_entries<false><<<ctx->num_sms * ctx->tune.eval_ctas_per_sm, 128, shm, ctx->stream>>>(*f, ctx->grid, d_min * d_min, *smp, pfx,
                                                                        tab, nullptr, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_eval_entries");
    return LT_OK;
}

// ------------------------------------------------------------------ allocation-free variant
// lt_eval_entries keeps its per-slice prefix in context scratch, which it grows
// with cudaMalloc.  Some hosts cannot allow that: an application that owns the
// whole device-memory budget and hands the library only its inputs and outputs
// (for example a renderer plugin running inside a frame loop), where a cudaMalloc
// could fail against the fixed budget or stall the device in the middle of a frame.
// For them the prefix lives in this fixed device array instead.  It is part of the
// module image, so every GPU that loads the library holds its 32 KB until exit.
constexpr int kNoAllocMaxSlices = 4096;
static __device__ __align__(256) int64_t g_noalloc_prefix[kNoAllocMaxSlices + 1];

namespace {
constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
int64_t* g_noalloc_addr[kNoAllocMaxDevices] = {};

// Device address of g_noalloc_prefix on the context's device.  In host code the
// symbol names a host-side stand-in, so the real address is looked up with that
// device current.  It is looked up again on every call (cheap, and it allocates
// nothing), so a module reloaded after a device reset is found where it now is; the
// last address seen per device is kept only for calls made while the context's
// stream is being captured, where the lookup is not attempted.
lt_status noalloc_prefix(lt_ctx* ctx, int64_t** out) {
    if (ctx->device < 0 || ctx->device >= kNoAllocMaxDevices)
        return lt_fail(ctx, LT_EINVAL, "lt_eval_entries_noalloc: device index out of range");
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    LT_CUDA(ctx, cudaStreamIsCapturing(ctx->stream, &cap));
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (cap != cudaStreamCaptureStatusNone) {
        if (!g_noalloc_addr[ctx->device])
            return lt_fail(ctx, LT_EINVAL,
                           "lt_eval_entries_noalloc: make one call on this device before capturing a stream");
        *out = g_noalloc_addr[ctx->device];
        return LT_OK;
    }
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_prefix);
    if (e != cudaSuccess) return lt_cuda_check(ctx, e, "cudaGetSymbolAddress(g_noalloc_prefix)");
    g_noalloc_addr[ctx->device] = (int64_t*)p;
    *out = (int64_t*)p;
    return LT_OK;
}
}  // namespace

extern "C" lt_status lt_eval_entries_noalloc(lt_ctx* ctx, const lt_frame* f, float d_min, lt_samples* smp) {
    if (!ctx || !frame_ok(f) || !samples_ok(smp))
        return lt_fail(ctx, LT_EINVAL, "lt_eval_entries_noalloc: bad arguments");
    if (f->S > kNoAllocMaxSlices)
        return lt_fail(ctx, LT_EINVAL,
                       "lt_eval_entries_noalloc: at most " + std::to_string(kNoAllocMaxSlices) + " slices");
    if (!ctx->d_cell_off) return lt_fail(ctx, LT_EINVAL, "lt_eval_entries_noalloc: no scene uploaded");
    LT_CUDA(ctx, cudaSetDevice(ctx->device));
    int64_t* pfx = nullptr;
    const lt_status st = noalloc_prefix(ctx, &pfx);
    if (st != LT_OK) return st;
    // every entry of the prefix that the evaluation reads is rewritten here first
    k_count_prefix<<<1, 1024, 0, ctx->stream>>>(*smp, f->S, pfx);
    LT_LAUNCH_CHECK(ctx, "k_count_prefix");
    const size_t shm = (size_t)(f->S + 1) * 8;
    if (shm > 16 * 1024)
        LT_CUDA(ctx, cudaFuncSetAttribute(k_eval_entries<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)shm));
    k_eval_entries<false><<<ctx->num_sms * ctx->tune.eval_ctas_per_sm, 128, shm, ctx->stream>>>(*f, ctx->grid, d_min * d_min, *smp, pfx,
                                                                        nullptr, nullptr, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_eval_entries");
    return LT_OK;
}

extern "C" lt_status lt_eval_stats(lt_ctx* ctx, const lt_frame* f, float d_min, const lt_samples* smp,
                                   int64_t* stats_host) {
    if (!ctx || !frame_ok(f) || !samples_ok(smp) || !stats_host)
        return lt_fail(ctx, LT_EINVAL, "lt_eval_stats: bad arguments");
    if (!ctx->d_cell_off) return lt_fail(ctx, LT_EINVAL, "lt_eval_stats: no scene uploaded");
    cudaSetDevice(ctx->device);
    lt_status st;
    char* p = (char*)lt_scratch(ctx, SCR_MISC, (size_t)(f->S + 1) * 8 + 512, &st);
    if (!p) return st;
    int64_t* pfx = (int64_t*)p;
    unsigned long long* stats = (unsigned long long*)(p + (((f->S + 1) * 8 + 255) & ~255));
    LT_CUDA(ctx, cudaMemsetAsync(stats, 0, 4 * 8, ctx->stream));
    k_count_prefix<<<1, 1024, 0, ctx->stream>>>(*smp, f->S, pfx);
    LT_LAUNCH_CHECK(ctx, "k_count_prefix");
    const size_t shm = (size_t)(f->S + 1) * 8;
    if (shm > 16 * 1024)
        LT_CUDA(ctx, cudaFuncSetAttribute(k_eval_entries<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)shm));
    lt_samples copy = *smp;
    k_eval_entries<true><<<ctx->num_sms * ctx->tune.eval_ctas_per_sm, 128, shm, ctx->stream>>>(*f, ctx->grid, d_min * d_min, copy, pfx,
                                                                       nullptr, stats, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_eval_entries<count>");
    unsigned long long h[4];
    LT_CUDA(ctx, cudaMemcpyAsync(h, stats, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
    LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    for (int i = 0; i < 4; ++i) stats_host[i] = (int64_t)h[i];
    return LT_OK;
}
