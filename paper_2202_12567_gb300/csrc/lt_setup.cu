// Setup of a frame: light tree and conservative global cut (Sec. 3 step 1, the
// splitting test parallel over the nodes of a level, Sec. 6), the cut's ancestor
// forest used by the coarsening, and the slicing of the matrix rows by k-means on
// position and normal (Sec. 3 step 2).
//
// Tree: Morton codes (float32 decisions, orientation class above the code), a
// bitonic sort of the unique 64-bit keys, Karras's parallel radix-tree
// construction and a bottom-up pass with one atomic counter per internal node.
#include <math.h>

#include <algorithm>

#include "lt_internal.cuh"

using namespace ltk;

namespace {

// ------------------------------------------------------------------ bitonic sort
__global__ void k_bitonic_step(unsigned long long* keys, int64_t n, int64_t j, int64_t k) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = i ^ j;
        if (l > i) {
            const unsigned long long a = keys[i], b = keys[l];
            const bool up = (i & k) == 0;
            if ((a > b) == up) {
                keys[i] = b;
                keys[l] = a;
            }
        }
    }
}

// Chunks of kSortChunk keys in shared memory.  first: sorts every chunk (all k up to
// the chunk, alternating direction); otherwise the steps j < kSortChunk of one k.
// A launch does up to 78 steps of the network where the global step does one: 377
// launches for the sorts of 16384 lights and 65536 points become 31.  (With the records of
// the cut below and the sums of the k-means: setup of that scene 8.03 to 5.01 ms.)
constexpr int kSortChunk = 4096;

__global__ void __launch_bounds__(1024) k_bitonic_chunk(unsigned long long* keys, int64_t n, int64_t k, bool first) {
    __shared__ unsigned long long sk[kSortChunk];
    const int64_t base = blockIdx.x * (int64_t)kSortChunk;
    const int cnt = (int)(n - base < kSortChunk ? n - base : kSortChunk);  // a power of two
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) sk[i] = keys[base + i];
    __syncthreads();
    for (int64_t kk = first ? 2 : k; kk <= (first ? (int64_t)cnt : k); kk <<= 1) {
        for (int j = (int)((kk < cnt ? kk : cnt) >> 1); j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < cnt / 2; i += blockDim.x) {
                const int a = 2 * i - (i & (j - 1)), b = a + j;  // the i-th pair of distance j
                const unsigned long long x = sk[a], y = sk[b];
                if ((x > y) == (((base + a) & kk) == 0)) {
                    sk[a] = y;
                    sk[b] = x;
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) keys[base + i] = sk[i];
}

lt_status bitonic_sort(lt_ctx* ctx, unsigned long long* keys, int64_t npow2) {
    if (npow2 < 2) return LT_OK;
    const int blocks = (int)std::min<int64_t>((npow2 + 255) / 256, 8 * (int64_t)ctx->num_sms);
    const unsigned chunks = (unsigned)((npow2 + kSortChunk - 1) / kSortChunk);
    k_bitonic_chunk<<<chunks, 1024, 0, ctx->stream>>>(keys, npow2, 0, true);
    LT_LAUNCH_CHECK(ctx, "k_bitonic_chunk");
    for (int64_t k = 2 * kSortChunk; k <= npow2; k <<= 1) {
        for (int64_t j = k >> 1; j >= kSortChunk; j >>= 1) {
            k_bitonic_step<<<blocks, 256, 0, ctx->stream>>>(keys, npow2, j, k);
            LT_LAUNCH_CHECK(ctx, "k_bitonic_step");
        }
        k_bitonic_chunk<<<chunks, 1024, 0, ctx->stream>>>(keys, npow2, k, false);
        LT_LAUNCH_CHECK(ctx, "k_bitonic_chunk");
    }
    return LT_OK;
}

int64_t next_pow2(int64_t x) {
    int64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

// ------------------------------------------------------------------ Morton keys
__device__ __forceinline__ uint32_t expand10(uint32_t v) {
    uint32_t out = 0;
    for (int b = 0; b < 10; ++b) out |= ((v >> b) & 1u) << (3 * b);
    return out;
}

__device__ __forceinline__ uint32_t morton3(float3 p, const float* lo, const float* ext) {
    const float pa[3] = {p.x, p.y, p.z};
    uint32_t q[3];
    for (int a = 0; a < 3; ++a) {
        const float x = __fdiv_rn(__fsub_rn(pa[a], lo[a]), ext[a]);
        int v = (int)floorf(__fmul_rn(x, 1024.0f));
        v = v < 0 ? 0 : (v > 1023 ? 1023 : v);
        q[a] = (uint32_t)v;
    }
    return (expand10(q[0]) << 2) | (expand10(q[1]) << 1) | expand10(q[2]);
}

// Single-block bounding box of a float4 plane (xyz of plane 0).
__global__ void k_bbox(const float4* __restrict__ pl, int64_t n, float* out6) {
    __shared__ float red[6][32];
    float lo[3] = {3e38f, 3e38f, 3e38f}, hi[3] = {-3e38f, -3e38f, -3e38f};
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const float4 p = pl[i];
        lo[0] = fminf(lo[0], p.x);
        lo[1] = fminf(lo[1], p.y);
        lo[2] = fminf(lo[2], p.z);
        hi[0] = fmaxf(hi[0], p.x);
        hi[1] = fmaxf(hi[1], p.y);
        hi[2] = fmaxf(hi[2], p.z);
    }
    for (int a = 0; a < 3; ++a) {
        lo[a] = warp_min(lo[a]);
        hi[a] = warp_max(hi[a]);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
        for (int a = 0; a < 3; ++a) {
            red[a][wid] = lo[a];
            red[3 + a][wid] = hi[a];
        }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int a = 0; a < 3; ++a) {
            float l = 3e38f, h = -3e38f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
                l = fminf(l, red[a][w]);
                h = fmaxf(h, red[3 + a][w]);
            }
            out6[a] = l;
            const float e = __fsub_rn(h, l);
            out6[3 + a] = e > 0.f ? e : 1.0f;  // extent
        }
    }
}

__global__ void k_vpl_keys(const float4* __restrict__ vpls, int64_t n, const float* __restrict__ box,
                           int64_t npad, unsigned long long* keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npad; i += (int64_t)gridDim.x * blockDim.x) {
        if (i >= n) {
            keys[i] = ~0ull;
            continue;
        }
        const float4 p = vpls[i], nr = vpls[n + i];
        const uint32_t code = morton3(make_float3(p.x, p.y, p.z), box, box + 3);
        int ax = 0;
        float best = fabsf(nr.x);
        if (fabsf(nr.y) > best) {
            ax = 1;
            best = fabsf(nr.y);
        }
        if (fabsf(nr.z) > best) ax = 2;
        const float comp = ax == 0 ? nr.x : (ax == 1 ? nr.y : nr.z);
        const uint32_t cls = 2u * ax + (comp > 0.f ? 1u : 0u);
        const unsigned long long hi = ((unsigned long long)cls << 30) | code;
        keys[i] = (hi << 32) | (unsigned long long)i;
    }
}

__device__ __forceinline__ int delta(const unsigned long long* k, int64_t n, int64_t i, int64_t j) {
    if (j < 0 || j > n - 1) return -1;
    return __clzll(k[i] ^ k[j]);
}

// Karras (HPG 2012): internal node i finds its key range and its split.
__global__ void k_karras(const unsigned long long* __restrict__ keys, int64_t n, lt_tree T) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n - 1; i += (int64_t)gridDim.x * blockDim.x) {
        const int d = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) > 0 ? 1 : -1;
        const int dmin = delta(keys, n, i, i - d);
        int64_t lmax = 2;
        while (delta(keys, n, i, i + lmax * d) > dmin) lmax *= 2;
        int64_t l = 0;
        for (int64_t t = lmax / 2; t >= 1; t /= 2)
            if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
        const int64_t j = i + l * d;
        const int dnode = delta(keys, n, i, j);
        int64_t s = 0;
        for (int64_t div = 2;; div *= 2) {
            const int64_t t = (l + div - 1) / div;
            if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
            if (t <= 1) break;
        }
        const int64_t gamma = i + s * d + min(d, 0);
        const int64_t a = min(i, j), b = max(i, j);
        const int64_t left = (a == gamma) ? (n - 1 + gamma) : gamma;
        const int64_t right = (b == gamma + 1) ? (n - 1 + gamma + 1) : gamma + 1;
        T.child[2 * i] = (int32_t)left;
        T.child[2 * i + 1] = (int32_t)right;
        T.parent[left] = (int32_t)i;
        T.parent[right] = (int32_t)i;
        T.range[2 * i] = (int32_t)a;
        T.range[2 * i + 1] = (int32_t)b;
    }
}

__global__ void k_tree_leaves(const unsigned long long* __restrict__ keys, const float4* __restrict__ vpls, int64_t n,
                              lt_tree T, int32_t* flags) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const int v = (int)(keys[j] & 0xffffffffu);
        const int64_t node = n - 1 + j;
        const float4 p = vpls[v], nr = vpls[n + v], L = vpls[2 * n + v];
        T.order[j] = v;
        T.child[2 * node] = -1;
        T.child[2 * node + 1] = -1;
        T.range[2 * node] = (int32_t)j;
        T.range[2 * node + 1] = (int32_t)j;
        T.rep[node] = v;
        T.I[node] = __fmul_rn(L.w, p.w);
        const float e = nr.w;
        T.B[node] = e > 0.f ? 0.5f * kInvPi + 0.5f * (e + 2.f) * (0.5f * kInvPi) : kInvPi;
        float* bb = T.aabb + 6 * node;
        bb[0] = p.x;
        bb[1] = p.y;
        bb[2] = p.z;
        bb[3] = p.x;
        bb[4] = p.y;
        bb[5] = p.z;
        if (j < n - 1) flags[j] = 0;
    }
    if (n == 1 && blockIdx.x == 0 && threadIdx.x == 0) T.parent[0] = -1;
}

// Bottom-up records: the second thread to reach a node combines its children.
__global__ void k_tree_up(int64_t n, lt_tree T, int32_t* flags) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        int64_t node = n - 1 + j;
        for (int guard = 0; guard < 128 && node > 0; ++guard) {
            const int p = T.parent[node];
            __threadfence();
            if (atomicAdd(&flags[p], 1) == 0) break;
            __threadfence();
            const int a = T.child[2 * p], b = T.child[2 * p + 1];
            const float Ia = *(volatile float*)&T.I[a], Ib = *(volatile float*)&T.I[b];
            T.I[p] = __fadd_rn(Ia, Ib);
            T.B[p] = fmaxf(*(volatile float*)&T.B[a], *(volatile float*)&T.B[b]);
            T.rep[p] = Ia >= Ib ? *(volatile int*)&T.rep[a] : *(volatile int*)&T.rep[b];
            for (int q = 0; q < 3; ++q) {
                T.aabb[6 * p + q] = fminf(*(volatile float*)&T.aabb[6 * a + q], *(volatile float*)&T.aabb[6 * b + q]);
                T.aabb[6 * p + 3 + q] =
                    fmaxf(*(volatile float*)&T.aabb[6 * a + 3 + q], *(volatile float*)&T.aabb[6 * b + 3 + q]);
            }
            node = p;
        }
    }
}

// ------------------------------------------------------------------ global cut
__device__ __forceinline__ float brdf_max(float alb, float gloss) {
    return gloss > 0.f ? 0.5f * alb * kInvPi + 0.5f * alb * (gloss + 2.f) * (0.5f * kInvPi) : alb * kInvPi;
}

// What a refinement round reads of a test row (once per setup) and of a cut node (once
// per round), gathered into records that the passes over rows and nodes read in order.
__global__ void k_cut_rows(const float4* __restrict__ pts, int64_t m, const int32_t* __restrict__ rows, int64_t nr,
                           float4* __restrict__ rec) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < nr; x += (int64_t)gridDim.x * blockDim.x) {
        const PointRec P = load_rec(pts, m, rows[x]);
        rec[x] = P.a;
        rec[nr + x] = P.b;
        rec[2 * nr + x] = P.c;
        rec[3 * nr + x] = make_float4(P.a.x, P.a.y, P.a.z, brdf_max(P.a.w, P.b.w));
    }
}

struct CutRecs {
    float4* l;     // [3][most] record of the representative VPL
    float4* box;   // [2][most] (lo xyz, hi x) (hi yz, I B, scale)
};

// The refinement runs on the device from the first round to the last: its kernels read the
// size of the cut, and whether it is done, from here.  (With a copy of the errors to the host, a
// sort there and the new cut back every round, and the forest built on the host, the setup
// of 65536 points and 16384 lights took 5.01 ms; 2.96 ms so.)
struct CutState {
    int32_t C;
    int32_t done;
    int32_t rounds;
};

__global__ void k_cut_state(CutState* st, int C) { *st = CutState{C, 0, 0}; }

__global__ void k_cut_nodes(const float4* __restrict__ vpls, int64_t n, lt_tree T, const int32_t* __restrict__ cut,
                            const CutState* __restrict__ st, int64_t most, CutRecs q) {
    if (st->done) return;
    const int C = st->C;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < C; c += gridDim.x * blockDim.x) {
        const int node = cut[c];
        const PointRec L = load_rec(vpls, n, T.rep[node]);
        const float* bb = T.aabb + 6 * (int64_t)node;
        q.l[c] = L.a;
        q.l[most + c] = L.b;
        q.l[2 * most + c] = L.c;
        q.box[c] = make_float4(bb[0], bb[1], bb[2], bb[3]);
        q.box[most + c] = make_float4(bb[4], bb[5], T.I[node] * T.B[node], __fdiv_rn(T.I[node], __fmul_rn(L.c.w, L.a.w)));
    }
}

// estimate(x) = sum over cut nodes of the unoccluded A(x, c); one CTA per test row.  The
// threads evaluate 256 nodes at a time; lane l of the first warp adds the terms l, l + 32,
// ... in that order and the lanes' sums are added by a butterfly (a warp per row alone
// leaves a chain of C / 32 dependent evaluations).
constexpr int kCutThreads = 256;

__global__ void __launch_bounds__(kCutThreads) k_cut_estimate(const float4* __restrict__ rec, int64_t nr, CutRecs q,
                                                              const CutState* __restrict__ st, int64_t most,
                                                              float dmin2, float* __restrict__ est) {
    __shared__ float2 v[2][kCutThreads];
    if (st->done) return;
    const int C = st->C;
    const int lane = threadIdx.x & 31;
    for (int64_t x = blockIdx.x; x < nr; x += gridDim.x) {
        PointRec P;
        P.a = rec[x];
        P.b = rec[nr + x];
        P.c = rec[2 * nr + x];
        float acc = 0.f;
        int h = 0;
        for (int c0 = 0; c0 < C; c0 += kCutThreads, h ^= 1) {
            const int c = c0 + threadIdx.x;
            float u = 0.f, sc = 0.f;
            if (c < C) {
                PointRec L;
                L.a = q.l[c];
                L.b = q.l[most + c];
                L.c = q.l[2 * most + c];
                sc = q.box[most + c].w;
                u = unoccluded(P, L, dmin2);
            }
            v[h][threadIdx.x] = make_float2(u, sc);  // u sc enters the sum through one multiply-add
            __syncthreads();
            if (threadIdx.x < 32) {
                const int k1 = min(kCutThreads, C - c0);
                for (int k = lane; k < k1; k += 32) acc = fmaf(v[h][k].x, v[h][k].y, acc);
            }
        }
        if (threadIdx.x < 32) {
            acc = warp_sum(acc);
            if (lane == 0) est[x] = acc;
        }
        __syncthreads();
    }
}

// error(c) = max over rows of bound(x, c) / estimate(x).  Small cuts: all 8 warps of a CTA
// on one node, until the nodes alone fill the chip (a maximum does not depend on the order).
__global__ void __launch_bounds__(kCutThreads) k_cut_error(const float4* __restrict__ rec, int64_t nr, CutRecs q,
                                                           const CutState* __restrict__ st, int64_t most,
                                                           const float* __restrict__ est, float dmin2,
                                                           float* __restrict__ err) {
    __shared__ float red[kCutThreads / 32];
    if (st->done) return;
    const int C = st->C;
    const int wpn = C < (int)gridDim.x ? 8 : C < 4 * (int)gridDim.x ? 2 : 1;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nodes = (kCutThreads / 32) / wpn;  // nodes of the CTA
    const int part = wid % wpn;
    const float4* row = rec + 3 * nr;
    for (int64_t c0 = blockIdx.x * (int64_t)nodes; c0 < C; c0 += (int64_t)gridDim.x * nodes) {
        const int64_t ci = c0 + wid / wpn;
        float e = 0.f;
        if (ci < C) {
            const float4 b0 = q.box[ci], b1 = q.box[most + ci];
            for (int64_t x = part * 32 + lane; x < nr; x += 32 * wpn) {
                const float4 p = __ldg(row + x);
                const float gx = fmaxf(0.f, fmaxf(b0.x - p.x, p.x - b0.w));
                const float gy = fmaxf(0.f, fmaxf(b0.y - p.y, p.y - b1.x));
                const float gz = fmaxf(0.f, fmaxf(b0.z - p.z, p.z - b1.y));
                const float d2 = gx * gx + gy * gy + gz * gz;
                const float b = b1.z * p.w / fmaxf(d2, dmin2);
                const float ex = est[x];
                const float ratio = ex > 0.f ? b / ex : (b > 0.f ? INFINITY : 0.f);
                e = fmaxf(e, ratio);
            }
        }
        e = warp_max(e);
        if (lane == 0) red[wid] = e;
        __syncthreads();
        if (ci < C && part == 0 && lane == 0) {
            for (int k = 1; k < wpn; ++k) e = fmaxf(e, red[wid + k]);
            err[ci] = e;
        }
        __syncthreads();
    }
}

// One refinement round: of the internal nodes of error above eps the `take` largest errors
// (ties: the lower node) are split in place, so that the cut stays in leaf order.  take is
// all of them, at most floor(growth C) (at least one) and at most max_cut - C.  One CTA: a
// radix select of the take-th key (error descending, node ascending) and one scan.  told, in
// host memory: the rounds so far, INT32_MAX after the last.
constexpr int kRefineThreads = 1024;
constexpr int kMaxRounds = 4096;

__global__ void __launch_bounds__(kRefineThreads) k_cut_refine(const int32_t* __restrict__ child,
                                                               const int32_t* __restrict__ range, int64_t n, float eps,
                                                               int32_t max_cut, float growth, int32_t* __restrict__ cut,
                                                               int32_t* __restrict__ nxt, const float* __restrict__ err,
                                                               CutState* st, volatile int32_t* told) {
    __shared__ int32_t ws[32];
    __shared__ int32_t hist[256];
    __shared__ unsigned long long sel[2];
    __shared__ int32_t krem;
    if (st->done) return;
    const int C = st->C;
    const int run = (C + kRefineThreads - 1) / kRefineThreads;
    const int lo = min(C, (int)threadIdx.x * run), hi = min(C, lo + run);
    auto wants = [&](int i) { return cut[i] < n - 1 && err[i] > eps; };
    auto key_of = [&](int i) {
        return (unsigned long long)(~__float_as_uint(err[i])) << 32 | (unsigned long long)(uint32_t)cut[i];
    };
    int mine = 0;
    for (int i = lo; i < hi; ++i) mine += wants(i);
    int cand;
    block_exclusive_scan<int>(mine, ws, &cand);
    int64_t room = (int64_t)max_cut - C;
    const int64_t grow = (int64_t)(growth * (float)C);
    room = min(room, grow > 1 ? grow : (int64_t)1);
    const int take = cand > room ? (int)(room > 0 ? room : 0) : cand;
    if (take == 0) {
        if (threadIdx.x == 0) {
            st->done = 1;
            *told = INT32_MAX;
        }
        return;
    }
    unsigned long long pivot = ~0ull;
    if (take < cand) {
        if (threadIdx.x == 0) {
            sel[0] = sel[1] = 0ull;
            krem = take - 1;
        }
        __syncthreads();
        for (int pass = 7; pass >= 0; --pass) {
            if (threadIdx.x < 256) hist[threadIdx.x] = 0;
            __syncthreads();
            const unsigned long long prefix = sel[0], mask = sel[1];
            for (int i = threadIdx.x; i < C; i += kRefineThreads)
                if (wants(i)) {
                    const unsigned long long k = key_of(i);
                    if ((k & mask) == prefix) atomicAdd(&hist[(k >> (8 * pass)) & 255], 1);
                }
            __syncthreads();
            if (threadIdx.x < 32) {  // the digit that holds position krem: eight counts a lane
                const int lane = threadIdx.x;
                int c[8], sum = 0;
#pragma unroll
                for (int b = 0; b < 8; ++b) sum += c[b] = hist[8 * lane + b];
                int before = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, before, o);
                    if (lane >= o) before += y;
                }
                before -= sum;
                const int k = krem;
                __syncwarp();
                if (before <= k && k < before + sum) {
                    int b = 0;
                    while (k >= before + c[b]) before += c[b++];
                    krem = k - before;
                    sel[0] = prefix | ((unsigned long long)(8 * lane + b) << (8 * pass));
                    sel[1] = mask | (255ull << (8 * pass));
                }
            }
            __syncthreads();
        }
        pivot = sel[0];
    }
    auto split = [&](int i) { return wants(i) && (take == cand || key_of(i) <= pivot); };
    int grown = 0;
    for (int i = lo; i < hi; ++i) grown += 1 + split(i);
    int total;
    int at = block_exclusive_scan<int>(grown, ws, &total);
    for (int i = lo; i < hi; ++i) {
        if (split(i)) {
            const int64_t a = child[2 * (int64_t)cut[i]], b = child[2 * (int64_t)cut[i] + 1];
            const bool swap = range[2 * b] < range[2 * a];  // a caller's tree may name the right child first
            nxt[at++] = (int32_t)(swap ? b : a);
            nxt[at++] = (int32_t)(swap ? a : b);
        } else {
            nxt[at++] = cut[i];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < total; i += kRefineThreads) cut[i] = nxt[i];
    if (threadIdx.x == 0) {
        st->C = total;
        const int rounds = ++st->rounds;
        const bool end = (take < cand && total >= max_cut) || rounds >= kMaxRounds;
        if (end) st->done = 1;
        *told = end ? INT32_MAX : rounds;
    }
}

// ------------------------------------------------------------------ forest of the cut
// The ancestors of the cut's nodes as a forest: leaves are the cut in order, internal nodes
// its ancestors by tree id.
struct ForestState {
    int32_t err;      // 1: a cut node out of range or repeated, 2: not a partition
    int32_t inner;    // ancestors found
    int32_t height;
};
constexpr int kMaxHeight = 2046;

__global__ void k_fo_init(int64_t NN, int C, int32_t* __restrict__ local, int32_t* __restrict__ anc,
                          int32_t* __restrict__ arrived, ForestState* st) {
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = i0; x < NN; x += step) {
        local[x] = -1;
        anc[x] = 0;
    }
    for (int64_t x = i0; x < C; x += step) arrived[x] = 0;
    if (i0 == 0) *st = ForestState{0, 0, 0};
}

__global__ void k_fo_mark(int64_t NN, const int32_t* __restrict__ parent, const int32_t* __restrict__ cut, int C,
                          int32_t* local, int32_t* anc, ForestState* st) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < C; c += gridDim.x * blockDim.x) {
        const int node = cut[c];
        if (node < 0 || node >= NN || atomicCAS(&local[node], -1, c) != -1) {
            atomicMax(&st->err, 1);
            continue;
        }
        // up to the first ancestor that another node has marked (the tree is at most 64 deep)
        for (int x = parent[node], it = 0; x >= 0 && it < kMaxHeight && atomicExch(&anc[x], 1) == 0; ++it) x = parent[x];
    }
}

// ancestors by tree id: a run of the tree per thread, one scan
__global__ void __launch_bounds__(1024) k_fo_scan(int64_t NN, int C, const int32_t* __restrict__ anc,
                                                  int32_t* __restrict__ local, int32_t* __restrict__ inner, ForestState* st) {
    __shared__ int32_t ws[32];
    const int64_t run = (NN + 1023) / 1024, lo = min(NN, (int64_t)threadIdx.x * run), hi = min(NN, lo + run);
    int mine = 0;
    for (int64_t x = lo; x < hi; ++x) mine += anc[x];
    int total;
    int at = block_exclusive_scan<int>(mine, ws, &total);
    if (threadIdx.x == 0) {
        st->inner = total;
        if (total != C - 1 && st->err == 0) st->err = 2;
    }
    if (total != C - 1) return;
    for (int64_t x = lo; x < hi; ++x)
        if (anc[x]) {
            inner[at] = (int32_t)x;
            local[x] = C + at++;
        }
}

// children of every ancestor, parents of all nodes (par: the root has none)
__global__ void k_fo_nodes(const int32_t* __restrict__ child, int C, const int32_t* __restrict__ local,
                           const int32_t* __restrict__ inner, int2* __restrict__ kid, int32_t* __restrict__ par,
                           ForestState* st) {
    if (st->err) return;
    const int i0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (i0 == 0) par[C > 1 ? C : 0] = -1;
    for (int i = i0; i < C - 1; i += gridDim.x * blockDim.x) {
        const int a = local[child[2 * (int64_t)inner[i]]], b = local[child[2 * (int64_t)inner[i] + 1]];
        kid[i] = make_int2(a, b);
        if (a < 0 || b < 0) {
            atomicMax(&st->err, 2);
        } else {
            par[a] = C + i;
            par[b] = C + i;
        }
    }
}

// leaf ranges and heights (span: first leaf, last leaf, height): the second child to arrive
// at a node combines both
__global__ void k_fo_up(int C, const int2* __restrict__ kid, const int32_t* __restrict__ par, int32_t* span,
                        int32_t* arrived, ForestState* st) {
    if (st->err) return;
    volatile int32_t* v = span;
    auto get = [&](int x, int k) { return x < C ? (k < 2 ? x : 0) : v[4 * (int64_t)(x - C) + k]; };
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < C; c += gridDim.x * blockDim.x) {
        int x = par[c];
        for (int it = 0; x >= C && it <= kMaxHeight; ++it) {
            __threadfence();
            if (atomicAdd(&arrived[x - C], 1) == 0) break;
            __threadfence();
            const int2 k = kid[x - C];
            const int64_t f = 4 * (int64_t)(x - C);
            v[f] = min(get(k.x, 0), get(k.y, 0));
            v[f + 1] = max(get(k.x, 1), get(k.y, 1));
            const int h = 1 + max(get(k.x, 2), get(k.y, 2));
            v[f + 2] = h;
            atomicMax(&st->height, h);
            x = par[x];
        }
    }
}

// The caller's arrays, which are written only when nothing is refused.  The first CTA lists
// the internal nodes of every height by id, and where each height starts: a run of the
// nodes per thread, one scan per height, the heights of the first kHeightStage nodes in
// shared memory (one CTA waits on each read; read from memory once per height, the setup
// of 65536 points and 16384 lights took 3.00 ms instead of 2.88).  The others write the forest.
constexpr int kHeightStage = 16384;

__global__ void __launch_bounds__(1024) k_fo_out(int C, const int32_t* __restrict__ cut, const int32_t* __restrict__ inner,
                                                 const int2* __restrict__ kid, const int32_t* __restrict__ par,
                                                 const int32_t* __restrict__ span, int32_t max_levels,
                                                 int32_t* __restrict__ forest, int32_t* __restrict__ level_off,
                                                 int32_t* __restrict__ level_nodes, const ForestState* __restrict__ st) {
    __shared__ int32_t ws[32];
    __shared__ uint16_t hs[kHeightStage];
    const int H = st->height;
    if (st->err || H > max_levels || H > kMaxHeight) return;
    if (blockIdx.x > 0) {
        for (int x = (blockIdx.x - 1) * 1024 + threadIdx.x; x < 2 * C - 1; x += (gridDim.x - 1) * 1024) {
            int32_t* f = forest + 8 * (int64_t)x;
            const int32_t* sp = span + 4 * (int64_t)(x - C);
            const int2 k = x < C ? make_int2(-1, -1) : kid[x - C];
            f[0] = x < C ? cut[x] : inner[x - C];
            f[1] = k.x;
            f[2] = k.y;
            f[3] = par[x];
            f[4] = x < C ? x : sp[0];
            f[5] = x < C ? x : sp[1];
            f[6] = x < C ? 0 : sp[2];
            f[7] = 0;
        }
        return;
    }
    for (int i = threadIdx.x; i < min(C - 1, kHeightStage); i += 1024) hs[i] = (uint16_t)span[4 * (int64_t)i + 2];
    __syncthreads();
    auto height = [&](int i) { return i < kHeightStage ? (int)hs[i] : span[4 * (int64_t)i + 2]; };
    const int run = (C - 1 + 1023) / 1024, lo = min(C - 1, (int)threadIdx.x * run), hi = min(C - 1, lo + run);
    int start = 0;
    if (threadIdx.x == 0) level_off[0] = 0;
    for (int h = 1; h <= H; ++h) {
        int mine = 0;
        for (int i = lo; i < hi; ++i) mine += height(i) == h;
        int total;
        int at = start + block_exclusive_scan<int>(mine, ws, &total);
        for (int i = lo; i < hi && mine > 0; ++i)
            if (height(i) == h) level_nodes[at++] = C + i;
        if (threadIdx.x == 0) level_off[h] = start;
        start += total;
    }
    if (threadIdx.x == 0) level_off[H + 1] = start;
}

// slice_off[0..S] from the clusters' counts
__global__ void k_slice_off(const int32_t* __restrict__ counts, int S, int32_t* __restrict__ off) {
    __shared__ int32_t ws[32];
    int carry = 0;
    for (int s0 = 0; s0 < S; s0 += blockDim.x) {
        const int s = s0 + threadIdx.x;
        int total;
        const int pre = block_exclusive_scan<int>(s < S ? counts[s] : 0, ws, &total);
        if (s < S) off[s] = carry + pre;
        carry += total;
    }
    if (threadIdx.x == 0) off[S] = carry;
}

// ------------------------------------------------------------------ k-means
__global__ void k_point_keys(const float4* __restrict__ pts, int64_t m, const float* __restrict__ box, int64_t npad,
                             unsigned long long* keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npad; i += (int64_t)gridDim.x * blockDim.x) {
        if (i >= m) {
            keys[i] = ~0ull;
            continue;
        }
        const float4 p = pts[i];
        keys[i] = ((unsigned long long)morton3(make_float3(p.x, p.y, p.z), box, box + 3) << 32) |
                  (unsigned long long)i;
    }
}

__device__ __forceinline__ void feature(const float4* pts, int64_t m, int64_t i, float w, float* f) {
    const float4 p = pts[i], nr = pts[m + i];
    f[0] = p.x;
    f[1] = p.y;
    f[2] = p.z;
    f[3] = w * nr.x;
    f[4] = w * nr.y;
    f[5] = w * nr.z;
}

__global__ void k_kmeans_seed(const float4* __restrict__ pts, int64_t m, const unsigned long long* __restrict__ keys,
                              int S, float w, float* cen) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < S; k += gridDim.x * blockDim.x) {
        const int64_t rank = (2 * (int64_t)k + 1) * m / (2 * (int64_t)S);
        const int64_t i = (int64_t)(keys[rank] & 0xffffffffu);
        feature(pts, m, i, w, cen + 6 * k);
    }
}

// Nearest centroid of every point and the sums of the clusters.  Points in image order
// put a warp's points into few clusters: the lanes of a cluster add up by shuffles and one
// of them adds to the cluster (the values are float32 and the sums float64, wide enough that
// their order does not show).  A cluster of fewer than kMinLanes of the warp's points takes
// their atomics one by one, as all do where the points come in no order.
// Slices of 65536 points in image order / in random order, ms: 64 clusters 2.00 / 1.83 with an
// atomic a value, 0.68 / 1.78 with every cluster of a warp by shuffles, 0.64 / 0.93 so; 512 clusters
// 1.75 / 1.71, 1.10 / 2.33, 0.95 / 0.79.  (From 3 lanes on 0.96 / 0.79, from 6 0.89 / 0.79, but then 16
// clusters in random order take 1.32 where they took 1.17; 1.16 so.)
constexpr int kMinLanes = 4;

__global__ void k_kmeans_assign(const float4* __restrict__ pts, int64_t m, int S, float w,
                                const float* __restrict__ cen, int32_t* __restrict__ lab, double* sums) {
    extern __shared__ float sc[];  // [S][6]
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 6 * S; i += blockDim.x) sc[i] = cen[i];
    __syncthreads();
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x; i0 < m; i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = i0 + threadIdx.x;
        float f[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        int best = -1;
        if (i < m) {
            feature(pts, m, i, w, f);
            best = 0;
            float bd = 3e38f;
            for (int k = 0; k < S; ++k) {
                float d = 0.f;
                for (int a = 0; a < 6; ++a) {
                    const float t = f[a] - sc[6 * k + a];
                    d += t * t;
                }
                if (d < bd) {
                    bd = d;
                    best = k;
                }
            }
            lab[i] = best;
        }
        if (!sums) continue;
        const unsigned peers = __match_any_sync(FULL, best);  // (every lane of the warp takes part)
        const bool many = best >= 0 && __popc(peers) >= kMinLanes;
        if (best >= 0 && !many) {
            double* sk = sums + 7 * best;
#pragma unroll
            for (int a = 0; a < 6; ++a) atomicAdd(sk + a, (double)f[a]);
            atomicAdd(sk + 6, 1.0);
        }
        unsigned left = __ballot_sync(FULL, many);
        while (left) {  // one cluster of the warp at a time
            const int k = __shfl_sync(FULL, best, __ffs(left) - 1);
            const unsigned mine = __ballot_sync(FULL, best == k);
            double v[6];
#pragma unroll
            for (int a = 0; a < 6; ++a) v[a] = warp_sum<double>(best == k ? (double)f[a] : 0.0);
            double* sk = sums + 7 * k;
#pragma unroll
            for (int a = 0; a < 6; ++a)
                if (lane == a) atomicAdd(sk + a, v[a]);
            if (lane == 6) atomicAdd(sk + 6, (double)__popc(mine));
            left &= ~mine;
        }
    }
}

__global__ void k_kmeans_update(int S, const double* __restrict__ sums, float* cen) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < S; k += gridDim.x * blockDim.x) {
        const double cnt = sums[7 * k + 6];
        if (cnt > 0)
            for (int a = 0; a < 6; ++a) cen[6 * k + a] = (float)(sums[7 * k + a] / cnt);
    }
}

__global__ void k_label_keys(const int32_t* __restrict__ lab, int64_t m, int64_t npad, unsigned long long* keys,
                             int32_t* counts) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npad; i += (int64_t)gridDim.x * blockDim.x) {
        if (i >= m) {
            keys[i] = ~0ull;
            continue;
        }
        keys[i] = ((unsigned long long)lab[i] << 32) | (unsigned long long)i;
        atomicAdd(&counts[lab[i]], 1);
    }
}

__global__ void k_perm_from_keys(const unsigned long long* __restrict__ keys, int64_t m, int32_t* perm) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        perm[i] = (int32_t)(keys[i] & 0xffffffffu);
}

bool tree_ok(const lt_tree* t) {
    return t && t->n >= 1 && t->order && t->child && t->parent && t->range && t->rep && t->I && t->B && t->aabb;
}

// ------------------------------------------------------------------ triangle BVH
// Linear BVH over triangles (the paper casts its shadow rays through a BVH, Sec. 6):
// Morton codes of the centroids in the centroids' box, sorted with the triangle index
// below them, the Karras topology, leaf boxes and a bottom-up refit.
__global__ void k_tri_prep(const float* __restrict__ tris, int64_t nt, float4* __restrict__ cen,
                           float4* __restrict__ rec) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nt; i += (int64_t)gridDim.x * blockDim.x) {
        const float* t = tris + 9 * i;
        const float3 a = make_float3(t[0], t[1], t[2]), b = make_float3(t[3], t[4], t[5]),
                     c = make_float3(t[6], t[7], t[8]);
        cen[i] = make_float4((a.x + b.x + c.x) * (1.f / 3.f), (a.y + b.y + c.y) * (1.f / 3.f),
                             (a.z + b.z + c.z) * (1.f / 3.f), 0.f);
        rec[3 * i] = make_float4(a.x, a.y, a.z, 0.f);
        rec[3 * i + 1] = make_float4(b.x - a.x, b.y - a.y, b.z - a.z, 0.f);
        rec[3 * i + 2] = make_float4(c.x - a.x, c.y - a.y, c.z - a.z, 0.f);
    }
}

__global__ void k_tri_keys(const float4* __restrict__ cen, int64_t nt, const float* __restrict__ box, int64_t npad,
                           unsigned long long* keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npad; i += (int64_t)gridDim.x * blockDim.x) {
        if (i >= nt) {
            keys[i] = ~0ull;
            continue;
        }
        const float4 c = cen[i];
        keys[i] = ((unsigned long long)morton3(make_float3(c.x, c.y, c.z), box, box + 3) << 32) |
                  (unsigned long long)i;
    }
}

__global__ void k_bvh_leaves(const unsigned long long* __restrict__ keys, const float* __restrict__ tris, int64_t nt,
                             int32_t* __restrict__ leaf_tri, float* __restrict__ aabb, int32_t* __restrict__ parent,
                             int32_t* __restrict__ flags) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nt; j += (int64_t)gridDim.x * blockDim.x) {
        const int t = (int)(keys[j] & 0xffffffffu);
        leaf_tri[j] = t;
        const float* v = tris + 9 * (int64_t)t;
        float* bb = aabb + 6 * (nt - 1 + j);
        for (int a = 0; a < 3; ++a) {
            bb[a] = fminf(v[a], fminf(v[3 + a], v[6 + a]));
            bb[3 + a] = fmaxf(v[a], fmaxf(v[3 + a], v[6 + a]));
        }
        if (j < nt - 1) flags[j] = 0;
    }
    if (nt == 1 && blockIdx.x == 0 && threadIdx.x == 0) parent[0] = -1;
}

// bottom-up boxes: the second thread to reach a node combines its children
__global__ void k_bvh_up(int64_t nt, const int32_t* __restrict__ child, const int32_t* __restrict__ parent,
                         float* aabb, int32_t* flags) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nt; j += (int64_t)gridDim.x * blockDim.x) {
        int64_t node = nt - 1 + j;
        for (int guard = 0; guard < 128 && node > 0; ++guard) {
            const int p = parent[node];
            __threadfence();
            if (atomicAdd(&flags[p], 1) == 0) break;
            __threadfence();
            const int a = child[2 * p], b = child[2 * p + 1];
            for (int q = 0; q < 3; ++q) {
                aabb[6 * p + q] = fminf(*(volatile float*)&aabb[6 * a + q], *(volatile float*)&aabb[6 * b + q]);
                aabb[6 * p + 3 + q] =
                    fmaxf(*(volatile float*)&aabb[6 * a + 3 + q], *(volatile float*)&aabb[6 * b + 3 + q]);
            }
            node = p;
        }
    }
}

// the records the walk reads: both children's boxes and ids per internal node, and the
// triangles in leaf order
__global__ void k_bvh_pack(int64_t nt, const int32_t* __restrict__ child, const float* __restrict__ aabb,
                           const int32_t* __restrict__ leaf_tri, const float4* __restrict__ rec,
                           float4* __restrict__ node, float4* __restrict__ leaf) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nt; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = leaf_tri[i];
        for (int k = 0; k < 3; ++k) leaf[3 * i + k] = rec[3 * t + k];
        if (i == nt - 1) continue;
        const int a = child[2 * i], b = child[2 * i + 1];
        const float *A = aabb + 6 * (int64_t)a, *B = aabb + 6 * (int64_t)b;
        node[4 * i] = make_float4(A[0], A[1], A[2], A[3]);
        node[4 * i + 1] = make_float4(A[4], A[5], B[0], B[1]);
        node[4 * i + 2] = make_float4(B[2], B[3], B[4], B[5]);
        node[4 * i + 3] = make_float4(__int_as_float(a), __int_as_float(b), 0.f, 0.f);
    }
}

}  // namespace

// ------------------------------------------------------------------ tree
extern "C" lt_status lt_build_tree(lt_ctx* ctx, const float* vpls, int64_t n, lt_tree* tree) {
    if (!ctx || !vpls || n < 1 || n > (1 << 28) || !tree_ok(tree) || tree->n != n || ((uintptr_t)vpls & 15))
        return lt_fail(ctx, LT_EINVAL, "lt_build_tree: bad arguments");
    cudaSetDevice(ctx->device);
    const int64_t npad = next_pow2(n);
    lt_status st;
    char* p = (char*)lt_scratch(ctx, SCR_SORT, (size_t)npad * 8 + (size_t)n * 4 + 1024, &st);
    if (!p) return st;
    unsigned long long* keys = (unsigned long long*)p;
    int32_t* flags = (int32_t*)(p + npad * 8);
    float* box = (float*)lt_scratch(ctx, SCR_MISC, 64, &st);
    if (!box) return st;
    const int blocks = (int)std::min<int64_t>((npad + 255) / 256, 16 * (int64_t)ctx->num_sms);
    k_bbox<<<1, 1024, 0, ctx->stream>>>((const float4*)vpls, n, box);
    LT_LAUNCH_CHECK(ctx, "k_bbox");
    k_vpl_keys<<<blocks, 256, 0, ctx->stream>>>((const float4*)vpls, n, box, npad, keys);
    LT_LAUNCH_CHECK(ctx, "k_vpl_keys");
    if ((st = bitonic_sort(ctx, keys, npad)) != LT_OK) return st;
    k_karras<<<blocks, 256, 0, ctx->stream>>>(keys, n, *tree);
    LT_LAUNCH_CHECK(ctx, "k_karras");
    k_tree_leaves<<<blocks, 256, 0, ctx->stream>>>(keys, (const float4*)vpls, n, *tree, flags);
    LT_LAUNCH_CHECK(ctx, "k_tree_leaves");
    if (n > 1) {
        LT_CUDA(ctx, cudaMemsetAsync(tree->parent, 0xff, sizeof(int32_t), ctx->stream));  // root has no parent
        k_tree_up<<<blocks, 256, 0, ctx->stream>>>(n, *tree, flags);
        LT_LAUNCH_CHECK(ctx, "k_tree_up");
    }
    return LT_OK;
}

// ------------------------------------------------------------------ global cut
namespace {
// Scratch of the refinement for nr test rows and cuts of up to `most` nodes.
struct CutWork {
    float4* rec;   // [4][nr]
    CutRecs q;
    float* est;    // [nr]
    float* err;    // [most]
    int32_t* nxt;  // [most]
    CutState* st;
    int64_t most;
};

lt_status cut_work(lt_ctx* ctx, int64_t nr, int64_t most, CutWork* w) {
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t b_rec = up((size_t)nr * 64), b_l = up((size_t)most * 48), b_box = up((size_t)most * 32),
                 b_est = up((size_t)nr * 4);
    lt_status st;
    const size_t b_err = up((size_t)most * 4);
    char* p = (char*)lt_scratch(ctx, SCR_CUT, b_rec + b_l + b_box + b_est + 2 * b_err + 256, &st);
    if (!p) return st;
    w->rec = (float4*)p;
    w->q.l = (float4*)(p + b_rec);
    w->q.box = (float4*)(p + b_rec + b_l);
    w->est = (float*)(p + b_rec + b_l + b_box);
    w->err = (float*)(p + b_rec + b_l + b_box + b_est);
    w->nxt = (int32_t*)(p + b_rec + b_l + b_box + b_est + b_err);
    w->st = (CutState*)(p + b_rec + b_l + b_box + b_est + 2 * b_err);
    w->most = most;
    return LT_OK;
}

lt_status cut_rows(lt_ctx* ctx, const float* pts, int64_t m, const int32_t* rows, int64_t nr, const CutWork& w) {
    k_cut_rows<<<(unsigned)std::min<int64_t>((nr + 255) / 256, 8 * (int64_t)ctx->num_sms), 256, 0, ctx->stream>>>(
        (const float4*)pts, m, rows, nr, w.rec);
    LT_LAUNCH_CHECK(ctx, "k_cut_rows");
    return LT_OK;
}

// est[nr] and err[C] of the cut (device arrays) whose size w.st holds; the refinement's
// per-round errors.
lt_status cut_errors(lt_ctx* ctx, const lt_tree* tree, const float* vpls, int64_t nr, const int32_t* cut, float d_min,
                     const CutWork& w, float* err) {
    const int nsm = ctx->num_sms;
    k_cut_nodes<<<(unsigned)std::min<int64_t>((w.most + 255) / 256, 8 * (int64_t)nsm), 256, 0, ctx->stream>>>(
        (const float4*)vpls, tree->n, *tree, cut, w.st, w.most, w.q);
    LT_LAUNCH_CHECK(ctx, "k_cut_nodes");
    k_cut_estimate<<<(unsigned)std::min<int64_t>(nr, 8 * (int64_t)nsm), kCutThreads, 0, ctx->stream>>>(
        w.rec, nr, w.q, w.st, w.most, d_min * d_min, w.est);
    LT_LAUNCH_CHECK(ctx, "k_cut_estimate");
    k_cut_error<<<8 * nsm, kCutThreads, 0, ctx->stream>>>(w.rec, nr, w.q, w.st, w.most, w.est, d_min * d_min, err);
    LT_LAUNCH_CHECK(ctx, "k_cut_error");
    return LT_OK;
}
}  // namespace

extern "C" lt_status lt_cut_errors(lt_ctx* ctx, const lt_tree* tree, const float* pts, int64_t m, const float* vpls,
                                   const int32_t* rows, int64_t nr, const int32_t* cut, int32_t C, float d_min,
                                   float* err) {
    if (!ctx || !tree_ok(tree) || !pts || !vpls || !rows || nr < 1 || m < 1 || !cut || C < 1 || !err)
        return lt_fail(ctx, LT_EINVAL, "lt_cut_errors: bad arguments");
    cudaSetDevice(ctx->device);
    CutWork w;
    lt_status st = cut_work(ctx, nr, C, &w);
    if (st != LT_OK) return st;
    if ((st = cut_rows(ctx, pts, m, rows, nr, w)) != LT_OK) return st;
    k_cut_state<<<1, 1, 0, ctx->stream>>>(w.st, C);
    LT_LAUNCH_CHECK(ctx, "k_cut_state");
    return cut_errors(ctx, tree, vpls, nr, cut, d_min, w, err);
}

extern "C" lt_status lt_build_global_cut(lt_ctx* ctx, const lt_tree* tree, const float* pts, int64_t m,
                                         const float* vpls, const int32_t* rows, int64_t nr, float eps,
                                         int32_t max_cut, float growth, float d_min, int32_t* cut,
                                         int32_t* cut_size_host) {
    if (!ctx || !tree_ok(tree) || !pts || !vpls || !rows || nr < 1 || m < 1 || max_cut < 1 || !cut ||
        !cut_size_host || !(growth > 0.f))
        return lt_fail(ctx, LT_EINVAL, "lt_build_global_cut: bad arguments");
    cudaSetDevice(ctx->device);
    const int64_t n = tree->n;
    CutWork w;
    lt_status st = cut_work(ctx, nr, std::min<int64_t>(max_cut, n), &w);
    if (st != LT_OK) return st;
    if ((st = cut_rows(ctx, pts, m, rows, nr, w)) != LT_OK) return st;
    LT_CUDA(ctx, cudaMemsetAsync(cut, 0, sizeof(int32_t), ctx->stream));  // the root
    k_cut_state<<<1, 1, 0, ctx->stream>>>(w.st, 1);
    LT_LAUNCH_CHECK(ctx, "k_cut_state");
    // The host launches one round beyond the one that it waits for, from a word in its memory,
    // so that the device goes on without it and at most two rounds are launched past the end
    // (four kernels each that return at once).  us a cut with no round ahead / one / two / four,
    // and with 20 rounds before the first look: ended with its first round 98 / 101 / 107 / 115, 310;
    // 64 lights, 10 rounds, 348 / 314 / 325 / 370, 445; 16384 lights, 21 rounds, 671 / 576 / 589 / 625,
    // 650.  (A word that does not come ends the wait when the stream is idle or failed.)
    constexpr int kAhead = 1, kLook = 64;
    volatile int32_t* told = ctx->h_status + 1;
    CutState* h = reinterpret_cast<CutState*>(ctx->h_status + 2);
    *told = 0;
    h->done = 0;
    for (int round = 1; !h->done; ++round) {
        if ((st = cut_errors(ctx, tree, vpls, nr, cut, d_min, w, w.err)) != LT_OK) return st;
        k_cut_refine<<<1, kRefineThreads, 0, ctx->stream>>>(tree->child, tree->range, n, eps, max_cut, growth, cut, w.nxt,
                                                            w.err, w.st, told);
        LT_LAUNCH_CHECK(ctx, "k_cut_refine");
        while (*told < round - kAhead && cudaStreamQuery(ctx->stream) == cudaErrorNotReady) {
        }
        if (*told != INT32_MAX && round % kLook) continue;
        LT_CUDA(ctx, cudaMemcpyAsync(h, w.st, sizeof(*h), cudaMemcpyDeviceToHost, ctx->stream));
        LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    }
    *cut_size_host = h->C;
    return LT_OK;
}

// ------------------------------------------------------------------ forest of the cut
extern "C" lt_status lt_cut_forest(lt_ctx* ctx, const lt_tree* tree, const int32_t* cut, int32_t C, int32_t* forest,
                                   int32_t* level_off, int32_t max_levels, int32_t* level_nodes,
                                   int32_t* height_host) {
    if (!ctx || !tree_ok(tree) || !cut || C < 1 || !forest || !level_off || max_levels < 1 || !height_host ||
        (C > 1 && !level_nodes))
        return lt_fail(ctx, LT_EINVAL, "lt_cut_forest: bad arguments");
    cudaSetDevice(ctx->device);
    const int64_t NN = 2 * tree->n - 1;
    if (C > tree->n) return lt_fail(ctx, LT_EINVAL, "lt_cut_forest: cut nodes out of range or repeated");
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    lt_status st;
    const size_t b_nn = up((size_t)NN * 4), b_c = up((size_t)C * 4);
    char* p = (char*)lt_scratch(ctx, SCR_CUT, 2 * b_nn + 4 * b_c + up((size_t)C * 16) + 256, &st);
    if (!p) return st;
    int32_t* local = (int32_t*)p;
    int32_t* anc = (int32_t*)(p + b_nn);
    int32_t* par = anc;  // (the marks are not read any more when the parents are written)
    p += 2 * b_nn;
    int32_t* arrived = (int32_t*)p;
    int32_t* inner = (int32_t*)(p + b_c);
    int2* kid = (int2*)(p + 2 * b_c);
    int32_t* span = (int32_t*)(p + 4 * b_c);
    ForestState* fs = (ForestState*)(p + 4 * b_c + up((size_t)C * 16));
    const int most = 8 * ctx->num_sms;
    k_fo_init<<<(unsigned)std::min<int64_t>((NN + 255) / 256, most), 256, 0, ctx->stream>>>(NN, C, local, anc, arrived, fs);
    LT_LAUNCH_CHECK(ctx, "k_fo_init");
    k_fo_mark<<<std::min((C + 127) / 128, most), 128, 0, ctx->stream>>>(NN, tree->parent, cut, C, local, anc, fs);
    LT_LAUNCH_CHECK(ctx, "k_fo_mark");
    k_fo_scan<<<1, 1024, 0, ctx->stream>>>(NN, C, anc, local, inner, fs);
    LT_LAUNCH_CHECK(ctx, "k_fo_scan");
    k_fo_nodes<<<std::min((C + 255) / 256, most), 256, 0, ctx->stream>>>(tree->child, C, local, inner, kid, par, fs);
    LT_LAUNCH_CHECK(ctx, "k_fo_nodes");
    k_fo_up<<<std::min((C + 127) / 128, most), 128, 0, ctx->stream>>>(C, kid, par, span, arrived, fs);
    LT_LAUNCH_CHECK(ctx, "k_fo_up");
    k_fo_out<<<1 + std::min((2 * C + 1023) / 1024, most), 1024, 0, ctx->stream>>>(C, cut, inner, kid, par, span, max_levels,
                                                                                 forest, level_off, level_nodes, fs);
    LT_LAUNCH_CHECK(ctx, "k_fo_out");
    ForestState h{};
    LT_CUDA(ctx, cudaMemcpyAsync(&h, fs, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
    LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    if (h.err == 1) return lt_fail(ctx, LT_EINVAL, "lt_cut_forest: cut nodes out of range or repeated");
    if (h.err) return lt_fail(ctx, LT_EINVAL, "lt_cut_forest: the cut is not a partition");
    if (h.height > max_levels || h.height > kMaxHeight)
        return lt_fail(ctx, LT_EINVAL, "lt_cut_forest: max_levels too small");
    *height_host = h.height;
    return LT_OK;
}

// ------------------------------------------------------------------ slicing
extern "C" lt_status lt_make_slices(lt_ctx* ctx, const float* pts, int64_t m, int32_t S, int32_t iters,
                                    float normal_weight, int32_t* row_perm, int32_t* slice_off) {
    if (!ctx || !pts || m < 1 || S < 1 || S > 4096 || S > m || iters < 0 || !row_perm || !slice_off ||
        ((uintptr_t)pts & 15))
        return lt_fail(ctx, LT_EINVAL, "lt_make_slices: bad arguments");
    cudaSetDevice(ctx->device);
    const int64_t npad = next_pow2(m);
    lt_status st;
    char* p = (char*)lt_scratch(ctx, SCR_SORT,
                                (size_t)npad * 8 + (size_t)m * 4 + (size_t)S * 7 * 8 + (size_t)S * 6 * 4 + S * 4 + 4096,
                                &st);
    if (!p) return st;
    unsigned long long* keys = (unsigned long long*)p;
    int32_t* lab = (int32_t*)(p + npad * 8);
    double* sums = (double*)(p + npad * 8 + ((m * 4 + 255) & ~255LL));
    float* cen = (float*)((char*)sums + ((S * 7 * 8 + 255) & ~255LL));
    int32_t* counts = (int32_t*)((char*)cen + ((S * 6 * 4 + 255) & ~255LL));
    float* box = (float*)lt_scratch(ctx, SCR_MISC, 64, &st);
    if (!box) return st;
    const int blocks = (int)std::min<int64_t>((npad + 255) / 256, 16 * (int64_t)ctx->num_sms);
    k_bbox<<<1, 1024, 0, ctx->stream>>>((const float4*)pts, m, box);
    LT_LAUNCH_CHECK(ctx, "k_bbox");
    k_point_keys<<<blocks, 256, 0, ctx->stream>>>((const float4*)pts, m, box, npad, keys);
    LT_LAUNCH_CHECK(ctx, "k_point_keys");
    if ((st = bitonic_sort(ctx, keys, npad)) != LT_OK) return st;
    k_kmeans_seed<<<(S + 255) / 256, 256, 0, ctx->stream>>>((const float4*)pts, m, keys, S, normal_weight, cen);
    LT_LAUNCH_CHECK(ctx, "k_kmeans_seed");
    const size_t shm = (size_t)S * 6 * 4;
    if (shm > 16 * 1024)
        LT_CUDA(ctx, cudaFuncSetAttribute(k_kmeans_assign, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    const int ablocks = (int)std::min<int64_t>((m + 255) / 256, 4 * (int64_t)ctx->num_sms);
    for (int it = 0; it < iters; ++it) {
        LT_CUDA(ctx, cudaMemsetAsync(sums, 0, (size_t)S * 7 * 8, ctx->stream));
        k_kmeans_assign<<<ablocks, 256, shm, ctx->stream>>>((const float4*)pts, m, S, normal_weight, cen, lab, sums);
        LT_LAUNCH_CHECK(ctx, "k_kmeans_assign");
        k_kmeans_update<<<(S + 255) / 256, 256, 0, ctx->stream>>>(S, sums, cen);
        LT_LAUNCH_CHECK(ctx, "k_kmeans_update");
    }
    k_kmeans_assign<<<ablocks, 256, shm, ctx->stream>>>((const float4*)pts, m, S, normal_weight, cen, lab, nullptr);
    LT_LAUNCH_CHECK(ctx, "k_kmeans_assign");
    LT_CUDA(ctx, cudaMemsetAsync(counts, 0, (size_t)S * 4, ctx->stream));
    k_label_keys<<<blocks, 256, 0, ctx->stream>>>(lab, m, npad, keys, counts);
    LT_LAUNCH_CHECK(ctx, "k_label_keys");
    if ((st = bitonic_sort(ctx, keys, npad)) != LT_OK) return st;
    k_perm_from_keys<<<blocks, 256, 0, ctx->stream>>>(keys, m, row_perm);
    LT_LAUNCH_CHECK(ctx, "k_perm_from_keys");
    k_slice_off<<<1, 1024, 0, ctx->stream>>>(counts, S, slice_off);
    LT_LAUNCH_CHECK(ctx, "k_slice_off");
    LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return LT_OK;
}

extern "C" lt_status lt_mesh_upload(lt_ctx* ctx, const float* tris, int64_t nt) {
    if (!ctx || nt < 0 || (nt > 0 && !tris) || nt > (1 << 26))
        return lt_fail(ctx, LT_EINVAL, "lt_mesh_upload: bad arguments");
    if (ctx->graphs > 0)
        return lt_fail(ctx, LT_EINVAL, "lt_mesh_upload: live frame graphs reference the current scene");
    if (!ctx->d_cell_off) return lt_fail(ctx, LT_EINVAL, "lt_mesh_upload: upload the boxes first");
    cudaSetDevice(ctx->device);
    LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    cudaFree(ctx->d_mesh);
    ctx->d_mesh = nullptr;
    Grid& g = ctx->grid;
    g.nt = 0;
    g.tri = nullptr;
    g.bvh_aabb = nullptr;
    g.bvh_child = nullptr;
    g.bvh_tri = nullptr;
    g.bvh_node = nullptr;
    g.bvh_leaf = nullptr;
    if (nt == 0) return LT_OK;
    const int64_t nn = 2 * nt - 1;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t b_rec = up((size_t)nt * 48), b_aabb = up((size_t)nn * 24), b_child = up((size_t)nn * 8),
                 b_par = up((size_t)nn * 4), b_range = up((size_t)nn * 8), b_leaf = up((size_t)nt * 4), b_node = up((size_t)nt * 64);
    char* m = nullptr;
    LT_CUDA(ctx, cudaMalloc(&m, 2 * b_rec + b_aabb + b_child + b_par + b_range + b_leaf + b_node));
    ctx->d_mesh = m;
    float4* rec = (float4*)m;
    float* aabb = (float*)(m + b_rec);
    int32_t* child = (int32_t*)(m + b_rec + b_aabb);
    int32_t* parent = (int32_t*)(m + b_rec + b_aabb + b_child);
    int32_t* range = (int32_t*)(m + b_rec + b_aabb + b_child + b_par);
    int32_t* leaf = (int32_t*)(m + b_rec + b_aabb + b_child + b_par + b_range);
    float4* node_rec = (float4*)(m + b_rec + b_aabb + b_child + b_par + b_range + b_leaf);
    float4* leaf_rec = (float4*)(m + b_rec + b_aabb + b_child + b_par + b_range + b_leaf + b_node);
    const int64_t npad = next_pow2(nt);
    lt_status st;
    char* p = (char*)lt_scratch(ctx, SCR_SORT, (size_t)npad * 8 + (size_t)nt * 4 + (size_t)nt * 16 + 1024, &st);
    if (!p) return st;
    unsigned long long* keys = (unsigned long long*)p;
    int32_t* flags = (int32_t*)(p + npad * 8);
    float4* cen = (float4*)(p + up(npad * 8 + (size_t)nt * 4));
    float* box = (float*)lt_scratch(ctx, SCR_MISC, 64, &st);
    if (!box) return st;
    const int blocks = (int)std::min<int64_t>((npad + 255) / 256, 16 * (int64_t)ctx->num_sms);
    k_tri_prep<<<blocks, 256, 0, ctx->stream>>>(tris, nt, cen, rec);
    LT_LAUNCH_CHECK(ctx, "k_tri_prep");
    k_bbox<<<1, 1024, 0, ctx->stream>>>(cen, nt, box);
    LT_LAUNCH_CHECK(ctx, "k_bbox");
    k_tri_keys<<<blocks, 256, 0, ctx->stream>>>(cen, nt, box, npad, keys);
    LT_LAUNCH_CHECK(ctx, "k_tri_keys");
    if ((st = bitonic_sort(ctx, keys, npad)) != LT_OK) return st;
    lt_tree view{};
    view.n = nt;
    view.child = child;
    view.parent = parent;
    view.range = range;
    k_karras<<<blocks, 256, 0, ctx->stream>>>(keys, nt, view);
    LT_LAUNCH_CHECK(ctx, "k_karras");
    k_bvh_leaves<<<blocks, 256, 0, ctx->stream>>>(keys, tris, nt, leaf, aabb, parent, flags);
    LT_LAUNCH_CHECK(ctx, "k_bvh_leaves");
    if (nt > 1) {
        LT_CUDA(ctx, cudaMemsetAsync(parent, 0xff, sizeof(int32_t), ctx->stream));  // the root
        k_bvh_up<<<blocks, 256, 0, ctx->stream>>>(nt, child, parent, aabb, flags);
        LT_LAUNCH_CHECK(ctx, "k_bvh_up");
    }
    k_bvh_pack<<<blocks, 256, 0, ctx->stream>>>(nt, child, aabb, leaf, rec, node_rec, leaf_rec);
    LT_LAUNCH_CHECK(ctx, "k_bvh_pack");
    LT_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    g.nt = (int)nt;
    g.tri = rec;
    g.bvh_aabb = aabb;
    g.bvh_child = child;
    g.bvh_tri = leaf;
    g.bvh_node = node_rec;
    g.bvh_leaf = leaf_rec;
    return LT_OK;
}

extern "C" lt_status lt_mesh_bvh(const lt_ctx* ctx, float* aabb, int32_t* child, int32_t* leaf_tri) {
    if (!ctx || ctx->grid.nt < 1 || !aabb || !child || !leaf_tri) return LT_EINVAL;
    cudaSetDevice(ctx->device);
    const Grid& g = ctx->grid;
    const int64_t nt = g.nt, nn = 2 * nt - 1;
    if (cudaMemcpy(aabb, g.bvh_aabb, (size_t)nn * 24, cudaMemcpyDeviceToDevice) != cudaSuccess ||
        cudaMemcpy(child, g.bvh_child, (size_t)(nt - 1) * 8, cudaMemcpyDeviceToDevice) != cudaSuccess ||
        cudaMemcpy(leaf_tri, g.bvh_tri, (size_t)nt * 4, cudaMemcpyDeviceToDevice) != cudaSuccess)
        return LT_ECUDA;
    return LT_OK;
}
