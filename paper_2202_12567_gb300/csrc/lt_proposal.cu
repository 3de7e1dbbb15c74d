// Learned pass-2 proposal: per-(slice, column) features after pass 1, a bfloat16
// MLP (32 -> 64 -> 64 -> 64 -> 1, SiLU) on the tensor cores (mma.sync m16n8k16,
// float32 accumulate), the slice softmax mixed with the pass-1 estimate g (Sec. 5)
// into pass-2 weights, and the training side: full slice matrices, leverage targets
// by subspace iteration, forward + backward + Adam.  The paper names a learned
// importance only as future work; every choice here is ours (layout of the features
// and of the parameters in include/lt.h).
#include <cuda_bf16.h>
#include <math.h>
#include <stddef.h>

#include <algorithm>

#include "lt_internal.cuh"

using namespace ltk;

namespace {

constexpr int NF = LT_MLP_FEATURES, NH = LT_MLP_HIDDEN, NPAR = LT_MLP_PARAMS;
constexpr int OW1 = 0, OB1 = OW1 + NH * NF, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH,
              OB3 = OW3 + NH * NH, OW4 = OB3 + NH, OB4 = OW4 + NH;
static_assert(OB4 + 1 == NPAR, "parameter layout");
constexpr uint32_t kTagLeverage = 4, kTagInit = 5;
constexpr int TM = 64;            // rows per tile
// 16 warps per CTA: warp w takes the 16 rows (or outputs) 16 (w & 3) .. and a quarter of
// the columns of every product of a tile.  The elementwise work and the parameter loads
// of a tile, which are most of its time, spread over four times the threads of one warp
// per 16 rows.  What bounds it: latency between the barriers of a tile (4 or 5 tiles a
// CTA).  A training step on 40 K rows (forward, softmax, backward, reduction, Adam):
// 0.118 ms, 0.223 ms with 4 warps, transposed copies of every operand and the loads of
// the reductions one at a time.
constexpr int MT = 512;
constexpr int L1 = NF + 8;        // bf16 row stride of 32-wide operands (conflict-free fragments)
constexpr int L2 = NH + 8;        // of 64-wide operands

typedef __nv_bfloat16 bf16;

// acc + v(e) for e = e0, e0 + step, ... < n, in that order, B loads in flight at a time
template <int B, class V>
__device__ __forceinline__ float sum_in_order(int e0, int n, int step, float acc, V v) {
    for (int e = e0; e < n; e += B * step) {
        float x[B];
#pragma unroll
        for (int u = 0; u < B; ++u) x[u] = v(min(e + u * step, n - 1));
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (e + u * step < n) acc += x[u];
    }
    return acc;
}

__device__ __forceinline__ float silu(float h) { return h / (1.f + expf(-h)); }
__device__ __forceinline__ float dsilu(float h) {
    const float s = 1.f / (1.f + expf(-h));
    return s * (1.f + h * (1.f - s));
}
__device__ __forceinline__ float rbf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t ld2(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

// One warp: C[16][8 NT] += A[16][K] B^T with A row-major (stride lda) and Bt = B^T
// row-major [8 NT][K] (stride ldb), K a multiple of 16.  Fragment layout of
// m16n8k16: g = lane / 4, t = lane % 4; A regs (g, 2t) (g+8, 2t) (g, 2t+8)
// (g+8, 2t+8); B regs (k 2t, n g) (k 2t+8, n g); C (g, 2t) (g, 2t+1) (g+8, 2t) (g+8, 2t+1).
template <int NT>
__device__ __forceinline__ void warp_gemm(const bf16* A, int lda, const bf16* Bt, int ldb, int K, float (&c)[NT][4]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    for (int k0 = 0; k0 < K; k0 += 16) {
        const uint32_t a0 = ld2(A + g * lda + k0 + 2 * t), a1 = ld2(A + (g + 8) * lda + k0 + 2 * t);
        const uint32_t a2 = ld2(A + g * lda + k0 + 8 + 2 * t), a3 = ld2(A + (g + 8) * lda + k0 + 8 + 2 * t);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const bf16* b = Bt + (8 * nt + g) * ldb + k0 + 2 * t;
            mma_bf16(c[nt], a0, a1, a2, a3, ld2(b), ld2(b + 8));
        }
    }
}

// 8x8 matrices of 16-bit values, transposed on the way in: lane 8 q + i gives row i of
// matrix q, and register q of lane (g, t) is element (2t, 2t + 1; g) of it
__device__ __forceinline__ void ldm4_trans(uint32_t (&r)[4], const bf16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldm2_trans(uint32_t (&r)[2], const bf16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}

// One warp: C[16][8 NT] += A B with B [K][8 NT] row-major (stride ldb) and A [16][K]
// row-major (AT false) or given as its transpose [K][16] (AT true).
template <int NT, bool AT>
__device__ __forceinline__ void warp_gemm_kn(const bf16* A, int lda, const bf16* B, int ldb, int K, float (&c)[NT][4]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    for (int k0 = 0; k0 < K; k0 += 16) {
        uint32_t a[4];
        if (AT) {  // matrices (k 0-7, m 0-7) (k 0-7, m 8-15) (k 8-15, m 0-7) (k 8-15, m 8-15)
            ldm4_trans(a, A + (k0 + (lane & 7) + (lane >= 16 ? 8 : 0)) * lda + ((lane & 8) ? 8 : 0));
        } else {
            a[0] = ld2(A + g * lda + k0 + 2 * t);
            a[1] = ld2(A + (g + 8) * lda + k0 + 2 * t);
            a[2] = ld2(A + g * lda + k0 + 8 + 2 * t);
            a[3] = ld2(A + (g + 8) * lda + k0 + 8 + 2 * t);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            uint32_t b[2];
            ldm2_trans(b, B + (k0 + (lane & 15)) * ldb + 8 * nt);
            mma_bf16(c[nt], a[0], a[1], a[2], a[3], b[0], b[1]);
        }
    }
}

template <int NT>
__device__ __forceinline__ void zero(float (&c)[NT][4]) {
#pragma unroll
    for (int i = 0; i < NT; ++i) c[i][0] = c[i][1] = c[i][2] = c[i][3] = 0.f;
}

// ---------------------------------------------------------------- parameters
struct MlpSmem {
    // every bf16 array starts on 16 bytes and has rows of a multiple of 16 bytes (ldmatrix)
    alignas(16) bf16 X[TM * L1];  // input tile, rows x 32
    alignas(16) bf16 W1[NH * L1];     // [out][in]
    alignas(16) bf16 W2[NH * L2];
    alignas(16) bf16 W3[NH * L2];
    alignas(16) bf16 A1[TM * L2];     // activations, rows x 64
    alignas(16) bf16 A2[TM * L2];
    alignas(16) bf16 A3[TM * L2];
    float b1[NH], b2[NH], b3[NH], w4[NH], b4;
    float z[TM];
};

__device__ void load_params(const float* __restrict__ th, MlpSmem& s) {
    for (int i = threadIdx.x; i < NH * NF; i += blockDim.x) s.W1[(i / NF) * L1 + i % NF] = __float2bfloat16_rn(th[OW1 + i]);
    for (int i = threadIdx.x; i < NH * NH; i += blockDim.x) {
        s.W2[(i / NH) * L2 + i % NH] = __float2bfloat16_rn(th[OW2 + i]);
        s.W3[(i / NH) * L2 + i % NH] = __float2bfloat16_rn(th[OW3 + i]);
    }
    for (int i = threadIdx.x; i < NH; i += blockDim.x) {
        s.b1[i] = th[OB1 + i];
        s.b2[i] = th[OB2 + i];
        s.b3[i] = th[OB3 + i];
        s.w4[i] = rbf(th[OW4 + i]);
    }
    if (threadIdx.x == 0) s.b4 = th[OB4];
}

// rows [r0, r0 + TM) of feat into s.X (rows >= n are zero)
__device__ void load_tile(const float* __restrict__ feat, int64_t r0, int64_t n, MlpSmem& s) {
    for (int i = threadIdx.x; i < TM * NF; i += blockDim.x) {
        const int row = i / NF, c = i % NF;
        const float v = r0 + row < n ? feat[(r0 + row) * NF + c] : 0.f;
        s.X[row * L1 + c] = __float2bfloat16_rn(v);
    }
}

// one hidden layer for the warp's 16 rows and 16 columns: H = A W^T + b, out =
// bf16(silu(H)); the pre-activations go to Hs (float [TM][NH]) when it is given
template <int K>
__device__ __forceinline__ void layer(const bf16* Ain, int lda, const bf16* W, int ldw, const float* b, bf16* Aout,
                                      float* Hs) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, w = threadIdx.x >> 5, wr = w & 3, wc = w >> 2;
    float c[2][4];
    zero(c);
    warp_gemm<2>(Ain + 16 * wr * lda, lda, W + 16 * wc * ldw, ldw, K, c);
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int row = 16 * wr + g + (q >= 2 ? 8 : 0), col = 16 * wc + 8 * nt + 2 * t + (q & 1);
            const float h = c[nt][q] + b[col];
            if (Hs) Hs[row * NH + col] = h;
            Aout[row * L2 + col] = __float2bfloat16_rn(silu(h));
        }
}

// forward of the tile in s.X: logits into s.z; ends with a CTA barrier
__device__ void forward_tile(MlpSmem& s, float* H1, float* H2, float* H3) {
    layer<NF>(s.X, L1, s.W1, L1, s.b1, s.A1, H1);
    __syncthreads();
    layer<NH>(s.A1, L2, s.W2, L2, s.b2, s.A2, H2);
    __syncthreads();
    layer<NH>(s.A2, L2, s.W3, L2, s.b3, s.A3, H3);
    __syncthreads();
    if (threadIdx.x < TM) {
        const int row = threadIdx.x;
        float z = s.b4;
#pragma unroll 8
        for (int j = 0; j < NH; j += 2) {
            const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(s.A3 + row * L2 + j);
            z = fmaf(__bfloat162float(a.x), s.w4[j], z);
            z = fmaf(__bfloat162float(a.y), s.w4[j + 1], z);
        }
        s.z[row] = z;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(MT) k_mlp_forward(const float* __restrict__ theta, const float* __restrict__ feat,
                                                     int64_t n_max, const int32_t* __restrict__ n_dev,
                                                     float* __restrict__ z) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MlpSmem& s = *reinterpret_cast<MlpSmem*>(smem_raw);
    const int64_t n = n_dev ? min((int64_t)*n_dev, n_max) : n_max;
    load_params(theta, s);
    for (int64_t r0 = (int64_t)blockIdx.x * TM; r0 < n; r0 += (int64_t)gridDim.x * TM) {
        __syncthreads();
        load_tile(feat, r0, n, s);
        __syncthreads();
        forward_tile(s, nullptr, nullptr, nullptr);
        for (int i = threadIdx.x; i < TM; i += blockDim.x)
            if (r0 + i < n) z[r0 + i] = s.z[i];
    }
}

// ---------------------------------------------------------------- training
struct BwdSmem {
    MlpSmem f;
    alignas(16) bf16 D[TM * L2];  // dH of the current layer, [rows][out]
    float H1[TM * NH], H2[TM * NH], H3[TM * NH];  // pre-activations, then dH in float
    float dz[TM];
    float grad[NPAR];      // this CTA's gradient, accumulated over its tiles
};

static_assert(offsetof(BwdSmem, D) % 16 == 0 && offsetof(MlpSmem, A1) % 16 == 0 && offsetof(MlpSmem, A2) % 16 == 0 &&
                  offsetof(MlpSmem, W2) % 16 == 0 && offsetof(MlpSmem, W3) % 16 == 0 && L1 % 8 == 0 && L2 % 8 == 0,
              "ldmatrix reads 16-byte rows");

// dW[out][in] += D^T X for the tile (both [rows][..]): warp w owns outputs 16 (w & 3) ..
// and NT x 8 inputs
template <int NT>
__device__ void weight_grad(const bf16* D, const bf16* X, int ldx, int K_in, float* gW) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, w = threadIdx.x >> 5, wr = w & 3, wc = w >> 2;
    float c[NT][4];
    zero(c);
    warp_gemm_kn<NT, true>(D + 16 * wr, L2, X + 8 * NT * wc, ldx, TM, c);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int o = 16 * wr + g + (q >= 2 ? 8 : 0), i = 8 * (NT * wc + nt) + 2 * t + (q & 1);
            gW[o * K_in + i] += c[nt][q];
        }
}

// the bias gradient of a layer: column sums of dH over the rows in order
__device__ void bias_grad(const float* Hf, float* gb) {
    if (threadIdx.x < NH) {
        float a = 0.f;
#pragma unroll 8
        for (int r = 0; r < TM; ++r) a += Hf[r * NH + threadIdx.x];
        gb[threadIdx.x] += a;
    }
}

// Hf [rows][NH] float holds dA of the layer on entry; turns it into dH = dA silu'(H)
// (H the pre-activations in Hpre) and fills D (bf16)
__device__ void act_grad(float* Hf, const float* Hpre, BwdSmem& s, int nrows) {
    for (int i = threadIdx.x; i < TM * NH; i += MT) {
        const int r = i / NH, c = i % NH;
        const float d = r < nrows ? Hf[i] * dsilu(Hpre[i]) : 0.f;
        Hf[i] = d;
        s.D[r * L2 + c] = __float2bfloat16_rn(d);
    }
}

// dA_prev[rows][in] = D[rows][out] W[out][in] into Hf
__device__ void input_grad(const BwdSmem& s, const bf16* W, float* Hf) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, w = threadIdx.x >> 5, wr = w & 3, wc = w >> 2;
    float c[2][4];
    zero(c);
    warp_gemm_kn<2, false>(s.D + 16 * wr * L2, L2, W + 16 * wc, L2, NH, c);
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int row = 16 * wr + g + (q >= 2 ? 8 : 0), col = 16 * wc + 8 * nt + 2 * t + (q & 1);
            Hf[row * NH + col] = c[nt][q];
        }
}

// Gradient of loss = sum_rows dz * z over rows [0, n); per CTA into part[blockIdx][NPAR].
__global__ void __launch_bounds__(MT, 1) k_mlp_backward(const float* __restrict__ theta, const float* __restrict__ feat,
                                                     const float* __restrict__ dz, int64_t n,
                                                     float* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BwdSmem& s = *reinterpret_cast<BwdSmem*>(smem_raw);
    load_params(theta, s.f);
    for (int i = threadIdx.x; i < NPAR; i += MT) s.grad[i] = 0.f;
    for (int64_t r0 = (int64_t)blockIdx.x * TM; r0 < n; r0 += (int64_t)gridDim.x * TM) {
        const int nrows = (int)min((int64_t)TM, n - r0);
        __syncthreads();
        load_tile(feat, r0, n, s.f);
        for (int i = threadIdx.x; i < TM; i += MT) s.dz[i] = i < nrows ? dz[r0 + i] : 0.f;
        __syncthreads();
        forward_tile(s.f, s.H1, s.H2, s.H3);
        // output layer: z = w4 . a3 + b4 (the last warps, beside the first ones' dH3)
        if (threadIdx.x >= MT - NH) {
            const int j = threadIdx.x - (MT - NH);
            float a = 0.f;
#pragma unroll 8
            for (int r = 0; r < TM; ++r) a += s.dz[r] * __bfloat162float(s.f.A3[r * L2 + j]);
            s.grad[OW4 + j] += a;
        } else if (threadIdx.x == MT - NH - 1) {
            float a = 0.f;
#pragma unroll 8
            for (int r = 0; r < TM; ++r) a += s.dz[r];
            s.grad[OB4] += a;
        }
        // dH3 = dz w4 silu'(H3), in place of the pre-activations
        for (int i = threadIdx.x; i < TM * NH; i += MT) {
            const int r = i / NH, c = i % NH;
            const float d = r < nrows ? s.dz[r] * s.f.w4[c] * dsilu(s.H3[i]) : 0.f;
            s.H3[i] = d;
            s.D[r * L2 + c] = __float2bfloat16_rn(d);
        }
        __syncthreads();
        weight_grad<2>(s.D, s.f.A2, L2, NH, s.grad + OW3);
        bias_grad(s.H3, s.grad + OB3);
        __syncthreads();
        // layer 2
        input_grad(s, s.f.W3, s.H3);  // dA2 into H3's storage
        __syncthreads();
        act_grad(s.H3, s.H2, s, nrows);
        __syncthreads();
        weight_grad<2>(s.D, s.f.A1, L2, NH, s.grad + OW2);
        bias_grad(s.H3, s.grad + OB2);
        __syncthreads();
        // layer 1
        input_grad(s, s.f.W2, s.H3);  // dA1
        __syncthreads();
        act_grad(s.H3, s.H1, s, nrows);
        __syncthreads();
        weight_grad<1>(s.D, s.f.X, L1, NF, s.grad + OW1);
        bias_grad(s.H3, s.grad + OB1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NPAR; i += MT) part[(int64_t)blockIdx.x * NPAR + i] = s.grad[i];
}

// softmax over each group's rows, dz = (softmax - target) / G, loss per group.  A warp per
// group; lane l has the rows a + l, a + l + 32, ..., the first kKeep of them in registers, so that the
// three passes over the group read memory once.  A step of the training on 40 K rows in 64
// groups: 115.4 to 110.6 us, with the loads of the gradient's parts in flight together.
__global__ void k_group_softmax(const float* __restrict__ z, const float* __restrict__ target,
                                const int32_t* __restrict__ goff, int G, float* __restrict__ dz,
                                float* __restrict__ gloss) {
    constexpr int kKeep = 24;
    const int lane = threadIdx.x & 31;
    for (int gi = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); gi < G; gi += gridDim.x * (blockDim.x >> 5)) {
        const int a = goff[gi] + lane, b = goff[gi + 1];
        float x[kKeep], y[kKeep];
#pragma unroll
        for (int u = 0; u < kKeep; ++u) {
            x[u] = a + 32 * u < b ? z[a + 32 * u] : -3.0e38f;
            y[u] = a + 32 * u < b ? target[a + 32 * u] : 0.f;
        }
        float mx = -3.0e38f;
#pragma unroll
        for (int u = 0; u < kKeep; ++u) mx = fmaxf(mx, x[u]);
        for (int i = a + 32 * kKeep; i < b; i += 32) mx = fmaxf(mx, z[i]);
        mx = warp_max(mx);
        float se = 0.f;
#pragma unroll
        for (int u = 0; u < kKeep; ++u)
            if (a + 32 * u < b) se += expf(x[u] - mx);
        for (int i = a + 32 * kKeep; i < b; i += 32) se += expf(z[i] - mx);
        se = warp_sum(se);
        const float lse = logf(se);
        float l = 0.f;
        auto row = [&](int i, float zi, float ti) {
            const float lp = zi - mx - lse;
            dz[i] = (expf(lp) - ti) / (float)G;
            l -= ti * lp;
        };
#pragma unroll
        for (int u = 0; u < kKeep; ++u)
            if (a + 32 * u < b) row(a + 32 * u, x[u], y[u]);
        for (int i = a + 32 * kKeep; i < b; i += 32) row(i, z[i], target[i]);
        l = warp_sum(l);
        if (lane == 0) gloss[gi] = l;
    }
}

// grad[p] = sum over the CTA partials in order; loss = sum of the group losses / G
__global__ void k_grad_reduce(const float* __restrict__ part, int nparts, float* __restrict__ grad,
                              const float* __restrict__ gloss, int G, float* __restrict__ loss) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < NPAR; p += gridDim.x * blockDim.x) {
        grad[p] = sum_in_order<32>(0, nparts, 1, 0.f, [&](int q) { return __ldg(part + (int64_t)q * NPAR + p); });
    }
    if (loss && blockIdx.x == 0 && threadIdx.x == 0) {
        *loss = sum_in_order<32>(0, G, 1, 0.f, [&](int g) { return __ldg(gloss + g); }) / (float)G;
    }
}

__global__ void k_adam(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ grad, int step, float lr) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < NPAR; p += gridDim.x * blockDim.x) {
        const float g = grad[p];
        const float mm = b1 * m[p] + (1.f - b1) * g;
        const float vv = b2 * v[p] + (1.f - b2) * g * g;
        m[p] = mm;
        v[p] = vv;
        theta[p] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    }
}

__global__ void k_mlp_init(uint64_t seed, float* __restrict__ theta) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < NPAR; p += gridDim.x * blockDim.x) {
        float v = 0.f;
        const bool w = p < OB1 || (p >= OW2 && p < OB2) || (p >= OW3 && p < OB3) || (p >= OW4 && p < OB4);
        if (w) {
            const float fan = p < OB1 ? (float)NF : (float)NH;
            const float u = (float)((double)philox((uint32_t)p, 0u, 0u, kTagInit, seed).x * 2.3283064365386963e-10 - 0.5);
            v = 2.f * u / sqrtf(fan);
        }
        theta[p] = v;
    }
}

// ---------------------------------------------------------------- features
// per slice: mean position and normal, AABB, mean pass-1 value, m', n'
constexpr int kSliceStats = 16;

__global__ void k_feat_slice(lt_frame F, lt_samples smp, float* __restrict__ st) {
    __shared__ float red[16][32];
    const int s = blockIdx.x;
    const int row0 = F.slice_off[s], ms = F.slice_off[s + 1] - row0;
    const float4* P0 = reinterpret_cast<const float4*>(F.pts);
    const float4* P1 = P0 + F.m;
    float acc[13];
#pragma unroll
    for (int k = 0; k < 13; ++k) acc[k] = k < 6 || k == 12 ? 0.f : k < 9 ? 3.0e38f : -3.0e38f;
#pragma unroll 4
    for (int i = threadIdx.x; i < ms; i += blockDim.x) {
        const float4 p = P0[row0 + i], nn = P1[row0 + i];
        acc[0] += p.x;
        acc[1] += p.y;
        acc[2] += p.z;
        acc[3] += nn.x;
        acc[4] += nn.y;
        acc[5] += nn.z;
        acc[6] = fminf(acc[6], p.x);
        acc[7] = fminf(acc[7], p.y);
        acc[8] = fminf(acc[8], p.z);
        acc[9] = fmaxf(acc[9], p.x);
        acc[10] = fmaxf(acc[10], p.y);
        acc[11] = fmaxf(acc[11], p.z);
    }
    const int n1 = smp.n1[s];
    const float* val = smp.val + smp.off[s];
    acc[12] = sum_in_order<16>(threadIdx.x, n1, blockDim.x, acc[12], [&](int e) { return __ldg(val + e); });
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < 13; ++k) {  // (unrolled: acc must not live in local memory)
        float v = acc[k];
        v = (k >= 6 && k < 9) ? warp_min(v) : (k >= 9 && k < 12) ? warp_max(v) : warp_sum(v);
        if (lane == 0) red[k][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < 13) {
        const int k = threadIdx.x;
        float v = red[k][0];
        for (int q = 1; q < nw; ++q) v = (k >= 6 && k < 9) ? fminf(v, red[k][q]) : (k >= 9 && k < 12) ? fmaxf(v, red[k][q]) : v + red[k][q];
        float* o = st + (int64_t)s * kSliceStats;
        if (k < 6) o[k] = ms > 0 ? v / (float)ms : 0.f;
        else if (k < 12) o[k] = ms > 0 ? v : 0.f;
        else {
            const float mu = n1 > 0 ? v / (float)n1 : 0.f;
            o[12] = mu > 0.f ? mu : 1.f;
            o[13] = logf((float)max(ms, 1)) / 10.f;
            o[14] = logf((float)max(smp.ncol[s], 1)) / 10.f;
        }
    }
}

__global__ void k_group_prefix(const int32_t* __restrict__ ncol, int S, int32_t* __restrict__ goff) {
    __shared__ int32_t ws[32];
    int carry = 0;
    for (int c0 = 0; c0 < S; c0 += blockDim.x) {
        const int s = c0 + threadIdx.x;
        const int x = s < S ? ncol[s] : 0;
        int tot;
        const int pre = block_exclusive_scan<int>(x, ws, &tot);
        if (s < S) goff[s] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) goff[S] = carry;
}

// first pass-1 entry of the slice (keys grouped by column, ascending) whose column >= j
// by one warp: 32 probes a step (a binary search is a chain of 15 loads)
__device__ __forceinline__ int first_col_at_least(const uint32_t* key, int n1, int j) {
    const int lane = threadIdx.x & 31;
    int a = 0, b = n1;  // the answer is in [a, b]
    while (a < b) {
        const int step = (b - a + 31) / 32, p = a + step * (lane + 1) - 1;
        const int c = __popc(__ballot_sync(0xffffffffu, p < b && (int)(key[p] & 0xffffu) < j));
        a += c * step;  // the probes below are a prefix
        b = min(b, a + step - 1);
        if (a > b) a = b;
    }
    return a;
}

// one warp per (slice, column): the 32 features into feat[goff[s] + j]
__global__ void k_feat_cols(lt_frame F, lt_samples smp, const float* __restrict__ st,
                            const int32_t* __restrict__ goff, float* __restrict__ feat) {
    const int lane = threadIdx.x & 31;
    const int C = F.C;
    const float4* V0 = reinterpret_cast<const float4*>(F.vpls);
    const float4* V1 = V0 + F.n;
    const float iroot = F.tree.I[0];
    const int s = blockIdx.y;
    const int ns = smp.ncol[s];
    for (int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < ns; j += gridDim.x * (blockDim.x >> 5)) {
        const uint32_t* key = smp.key + smp.off[s];
        const float* val = smp.val + smp.off[s];
        const int n1 = smp.n1[s];
        const int lo = first_col_at_least(key, n1, j), hi = first_col_at_least(key, n1, j + 1);
        const int cnt = hi - lo;
        float sum = 0.f, mn = 3.0e38f, mx = -3.0e38f;
        for (int e = lo + lane; e < hi; e += 32) {
            const float v = val[e];
            sum += v;
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        }
        sum = warp_sum(sum);
        mn = warp_min(mn);
        mx = warp_max(mx);
        const float mean = cnt > 0 ? sum / (float)cnt : 0.f;
        float sq = 0.f;
        for (int e = lo + lane; e < hi; e += 32) {
            const float d = val[e] - mean;
            sq += d * d;
        }
        sq = warp_sum(sq);
        const float* ss = st + (int64_t)s * kSliceStats;
        const float mu = ss[12];
        const int node = smp.col_node[(int64_t)s * C + j];
        const int rep = F.tree.rep[node];
        float v = 0.f;
        if (lane < 12) v = ss[lane];
        else if (lane < 18) v = F.tree.aabb[(int64_t)node * 6 + (lane - 12)];
        else if (lane < 24) {
            const float4 p = lane < 21 ? V0[rep] : V1[rep];
            const int k = (lane - 18) % 3;
            v = k == 0 ? p.x : k == 1 ? p.y : p.z;
        } else if (lane == 24) v = logf(F.tree.I[node] / iroot);
        else if (lane == 25) v = mean / mu;
        else if (lane == 26) v = cnt > 0 ? sqrtf(sq / (float)cnt) / mu : 0.f;
        else if (lane == 27) v = log1pf((float)cnt);
        else if (lane == 28) v = cnt > 0 ? mn / mu : 0.f;
        else if (lane == 29) v = cnt > 0 ? mx / mu : 0.f;
        else if (lane == 30) v = ss[13];
        else v = ss[14];
        feat[((int64_t)goff[s] + j) * NF + lane] = v;
    }
}

// pass-2 weights w[s][j] = mix softmax_s(z)_j + (1 - mix) g_j / sum g (one warp per slice)
__global__ void k_mix_weights(lt_frame F, lt_samples smp, const int32_t* __restrict__ goff,
                              const float* __restrict__ z, float mix, float* __restrict__ w) {
    const int lane = threadIdx.x & 31;
    for (int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); s < F.S; s += gridDim.x * (blockDim.x >> 5)) {
        const int ns = smp.ncol[s];
        const float* zz = z + goff[s];
        const float* g = smp.g + (int64_t)s * F.C;
        float mx = -3.0e38f, gs = 0.f;
        for (int j = lane; j < ns; j += 32) {
            mx = fmaxf(mx, zz[j]);
            gs += fmaxf(g[j], 0.f);
        }
        mx = warp_max(mx);
        gs = warp_sum(gs);
        float se = 0.f;
        for (int j = lane; j < ns; j += 32) se += expf(zz[j] - mx);
        se = warp_sum(se);
        for (int j = lane; j < ns; j += 32) {
            const float pg = gs > 0.f ? fmaxf(g[j], 0.f) / gs : 1.f / (float)ns;
            w[(int64_t)s * F.C + j] = mix * (expf(zz[j] - mx) / se) + (1.f - mix) * pg;
        }
    }
}

// ---------------------------------------------------------------- targets
// M_s[i][c] = A(row0 + i, column c) for every slice, at M + moff[s]
__global__ void k_moff(lt_frame F, lt_samples smp, int64_t* __restrict__ moff) {
    __shared__ int64_t ws[32];
    int64_t carry = 0;
    for (int c0 = 0; c0 < F.S; c0 += blockDim.x) {
        const int s = c0 + threadIdx.x;
        const int64_t x = s < F.S ? (int64_t)(F.slice_off[s + 1] - F.slice_off[s]) * smp.ncol[s] : 0;
        int64_t tot;
        const int64_t pre = block_exclusive_scan<int64_t>(x, ws, &tot);
        if (s < F.S) moff[s] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) moff[F.S] = carry;
}

// A thread keeps one column (its VPL record and scale in registers) and walks a run of
// kMatRows rows, so that an entry costs one broadcast point record and its shadow ray.
// Bound by the instructions of the entry model.
constexpr int kMatRows = 32;

__global__ void __launch_bounds__(128) k_slice_matrix(lt_frame F, lt_samples smp, Grid g, float dmin2,
                                                      const int64_t* __restrict__ moff, int64_t cap,
                                                      float* __restrict__ M, int32_t* status) {
    const float4* pts = reinterpret_cast<const float4*>(F.pts);
    const float4* vpls = reinterpret_cast<const float4*>(F.vpls);
    if (moff[F.S] > cap) {
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) latch(status, LT_ELIMIT);
        return;
    }
    const int s = blockIdx.y;
    const int row0 = F.slice_off[s], ms = F.slice_off[s + 1] - row0, ns = smp.ncol[s];
    const int tc = (ns + 127) / 128, tiles = tc * ((ms + kMatRows - 1) / kMatRows);
    float* out = M + moff[s];
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int c = (t % tc) * 128 + threadIdx.x, i0 = (t / tc) * kMatRows, i1 = min(i0 + kMatRows, ms);
        if (c >= ns) continue;
        const int node = smp.col_node[(int64_t)s * F.C + c];
        const PointRec L = load_rec(vpls, F.n, F.tree.rep[node]);
        // I_c / I_rep(c), I = flux * albedo, rounded as in the sampling passes
        const float scale = __fdiv_rn(F.tree.I[node], __fmul_rn(L.c.w, L.a.w));
        for (int i = i0; i < i1; ++i) {
            const PointRec P = load_rec(pts, F.m, row0 + i);
            out[(int64_t)i * ns + c] = entry_value(P, L, scale, dmin2, g);
        }
    }
}

// G_s = M_s^T M_s (n' rows of gram_ld(n') floats, so that every row starts on 16 bytes) at
// G + goff2[s], goff2 the prefix of their sizes
__host__ __device__ __forceinline__ int gram_ld(int n) { return (n + 3) & ~3; }

constexpr int kGramTile = 128;
constexpr int kGramStep = 16;

// goff2 and the prefix of the tiles on or above the diagonal of every G_s.  A latched
// LT_ELIMIT may be that of the slice matrices (a total beyond the caller's capacity): M then
// holds less than the slices' rows and columns say, and goff2[S] tells the kernels that
// follow to read none of it.
__global__ void k_goff(lt_samples smp, int S, int64_t* __restrict__ goff2, int64_t* __restrict__ tpfx,
                       int64_t gcap, int32_t* status) {
    __shared__ int64_t ws[32];
    int64_t carry = 0, tcarry = 0;
    for (int c0 = 0; c0 < S; c0 += blockDim.x) {
        const int s = c0 + threadIdx.x;
        const int64_t n = s < S ? smp.ncol[s] : 0, t = (n + kGramTile - 1) / kGramTile;
        int64_t tot;
        int64_t pre = block_exclusive_scan<int64_t>(n * gram_ld((int)n), ws, &tot);
        if (s < S) goff2[s] = carry + pre;
        carry += tot;
        pre = block_exclusive_scan<int64_t>(t * (t + 1) / 2, ws, &tot);
        if (s < S) tpfx[s] = tcarry + pre;
        tcarry += tot;
    }
    if (threadIdx.x == 0) {
        goff2[S] = *status == LT_ELIMIT ? INT64_MAX : carry;
        if (carry > gcap) latch(status, LT_ELIMIT);
        tpfx[S] = tcarry;
    }
}

// G_s is symmetric: a persistent grid takes the 128 x 128 tiles on or above the diagonal
// and writes each twice.  A thread holds 8 x 8 outputs; the rows of M stream through
// shared memory 16 at a time, the next 16 loaded while these are added.  Every output
// is one chain of multiply-adds over the rows in order.  Bound by the FP32 pipe.  With
// this, k_slice_matrix and the split subspace iteration the training data of a scene of 65536
// points (64 slices of about 630 columns, 30 rounds at rank 16) take 4.6 ms, 54.1 ms with
// 32 x 32 tiles and one CTA per slice for the whole iteration.
__global__ void __launch_bounds__(256, 2) k_gram(lt_frame F, lt_samples smp, const float* __restrict__ M,
                                                 const int64_t* __restrict__ moff, const int64_t* __restrict__ goff2,
                                                 const int64_t* __restrict__ tpfx, int64_t gcap,
                                                 float* __restrict__ G) {
    __shared__ __align__(16) float A[kGramStep][kGramTile], B[kGramStep][kGramTile];
    if (goff2[F.S] > gcap) return;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int lc = threadIdx.x & 127, lr = threadIdx.x >> 7;  // the loads: column lc of rows lr, lr + 2, ...
    for (int64_t w = blockIdx.x; w < tpfx[F.S]; w += gridDim.x) {
        int lo = 0, hi = F.S;  // tpfx[lo] <= w < tpfx[lo + 1]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (tpfx[mid] <= w) lo = mid;
            else hi = mid;
        }
        const int s = lo;
        const int ms = F.slice_off[s + 1] - F.slice_off[s], ns = smp.ncol[s];
        int t = (int)(w - tpfx[s]), bi = 0;
        for (int left = (ns + kGramTile - 1) / kGramTile; t >= left; --left, ++bi) t -= left;
        const int ti = bi * kGramTile, tj = (bi + t) * kGramTile;
        const float* Ms = M + moff[s];
        float acc[8][8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
        float pa[8], pb[8];
        auto fetch = [&](int r0) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int r = r0 + lr + 2 * q;
                pa[q] = (r < ms && ti + lc < ns) ? __ldg(Ms + (int64_t)r * ns + ti + lc) : 0.f;
                pb[q] = (r < ms && tj + lc < ns) ? __ldg(Ms + (int64_t)r * ns + tj + lc) : 0.f;
            }
        };
        fetch(0);
        for (int r0 = 0; r0 < ms; r0 += kGramStep) {
            __syncthreads();  // the last step's rows have been read
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                A[lr + 2 * q][lc] = pa[q];
                B[lr + 2 * q][lc] = pb[q];
            }
            __syncthreads();
            if (r0 + kGramStep < ms) fetch(r0 + kGramStep);
#pragma unroll
            for (int k = 0; k < kGramStep; ++k) {
                float a[8], b[8];
                *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&A[k][4 * ty]);
                *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(&A[k][64 + 4 * ty]);
                *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&B[k][4 * tx]);
                *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(&B[k][64 + 4 * tx]);
#pragma unroll
                for (int u = 0; u < 8; ++u)
#pragma unroll
                    for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
            }
        }
        float* Gs = G + goff2[s];
        const int ld = gram_ld(ns);
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const int i = ti + (u >> 2) * 64 + 4 * ty + (u & 3), j = tj + (v >> 2) * 64 + 4 * tx + (v & 3);
                if (i < ns && j < ns) {
                    Gs[(int64_t)i * ld + j] = acc[u][v];
                    if (ti != tj) Gs[(int64_t)j * ld + i] = acc[u][v];
                }
            }
    }
}

// Subspace iteration per slice: Q (n' x r, float, in global scratch) from Philox,
// `iters` rounds of Q <- mgs(G Q), then p_c = (|Q_c|^2 + 1/n') / (r' + 1) with r' the
// columns kept.  The product runs on the whole chip (k_lev_mult), the Gram-Schmidt one
// CTA per slice (k_lev_mgs) with block reductions in a fixed order: one CTA per slice
// for both spent 46.8 ms on the workload named above, most of it on 120 dependent block
// reductions a round and on the product at 64 of 152 SMs.
constexpr int kLevThreads = 512;

__device__ float block_sum(float v, float* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    float t = 0.f;
    for (int q = 0; q < nw; ++q) t += red[q];
    return t;
}

// Modified Gram-Schmidt on the columns of Q in global memory (any n and r).
__device__ void mgs_cols(float* Q, int n, int r, float* red) {
    for (int k = 0; k < r; ++k) {
        for (int j = 0; j < k; ++j) {
            float d = 0.f;
            for (int i = threadIdx.x; i < n; i += blockDim.x) d += Q[(int64_t)i * r + j] * Q[(int64_t)i * r + k];
            d = block_sum(d, red);
            for (int i = threadIdx.x; i < n; i += blockDim.x) Q[(int64_t)i * r + k] -= d * Q[(int64_t)i * r + j];
            __syncthreads();
        }
        float q2 = 0.f;
        for (int i = threadIdx.x; i < n; i += blockDim.x) q2 += Q[(int64_t)i * r + k] * Q[(int64_t)i * r + k];
        q2 = block_sum(q2, red);
        const float inv = q2 > 0.f ? 1.f / sqrtf(q2) : 0.f;
        for (int i = threadIdx.x; i < n; i += blockDim.x) Q[(int64_t)i * r + k] *= inv;
        __syncthreads();
    }
}

// The same with every row in registers (thread t holds rows t + 512 p, p < NR; at most
// 16 columns).  Column j, once normalised, is taken out of all later columns at once:
// each of them meets the earlier ones in the same order and with the same sums as in
// mgs_cols, so the bits are the same, with 2 block reductions per column in place of
// one per pair of columns.  The sums of 16 values over a warp share their shuffles: a
// lane hands on half of its values at each of the first four steps of the butterfly.
template <int NR>
__device__ void mgs_regs(float* __restrict__ Q, int n, int r, float* red, float (*part)[16], float* dots) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool vec = r == 16 && ((uintptr_t)Q & 15) == 0;  // rows of 64 bytes
    float q[NR][16];
#pragma unroll
    for (int p = 0; p < NR; ++p) {
        const int i = threadIdx.x + kLevThreads * p;
        if (vec && i < n) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 t = *reinterpret_cast<const float4*>(Q + (int64_t)i * 16 + 4 * k);
                q[p][4 * k] = t.x;
                q[p][4 * k + 1] = t.y;
                q[p][4 * k + 2] = t.z;
                q[p][4 * k + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) q[p][k] = (i < n && k < r) ? Q[(int64_t)i * r + k] : 0.f;
        }
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        if (j < r) {  // uniform
            float q2 = 0.f;
#pragma unroll
            for (int p = 0; p < NR; ++p) q2 = fmaf(q[p][j], q[p][j], q2);
            q2 = warp_sum(q2);
            if (lane == 0) red[w] = q2;
            __syncthreads();  // (the next write of red is two barriers away)
            q2 = 0.f;
#pragma unroll
            for (int x = 0; x < kLevThreads / 32; ++x) q2 += red[x];
            const float inv = q2 > 0.f ? 1.f / sqrtf(q2) : 0.f;
#pragma unroll
            for (int p = 0; p < NR; ++p) q[p][j] *= inv;
            if (j + 1 < r) {
                float d[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    d[k] = 0.f;
                    if (k > j) {
#pragma unroll
                        for (int p = 0; p < NR; ++p) d[k] = fmaf(q[p][j], q[p][k], d[k]);
                    }
                }
#pragma unroll
                for (int o = 16, h = 8; o > 1; o >>= 1, h >>= 1) {
#pragma unroll
                    for (int k = 0; k < h; ++k) {
                        const bool up = lane & o;
                        const float send = up ? d[k] : d[k + h], keep = up ? d[k + h] : d[k];
                        d[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                }
                d[0] += __shfl_xor_sync(0xffffffffu, d[0], 1);
                if (!(lane & 1)) part[w][lane >> 1] = d[0];  // lane bits 4..1 name the value
                __syncthreads();
                if (threadIdx.x < 16) {
                    float t = 0.f;
#pragma unroll
                    for (int x = 0; x < kLevThreads / 32; ++x) t += part[x][threadIdx.x];
                    dots[threadIdx.x] = t;
                }
                __syncthreads();
#pragma unroll
                for (int k = j + 1; k < 16; ++k) {
                    const float dk = dots[k];
#pragma unroll
                    for (int p = 0; p < NR; ++p) q[p][k] = fmaf(-dk, q[p][j], q[p][k]);
                }
            }
        }
    }
#pragma unroll
    for (int p = 0; p < NR; ++p) {
        const int i = threadIdx.x + kLevThreads * p;
        if (vec && i < n) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                *reinterpret_cast<float4*>(Q + (int64_t)i * 16 + 4 * k) =
                    make_float4(q[p][4 * k], q[p][4 * k + 1], q[p][4 * k + 2], q[p][4 * k + 3]);
        } else {
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if (i < n && k < r) Q[(int64_t)i * r + k] = q[p][k];
        }
    }
    __syncthreads();
}

// Orthonormalises Q of every slice: from Philox first (start), else the product k_lev_mult
// left there; after the last round also the targets.
__global__ void __launch_bounds__(kLevThreads) k_lev_mgs(lt_samples smp, const int32_t* __restrict__ slice_id, int S,
                                                         int C, const int64_t* __restrict__ goff2, int64_t gcap, int r,
                                                         bool start, bool last, uint64_t seed, float* __restrict__ Qall,
                                                         float* __restrict__ Yall, const int32_t* __restrict__ goff,
                                                         float* __restrict__ target) {
    __shared__ float red[32];
    __shared__ float part[kLevThreads / 32][16];
    __shared__ float dots[16];
    if (goff2[S] > gcap) return;
    const int s = blockIdx.x;
    const int ns = smp.ncol[s];
    if (ns == 0) return;
    const int rr = min(r, ns);
    float* Q = Qall + (int64_t)s * C * r;
    float* Y = Yall + (int64_t)s * C * r;
    if (start) {
        for (int e = threadIdx.x; e < ns * rr; e += blockDim.x) {
            const int c = e / rr, k = e % rr;
            Q[e] = (float)((double)philox((uint32_t)k, (uint32_t)c, slice_key(slice_id, s), kTagLeverage, seed).x *
                               2.3283064365386963e-10 - 0.5);
        }
        __syncthreads();
    }
    const int nr = (ns + kLevThreads - 1) / kLevThreads;
    if (rr > 16 || nr > 4) mgs_cols(Q, ns, rr, red);
    else if (nr == 1) mgs_regs<1>(Q, ns, rr, red, part, dots);
    else if (nr == 2) mgs_regs<2>(Q, ns, rr, red, part, dots);
    else if (nr == 3) mgs_regs<3>(Q, ns, rr, red, part, dots);
    else mgs_regs<4>(Q, ns, rr, red, part, dots);
    if (!last) return;
    float tot = 0.f;
    for (int c = threadIdx.x; c < ns; c += blockDim.x) {
        float l = 0.f;
        for (int k = 0; k < rr; ++k) l += Q[(int64_t)c * rr + k] * Q[(int64_t)c * rr + k];
        Y[c] = l + 1.f / (float)ns;
        tot += Y[c];
    }
    tot = block_sum(tot, red);
    for (int c = threadIdx.x; c < ns; c += blockDim.x) target[goff[s] + c] = Y[c] / tot;
}

// Y = G Q of every slice, 128 rows of G and 16 columns of Q by a CTA, 4 x 4 outputs by a
// thread.  Row i of G is read as column i (G is symmetric to the bit): the CTA's 128 columns
// of 16 rows at a time go through a ring of kLevStages tiles in shared memory (cp.async, 16
// bytes), the rows of Q beside them.  Sums over j in order.  Bound by what shared memory
// returns (a 16-byte load of a warp takes four cycles, also where lanes share it): a row and
// 16 columns a thread read 17 cycles' worth per step, 4 x 4 outputs 8.  Training data of a
// scene of 65536 points: 6.37 ms with G loaded straight into registers, 5.14 ms from the
// ring with a row a thread, 4.60 ms with 4 x 4 outputs.
constexpr int kLevRows = 128, kLevTile = 16, kLevStages = 6;

struct LevStage {
    float g[kLevTile][kLevRows];
    float q[kLevTile][16];
};

__global__ void __launch_bounds__(kLevRows) k_lev_mult(lt_samples smp, int S, int C, const float* __restrict__ G,
                                                       const int64_t* __restrict__ goff2, int64_t gcap, int r,
                                                       const float* __restrict__ Qall, float* __restrict__ Yall) {
    extern __shared__ __align__(16) unsigned char lev_raw[];
    LevStage* ring = reinterpret_cast<LevStage*>(lev_raw);
    if (goff2[S] > gcap) return;
    const int s = blockIdx.y;
    const int ns = smp.ncol[s];
    const int rr = min(r, ns), ld = gram_ld(ns), blocks = (ns + kLevRows - 1) / kLevRows, parts = (rr + 15) / 16;
    const int steps = (ns + kLevTile - 1) / kLevTile;
    const float* Gs = G + goff2[s];
    const float* Q = Qall + (int64_t)s * C * r;
    float* Y = Yall + (int64_t)s * C * r;
    for (int b = blockIdx.x; b < blocks * parts; b += gridDim.x) {
        const int i0 = (b % blocks) * kLevRows, k0 = (b / blocks) * 16;
        // tile t: rows 16 t .. of G, columns i0 .. (zeros past the last row and past column ld)
        auto fill = [&](int t) {
            if (t < steps) {
                LevStage& st = ring[t % kLevStages];
                const int j0 = t * kLevTile;
#pragma unroll
                for (int e = threadIdx.x; e < kLevTile * (kLevRows / 4); e += kLevRows) {
                    const int j = e / (kLevRows / 4), c = 4 * (e % (kLevRows / 4));
                    const bool live = j0 + j < ns && i0 + c < ld;
                    const float* p = live ? Gs + (int64_t)(j0 + j) * ld + i0 + c : Gs;
                    const unsigned d = (unsigned)__cvta_generic_to_shared(&st.g[j][c]);
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(p), "r"(live ? 16 : 0)
                                 : "memory");
                }
#pragma unroll
                for (int e = threadIdx.x; e < kLevTile * 16; e += kLevRows) {
                    const int j = e >> 4, k = e & 15;
                    const bool live = j0 + j < ns && k0 + k < rr;
                    const float* p = live ? Q + (int64_t)(j0 + j) * rr + k0 + k : Q;
                    const unsigned d = (unsigned)__cvta_generic_to_shared(&st.q[j][k]);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(p), "r"(live ? 4 : 0)
                                 : "memory");
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // rows 4 rq .. and columns 4 kq .. of the CTA's 128 x 16
        const int rq = threadIdx.x >> 2, kq = threadIdx.x & 3;
        float a[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int k = 0; k < 4; ++k) a[u][k] = 0.f;
#pragma unroll 1
        for (int t = 0; t < kLevStages - 1; ++t) fill(t);
        for (int t = 0; t < steps; ++t) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kLevStages - 2) : "memory");
            __syncthreads();  // tile t is here for every thread, tile t - 1 has been read
            fill(t + kLevStages - 1);
            const LevStage& st = ring[t % kLevStages];
#pragma unroll
            for (int j = 0; j < kLevTile; ++j) {
                const float4 g = *reinterpret_cast<const float4*>(&st.g[j][4 * rq]);
                const float4 x = *reinterpret_cast<const float4*>(&st.q[j][4 * kq]);
                const float gu[4] = {g.x, g.y, g.z, g.w}, xk[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int k = 0; k < 4; ++k) a[u][k] = fmaf(gu[u], xk[k], a[u][k]);
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // the ring is free for the next block
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + 4 * rq + u;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i < ns && k0 + 4 * kq + k < rr) Y[(int64_t)i * rr + k0 + 4 * kq + k] = a[u][k];
        }
    }
}

bool frame_ok3(const lt_frame* f) { return f && f->slice_off && f->S > 0 && f->S <= 1024 && f->C >= 1 && f->pts; }

}  // namespace

// ---------------------------------------------------------------- C ABI
extern "C" lt_status lt_proposal_features(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, float* feat,
                                          int32_t* group_off) {
    if (!ctx || !frame_ok3(f) || !smp || !smp->ncol || !smp->key || !smp->val || !smp->n1 || !smp->col_node || !feat ||
        !group_off)
        return lt_fail(ctx, LT_EINVAL, "lt_proposal_features: bad arguments");
    cudaSetDevice(ctx->device);
    lt_status st;
    float* stats = (float*)lt_scratch(ctx, SCR_PROPOSAL, (size_t)f->S * kSliceStats * 4, &st);
    if (!stats) return st;
    k_feat_slice<<<f->S, 256, 0, ctx->stream>>>(*f, *smp, stats);
    LT_LAUNCH_CHECK(ctx, "k_feat_slice");
    k_group_prefix<<<1, 1024, 0, ctx->stream>>>(smp->ncol, f->S, group_off);
    LT_LAUNCH_CHECK(ctx, "k_group_prefix");
    const unsigned grid = (unsigned)std::max(1, std::min((f->C + 7) / 8, 8 * ctx->num_sms / f->S));
    k_feat_cols<<<dim3(grid, f->S), 256, 0, ctx->stream>>>(*f, *smp, stats, group_off, feat);
    LT_LAUNCH_CHECK(ctx, "k_feat_cols");
    return LT_OK;
}

extern "C" lt_status lt_proposal_forward(lt_ctx* ctx, const float* theta, const float* feat, int64_t n_max,
                                         const int32_t* n_dev, float* z) {
    if (!ctx || !theta || !feat || !z || n_max < 0) return lt_fail(ctx, LT_EINVAL, "lt_proposal_forward: bad arguments");
    if (n_max == 0) return LT_OK;
    cudaSetDevice(ctx->device);
    const size_t shm = sizeof(MlpSmem);
    LT_CUDA(ctx, cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_max + TM - 1) / TM, 3 * ctx->num_sms));
    k_mlp_forward<<<grid, MT, shm, ctx->stream>>>(theta, feat, n_max, n_dev, z);
    LT_LAUNCH_CHECK(ctx, "k_mlp_forward");
    return LT_OK;
}

extern "C" lt_status lt_proposal_weights(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp,
                                         const int32_t* group_off, const float* z, float mix, float* w) {
    if (!ctx || !frame_ok3(f) || !smp || !smp->ncol || !smp->g || !group_off || !z || !w || !(mix >= 0.f && mix <= 1.f))
        return lt_fail(ctx, LT_EINVAL, "lt_proposal_weights: bad arguments");
    cudaSetDevice(ctx->device);
    k_mix_weights<<<(f->S + 7) / 8, 256, 0, ctx->stream>>>(*f, *smp, group_off, z, mix, w);
    LT_LAUNCH_CHECK(ctx, "k_mix_weights");
    return LT_OK;
}

extern "C" lt_status lt_slice_matrices(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, float d_min, float* M,
                                       int64_t cap, int64_t* moff) {
    if (!ctx || !frame_ok3(f) || !smp || !smp->ncol || !smp->col_node || !M || !moff || cap < 0)
        return lt_fail(ctx, LT_EINVAL, "lt_slice_matrices: bad arguments");
    if (!ctx->d_cell_off) return lt_fail(ctx, LT_EINVAL, "lt_slice_matrices: no scene uploaded");
    cudaSetDevice(ctx->device);
    k_moff<<<1, 1024, 0, ctx->stream>>>(*f, *smp, moff);
    LT_LAUNCH_CHECK(ctx, "k_moff");
    k_slice_matrix<<<dim3(std::max(1, 32 * ctx->num_sms / f->S), f->S), 128, 0, ctx->stream>>>(
        *f, *smp, ctx->grid, d_min * d_min, moff, cap, M, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_slice_matrix");
    return LT_OK;
}

extern "C" lt_status lt_leverage_targets(lt_ctx* ctx, const lt_frame* f, const lt_samples* smp, const float* M,
                                         const int64_t* moff, const int32_t* group_off, int32_t r, int32_t iters,
                                         uint64_t seed, float* target) {
    if (!ctx || !frame_ok3(f) || !smp || !smp->ncol || !M || !moff || !group_off || !target || r < 1 || r > 64 ||
        iters < 0)
        return lt_fail(ctx, LT_EINVAL, "lt_leverage_targets: bad arguments");
    cudaSetDevice(ctx->device);
    const int S = f->S, C = f->C;
    // Gram capacity: slices of any n' whose squares add up to at most S min(C, 4096)^2
    // floats, and the padding of their rows, at most 3 floats each (S slices whose squares add
    // up to S nmax^2 have at most S nmax rows).  More latches LT_ELIMIT and no target is written.
    const int64_t nmax = std::min<int64_t>(C, 4096);
    const int64_t gcap = (int64_t)S * (nmax * nmax + 3 * nmax);
    lt_status st;
    auto up = [](size_t n) { return (n + 255) & ~(size_t)255; };  // each part starts on 256 bytes
    const size_t b_g = up((size_t)gcap * 4), b_q = up((size_t)S * C * r * 4);
    char* p = (char*)lt_scratch(ctx, SCR_PROPOSAL_T, b_g + 2 * b_q + (size_t)(S + 1) * 16, &st);
    if (!p) return st;
    float* G = (float*)p;
    float* Q = (float*)(p + b_g);
    float* Y = (float*)(p + b_g + b_q);
    int64_t* goff2 = (int64_t*)(p + b_g + 2 * b_q);
    int64_t* tpfx = goff2 + S + 1;
    k_goff<<<1, 1024, 0, ctx->stream>>>(*smp, S, goff2, tpfx, gcap, ctx->d_status);
    LT_LAUNCH_CHECK(ctx, "k_goff");
    k_gram<<<2 * ctx->num_sms, 256, 0, ctx->stream>>>(*f, *smp, M, moff, goff2, tpfx, gcap, G);
    LT_LAUNCH_CHECK(ctx, "k_gram");
    // Q of a round is the product of the round before: the two buffers change roles
    const unsigned rows = (unsigned)std::max(1, std::min((C + kLevRows - 1) / kLevRows, 8 * ctx->num_sms / S));
    const size_t shm = kLevStages * sizeof(LevStage);
    LT_CUDA(ctx, cudaFuncSetAttribute(k_lev_mult, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    for (int it = 0; it <= iters; ++it) {
        k_lev_mgs<<<S, kLevThreads, 0, ctx->stream>>>(*smp, f->slice_id, S, C, goff2, gcap, r, it == 0, it == iters, seed,
                                                      Q, Y, group_off, target);
        LT_LAUNCH_CHECK(ctx, "k_lev_mgs");
        if (it < iters) {
            k_lev_mult<<<dim3(rows, S), kLevRows, shm, ctx->stream>>>(*smp, S, C, G, goff2, gcap, r, Q, Y);
            LT_LAUNCH_CHECK(ctx, "k_lev_mult");
            std::swap(Q, Y);
        }
    }
    return LT_OK;
}

extern "C" lt_status lt_proposal_init(lt_ctx* ctx, uint64_t seed, float* theta) {
    if (!ctx || !theta) return lt_fail(ctx, LT_EINVAL, "lt_proposal_init: bad arguments");
    cudaSetDevice(ctx->device);
    k_mlp_init<<<(NPAR + 255) / 256, 256, 0, ctx->stream>>>(seed, theta);
    LT_LAUNCH_CHECK(ctx, "k_mlp_init");
    return LT_OK;
}

extern "C" lt_status lt_proposal_grad(lt_ctx* ctx, const float* theta, const float* feat, const float* target,
                                      const int32_t* group_off, int32_t ngroups, int64_t n, float* grad, float* loss) {
    if (!ctx || !theta || !feat || !target || !group_off || !grad || ngroups < 1 || n < 1)
        return lt_fail(ctx, LT_EINVAL, "lt_proposal_grad: bad arguments");
    cudaSetDevice(ctx->device);
    const int nparts = (int)std::min<int64_t>((n + TM - 1) / TM, ctx->num_sms);
    lt_status st;
    char* p = (char*)lt_scratch(ctx, SCR_PROPOSAL_G,
                                (size_t)n * 8 + (size_t)ngroups * 4 + (size_t)nparts * NPAR * 4 + 4 * 256, &st);
    if (!p) return st;
    float* z = (float*)p;
    float* dz = z + n;
    float* gloss = (float*)((char*)p + (((size_t)n * 8 + 255) & ~(size_t)255));
    float* part = (float*)((char*)gloss + (((size_t)ngroups * 4 + 255) & ~(size_t)255));
    lt_status s1 = lt_proposal_forward(ctx, theta, feat, n, nullptr, z);
    if (s1 != LT_OK) return s1;
    k_group_softmax<<<ngroups, 32, 0, ctx->stream>>>(z, target, group_off, ngroups, dz, gloss);
    LT_LAUNCH_CHECK(ctx, "k_group_softmax");
    const size_t shm = sizeof(BwdSmem);
    LT_CUDA(ctx, cudaFuncSetAttribute(k_mlp_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    k_mlp_backward<<<nparts, MT, shm, ctx->stream>>>(theta, feat, dz, n, part);
    LT_LAUNCH_CHECK(ctx, "k_mlp_backward");
    k_grad_reduce<<<(NPAR + 63) / 64, 64, 0, ctx->stream>>>(part, nparts, grad, gloss, ngroups, loss);
    LT_LAUNCH_CHECK(ctx, "k_grad_reduce");
    return LT_OK;
}

extern "C" lt_status lt_proposal_adam(lt_ctx* ctx, float* theta, float* m, float* v, const float* grad, int32_t step,
                                      float lr) {
    if (!ctx || !theta || !m || !v || !grad || step < 1 || !(lr >= 0.f))
        return lt_fail(ctx, LT_EINVAL, "lt_proposal_adam: bad arguments");
    cudaSetDevice(ctx->device);
    k_adam<<<(NPAR + 255) / 256, 256, 0, ctx->stream>>>(theta, m, v, grad, step, lr);
    LT_LAUNCH_CHECK(ctx, "k_adam");
    return LT_OK;
}
