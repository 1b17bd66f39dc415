// Learned interpolation: the 112-128-128-16 ReLU MLP that predicts a fine point's row of
// P from its features, trained on the least-squares rows of Algorithm 2 (Eq. (3.6)).
// The paper has no learned interpolation; the definitions (features, bfloat16-rounded
// product inputs with FP32 sums, masked MSE, Adam of Kingma & Ba with beta1 = 0.9,
// beta2 = 0.999, eps = 1e-8, He-uniform initialisation from SplitMix64) are those of the
// interface declared in include/bamg.h.
//
// All products run on the tensor cores (mma.sync m16n8k16, bf16 in, FP32 accumulate), the
// weights staged once per block in shared memory with a padded row stride: in the forward pass
// one warp takes 16 rows through all layers, in a training step four warps do.  The training
// backward's products (input gradients through the ReLU masks, weight gradients summed over the
// batch) use the same instruction with the incoming gradient rounded to bf16; bias gradients and
// Adam stay in FP32.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstddef>
#include <cstdio>
#include <vector>

#include "kernels.cuh"

namespace bamg {

// ------------------------------------------------------------------ parameter layout
// One flat FP32 buffer [W1 | b1 | W2 | b2 | W3 | b3]; W_l is out x in, row-major.  The
// bfloat16 copies of W1, W2, W3 sit in one buffer in the same order, their rows padded as the
// kernels keep them in shared memory (ldmatrix rows on distinct banks), so that a block stages
// all of them with one flat copy.
constexpr int64_t OFF_W1 = 0;
constexpr int64_t OFF_B1 = OFF_W1 + (int64_t)MLP_H * MLP_F;
constexpr int64_t OFF_W2 = OFF_B1 + MLP_H;
constexpr int64_t OFF_B2 = OFF_W2 + (int64_t)MLP_H * MLP_H;
constexpr int64_t OFF_W3 = OFF_B2 + MLP_H;
constexpr int64_t OFF_B3 = OFF_W3 + (int64_t)MLP_S * MLP_H;
constexpr int64_t NPARAM = OFF_B3 + MLP_S;
constexpr int NET_LD1 = MLP_F + 8, NET_LD2 = MLP_H + 8;  // padded strides of the bf16 copies
constexpr int64_t BOFF_W1 = 0;
constexpr int64_t BOFF_W2 = BOFF_W1 + (int64_t)MLP_H * NET_LD1;
constexpr int64_t BOFF_W3 = BOFF_W2 + (int64_t)MLP_H * NET_LD2;
constexpr int64_t NBF = BOFF_W3 + (int64_t)MLP_S * NET_LD2;

int64_t mlp_param_count() { return NPARAM; }

// index of a flat parameter in the bf16 copy, or -1 for a bias
__device__ __forceinline__ int64_t bf_index(int64_t q) {
    const int i = (int)q;
    if (q < OFF_B1) return BOFF_W1 + i / MLP_F * NET_LD1 + i % MLP_F;
    if (q >= OFF_W2 && q < OFF_B2) return BOFF_W2 + (i - (int)OFF_W2) / MLP_H * NET_LD2 + (i - (int)OFF_W2) % MLP_H;
    if (q >= OFF_W3 && q < OFF_B3) return BOFF_W3 + (i - (int)OFF_W3) / MLP_H * NET_LD2 + (i - (int)OFF_W3) % MLP_H;
    return -1;
}

// He-uniform weights W = (2u - 1) sqrt(6 / fan_in), u = SplitMix64 uniform of
// (seed, stream = layer, index); biases zero.
__global__ void k_mlp_init(uint64_t seed, float* __restrict__ P) {
    pdl_begin();
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= NPARAM) return;
    int layer = -1;
    int64_t idx = 0;
    int fan = 1;
    if (q < OFF_B1) {
        layer = 0, idx = q, fan = MLP_F;
    } else if (q >= OFF_W2 && q < OFF_B2) {
        layer = 1, idx = q - OFF_W2, fan = MLP_H;
    } else if (q >= OFF_W3 && q < OFF_B3) {
        layer = 2, idx = q - OFF_W3, fan = MLP_H;
    }
    if (layer < 0) {
        P[q] = 0.f;
        return;
    }
    const double u = counter_uniform(seed, (uint64_t)layer, (uint64_t)idx);
    P[q] = (float)((2.0 * u - 1.0) * sqrt(6.0 / (double)fan));
}

__global__ void k_mlp_to_bf16(const float* __restrict__ P, __nv_bfloat16* __restrict__ Wb) {
    pdl_begin();
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= NPARAM) return;
    const int64_t b = bf_index(q);
    if (b >= 0) Wb[b] = __float2bfloat16_rn(P[q]);
}

// ------------------------------------------------------------------ forward (tensor cores)
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // one conversion instruction for both
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t load_pair(const float* p) {  // elements p[0], p[1] as bf16x2
    const float2 v = *reinterpret_cast<const float2*>(p);
    return pack_bf16(v.x, v.y);
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ------------------------------------------------------------------ the network in one kernel
// All three layers of a row tile in one warp, the activations in registers: an m16n8
// accumulator holds the same elements of a row as the m16k16 fragment of the next product
// needs, so relu and the rounding to bf16 turn it into the next layer's A operand in place.
// The k-steps run in the order of a layer on its own, so the values are those of three
// separate layer kernels, bit for bit.
//
// What bounds it: the tensor pipe under mma.sync (29 us at its rate for 2^18 rows, ncu), then HBM
// (134 MB in and out, 20 us of the copy rate).  Three layer kernels passed H1 and H2 through memory
// (400 MB), loaded weight fragments four bytes at a time and staged the weights in every block of
// 64 rows: 178 us.  Here one block per SM keeps all weights in shared memory (71 KB, staged once)
// and its 12 warps walk the 16-row tiles; ldmatrix fetches four fragment registers at a time, and
// each warp's next feature tile arrives by cp.async while the current one is computed: 45 us.
// Measured besides: two row tiles a warp sharing each weight fragment, 52 us with 8 warps and 64
// with 10 (registers), 58 with 12 and no feature staging; one row tile with 16 warps, 48 us.
constexpr int NET_WARPS = 12;
constexpr int NET_LDX = MLP_F + 8;  // of a feature tile: the fragment loads of a half warp on distinct banks
struct NetSmem {
    __nv_bfloat16 w1[MLP_H * NET_LD1];
    __nv_bfloat16 w2[MLP_H * NET_LD2];
    __nv_bfloat16 w3[MLP_S * NET_LD2];
    float b1[MLP_H], b2[MLP_H], b3[MLP_S];
};

__device__ __forceinline__ void net_cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// All weights and biases into shared memory; every thread of the block calls it.
static_assert(offsetof(NetSmem, b1) == sizeof(__nv_bfloat16) * NBF && NBF % 8 == 0, "one flat copy of the weights");
template <int THREADS>
__device__ __forceinline__ void net_stage_weights(NetSmem& sm, const __nv_bfloat16* __restrict__ Wb,
                                                  const float* __restrict__ P) {
    constexpr int C = (int)(NBF / 8);  // 16-byte pieces
#pragma unroll
    for (int e = 0; e < (C + THREADS - 1) / THREADS; ++e) {
        const int c = e * THREADS + threadIdx.x;
        if (c < C) net_cp16(sm.w1 + 8 * c, Wb + 8 * c);
    }
    for (int e = threadIdx.x; e < MLP_H; e += blockDim.x) {
        sm.b1[e] = P[OFF_B1 + e];
        sm.b2[e] = P[OFF_B2 + e];
        if (e < MLP_S) sm.b3[e] = P[OFF_B3 + e];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
}

// the fragments b0, b1 of two neighbouring n8 tiles at one k16 step: w = the element (n, k) of
// the first tile's corner, rows of LD
template <int LD>
__device__ __forceinline__ void net_ldb(uint32_t (&b)[4], const __nv_bfloat16* w, int lane) {
    const __nv_bfloat16* p = w + ((lane & 7) + ((lane >> 4) << 3)) * LD + ((lane >> 3) & 1) * 8;
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
// acc (NT n8 tiles) = A W^T for the NT * 8 outputs whose weights start at w
template <int NT, int KS, int LD>
__device__ __forceinline__ void net_product(float (&acc)[NT][4], const uint32_t (&A)[KS][4], const __nv_bfloat16* w,
                                            int lane) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll
    for (int k = 0; k < KS; ++k) {
#pragma unroll
        for (int n = 0; n < NT; n += 2) {
            uint32_t b[4];
            net_ldb<LD>(b, w + n * 8 * LD + k * 16, lane);
            mma_bf16(acc[n], A[k][0], A[k][1], A[k][2], A[k][3], b[0], b[1]);
            mma_bf16(acc[n + 1], A[k][0], A[k][1], A[k][2], A[k][3], b[2], b[3]);
        }
    }
}
// One hidden layer: the next layer's A operand from this one's (128 outputs in slices of 32)
template <int KS, int LD>
__device__ __forceinline__ void net_hidden(const uint32_t (&A)[KS][4], uint32_t (&H)[8][4], const __nv_bfloat16* w,
                                           const float* bias, int lane) {
    const int t = lane & 3;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float acc[4][4];
        net_product<4, KS, LD>(acc, A, w + c * 32 * LD, lane);
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const float2 bb = *reinterpret_cast<const float2*>(bias + c * 32 + n * 8 + 2 * t);
            uint32_t* h = H[2 * c + (n >> 1)] + 2 * (n & 1);
            h[0] = pack_bf16(fmaxf(acc[n][0] + bb.x, 0.f), fmaxf(acc[n][1] + bb.y, 0.f));
            h[1] = pack_bf16(fmaxf(acc[n][2] + bb.x, 0.f), fmaxf(acc[n][3] + bb.y, 0.f));
        }
    }
}

// Copies ROWS rows of X from r0 (those < M; 448 bytes each, contiguous) into a tile buffer by one
// warp, asynchronously: 16-byte pieces where X allows them (wide), else 8-byte ones.
template <int ROWS>
__device__ __forceinline__ void net_fetch(float* buf, const float* __restrict__ X, int64_t r0, int64_t M, bool wide,
                                          int lane) {
    const int rows = (int)(M - r0 < ROWS ? M - r0 : ROWS);
    const float* src = X + r0 * MLP_F;
    if (wide) {
        constexpr int C = MLP_F / 4;
#pragma unroll
        for (int e = lane; e < ROWS * C; e += 32) {
            const int r = e / C, c = e - r * C;
            if (r < rows) net_cp16(buf + r * NET_LDX + 4 * c, src + 4 * e);
        }
    } else {
        constexpr int C = MLP_F / 2;
        for (int e = lane; e < rows * C; e += 32) {
            const int r = e / C, c = e - r * C;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                             (unsigned)__cvta_generic_to_shared(buf + r * NET_LDX + 2 * c)),
                         "l"(src + 2 * e)
                         : "memory");
        }
    }
}

// The first product's A operand from a feature tile (va, vb: rows g and g + 8 exist)
__device__ __forceinline__ void net_inputs(uint32_t (&A)[MLP_F / 16][4], const float* buf, bool va, bool vb, int g,
                                           int t) {
    const float* p = buf + g * NET_LDX + 2 * t;
#pragma unroll
    for (int k = 0; k < MLP_F / 16; ++k) {
        A[k][0] = va ? load_pair(p + 16 * k) : 0u;
        A[k][1] = vb ? load_pair(p + 8 * NET_LDX + 16 * k) : 0u;
        A[k][2] = va ? load_pair(p + 16 * k + 8) : 0u;
        A[k][3] = vb ? load_pair(p + 8 * NET_LDX + 16 * k + 8) : 0u;
    }
}

__global__ void __launch_bounds__(NET_WARPS * 32)
    k_mlp_net(int64_t M, const float* __restrict__ X, const __nv_bfloat16* __restrict__ Wb, const float* __restrict__ P,
              float* __restrict__ Y) {
    pdl_begin();
    extern __shared__ __align__(16) unsigned char net_raw[];
    NetSmem& sm = *reinterpret_cast<NetSmem*>(net_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    float* buf = reinterpret_cast<float*>(net_raw + sizeof(NetSmem)) + warp * (16 * NET_LDX);
    const int64_t tiles = (M + 15) / 16, step = (int64_t)gridDim.x * NET_WARPS;
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    // neighbouring tiles on different SMs, so that few rows spread over the whole chip
    int64_t q = blockIdx.x + (int64_t)gridDim.x * warp;
    if (q < tiles) net_fetch<16>(buf, X, q * 16, M, wide, lane);
    net_stage_weights<NET_WARPS * 32>(sm, Wb, P);
    for (; q < tiles; q += step) {
        const int64_t ra = q * 16 + g, rb = ra + 8;
        const bool va = ra < M, vb = rb < M;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        uint32_t H1[8][4], H2[8][4];
        {
            uint32_t A[MLP_F / 16][4];
            net_inputs(A, buf, va, vb, g, t);
            __syncwarp();  // the tile is in registers: its buffer takes the next one meanwhile
            if (q + step < tiles) net_fetch<16>(buf, X, (q + step) * 16, M, wide, lane);
            net_hidden<MLP_F / 16, NET_LD1>(A, H1, sm.w1, sm.b1, lane);
        }
        net_hidden<MLP_H / 16, NET_LD2>(H1, H2, sm.w2, sm.b2, lane);
        float acc[2][4];
        net_product<2, MLP_H / 16, NET_LD2>(acc, H2, sm.w3, lane);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int c = n * 8 + 2 * t;
            const float2 bb = *reinterpret_cast<const float2*>(sm.b3 + c);
            if (va) *reinterpret_cast<float2*>(Y + ra * MLP_S + c) = make_float2(acc[n][0] + bb.x, acc[n][1] + bb.y);
            if (vb) *reinterpret_cast<float2*>(Y + rb * MLP_S + c) = make_float2(acc[n][2] + bb.x, acc[n][3] + bb.y);
        }
    }
}

// ------------------------------------------------------------------ backward
// A training step is two kernels and the optimiser.  k_mlp_step takes a row tile through the
// forward pass, the masked loss and the input gradients in four warps, which pass it on through
// shared memory; the gradient that enters a product is rounded to bf16 like the forward's inputs.  It
// leaves H1, H2 and (up to KEEP_ROWS rows) the rounded gradients in memory (bf16) for the weight gradients
// and the unrounded gradients (FP32) for the bias gradients (k_mlp_wgrad, all layers in one launch),
// and adds up the loss.
//
// What bounds it: launches and latency (a batch of 4096 rows is 0.9 GFLOP and 6 MB; 10 us of
// dependent instructions in k_mlp_step and 6 in k_mlp_wgrad, tensor pipe below 10%).  It took 14
// launches and 143 us, 88 of them in column sums that one block per column walked row by row, 26 in
// the transposing loads of each weight gradient; now three launches and 30 us.  (Summing the bias
// gradients in k_mlp_step's warps and 128 rows a weight block measured 27 us; the order of the sums
// here, 256 rows a chain and the column sums' tree, is the one the results always had.)

// B fragments of two neighbouring n8 tiles at one k16 step for a product with W itself (k = the
// row of w, n = the column): w = the corner (k, n), rows of LD
template <int LD>
__device__ __forceinline__ void net_ldb_t(uint32_t (&b)[4], const __nv_bfloat16* w, int lane) {
    const __nv_bfloat16* p = w + ((lane & 7) + ((lane >> 3) & 1) * 8) * LD + ((lane >> 4) << 3);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
// A operand of one k16 step from a 16-row bf16 tile in shared memory (rows of NET_LD2)
__device__ __forceinline__ void net_lda(uint32_t (&a)[4], const __nv_bfloat16* tile, int k, int lane) {
    const __nv_bfloat16* p = tile + ((lane & 7) + ((lane >> 3) & 1) * 8) * NET_LD2 + 16 * k + ((lane >> 4) << 3);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
// The warp's 32 columns (from c0) of a row tile in the A-operand layout, to the tile in shared
// memory and to rows ra, rb of a row-major bf16 matrix (OUT)
template <bool OUT = true>
__device__ __forceinline__ void step_put(__nv_bfloat16* tile, __nv_bfloat16* __restrict__ O, const uint32_t (&H)[2][4],
                                         int c0, int64_t ra, int64_t rb, bool va, bool vb, int g, int t) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int c = c0 + 16 * k + 8 * e + 2 * t;
            if (tile) {
                *reinterpret_cast<uint32_t*>(tile + g * NET_LD2 + c) = H[k][2 * e];
                *reinterpret_cast<uint32_t*>(tile + (g + 8) * NET_LD2 + c) = H[k][2 * e + 1];
            }
            if (OUT && va) *reinterpret_cast<uint32_t*>(O + ra * MLP_H + c) = H[k][2 * e];
            if (OUT && vb) *reinterpret_cast<uint32_t*>(O + rb * MLP_H + c) = H[k][2 * e + 1];
        }
}
// relu(acc + bias) of the warp's 32 columns, rounded
__device__ __forceinline__ void step_relu(uint32_t (&H)[2][4], const float (&acc)[4][4], const float* bias, int t) {
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const float2 bb = *reinterpret_cast<const float2*>(bias + n * 8 + 2 * t);
        uint32_t* h = H[n >> 1] + 2 * (n & 1);
        h[0] = pack_bf16(fmaxf(acc[n][0] + bb.x, 0.f), fmaxf(acc[n][1] + bb.y, 0.f));
        h[1] = pack_bf16(fmaxf(acc[n][2] + bb.x, 0.f), fmaxf(acc[n][3] + bb.y, 0.f));
    }
}
// The gradient through the ReLU mask H > 0 to F (FP32, row-major), rounded into O
__device__ __forceinline__ void step_mask(uint32_t (&O)[2][4], const float (&acc)[4][4], const uint32_t (&H)[2][4],
                                          float* __restrict__ F, int c0, int64_t ra, int64_t rb, bool va, bool vb,
                                          int t) {
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const int k = n >> 1, e = 2 * (n & 1), c = c0 + 8 * n + 2 * t;
        const __nv_bfloat162 ha = *reinterpret_cast<const __nv_bfloat162*>(&H[k][e]);
        const __nv_bfloat162 hb = *reinterpret_cast<const __nv_bfloat162*>(&H[k][e + 1]);
        const float v0 = __low2float(ha) > 0.f ? acc[n][0] : 0.f, v1 = __high2float(ha) > 0.f ? acc[n][1] : 0.f;
        const float v2 = __low2float(hb) > 0.f ? acc[n][2] : 0.f, v3 = __high2float(hb) > 0.f ? acc[n][3] : 0.f;
        O[k][e] = pack_bf16(v0, v1);
        O[k][e + 1] = pack_bf16(v2, v3);
        if (va) *reinterpret_cast<float2*>(F + ra * MLP_H + c) = make_float2(v0, v1);
        if (vb) *reinterpret_cast<float2*>(F + rb * MLP_H + c) = make_float2(v2, v3);
    }
}

// Forward, loss (sum mask (Y - T)^2 / M added to *loss; mask = the features' slot-valid flags) and
// input gradients of M rows.
//
// Four warps share a row tile, 32 columns of every layer each, and pass the tile on through shared
// memory: a batch of 4096 rows has only 256 tiles, and one warp through all the products of a
// tile took 13 us of dependent instructions.  `early`: X was complete before the preceding kernel
// began, so the first feature tile is fetched while that one still runs.
//
// KEEP: the rounded gradients are left in memory beside the unrounded ones (gradients() chooses).
constexpr int STEP_GROUPS = 2, STEP_WARPS = 4 * STEP_GROUPS;
struct StepOut {
    __nv_bfloat16 *H1, *H2, *D1, *D2, *D3;  // activations and rounded gradients, M x 128 (D3: M x 16; D with KEEP)
    float *F1, *F2, *F3;                    // the gradients unrounded
    float* G;                               // the flat gradient
    double* loss;
};
struct StepSmem {
    NetSmem net;
    float x[STEP_GROUPS][16 * NET_LDX];            // feature tiles
    __nv_bfloat16 h[STEP_GROUPS][2][16 * NET_LD2];  // H1 then D2, and H2
};
__device__ __forceinline__ void step_sync(int group) {
    asm volatile("bar.sync %0, 128;" ::"r"(group + 1) : "memory");
}
// net_fetch by the four warps of a group
__device__ __forceinline__ void step_fetch(float* buf, const float* __restrict__ X, int64_t r0, int64_t M, bool wide,
                                           int w, int lane) {
    if (r0 + 4 * w < M) net_fetch<4>(buf + 4 * w * NET_LDX, X, r0 + 4 * w, M, wide, lane);
}
template <bool KEEP>
__global__ void __launch_bounds__(STEP_WARPS * 32)
    k_mlp_step(int64_t M, const float* __restrict__ X, const float* __restrict__ Tg, const __nv_bfloat16* __restrict__ Wb,
               const float* __restrict__ P, const StepOut out, bool early) {
    extern __shared__ __align__(16) unsigned char net_raw[];
    StepSmem& sm = *reinterpret_cast<StepSmem*>(net_raw);
    __shared__ double s_loss[STEP_GROUPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int group = warp >> 2, w = warp & 3, c0 = 32 * w;
    float* buf = sm.x[group];
    __nv_bfloat16 *h1t = sm.h[group][0], *h2t = sm.h[group][1];
    const int64_t tiles = (M + 15) / 16, step = (int64_t)gridDim.x * STEP_GROUPS;
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    int64_t q = blockIdx.x + (int64_t)gridDim.x * group;
    if (early && q < tiles) step_fetch(buf, X, q * 16, M, wide, w, lane);
    pdl_begin();
    if (!early && q < tiles) step_fetch(buf, X, q * 16, M, wide, w, lane);
    net_stage_weights<STEP_WARPS * 32>(sm.net, Wb, P);
    double l = 0.0;
    const float fm = (float)M;
    for (; q < tiles; q += step) {
        const int64_t ra = q * 16 + g, rb = ra + 8;
        const bool va = ra < M, vb = rb < M;
        float tg[2][4];  // targets of this lane's eight outputs (they may be only 4-byte aligned)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = n * 8 + 2 * t + (e & 1);
                tg[n][e] = (e < 2 ? va : vb) ? Tg[(e < 2 ? ra : rb) * MLP_S + c] : 0.f;
            }
        asm volatile("cp.async.wait_all;" ::: "memory");
        step_sync(group);
        uint32_t H1[2][4], H2[2][4], D[2][4];
        unsigned on = 0u;  // slot-valid flags of this lane's eight outputs
        float acc[4][4];
        {
            uint32_t A[MLP_F / 16][4];
            net_inputs(A, buf, va, vb, g, t);
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float* f = buf + g * NET_LDX + MLP_NF_SLOT * (n * 8 + 2 * t + e);
                    if (va && f[0] > 0.f) on |= 1u << (4 * n + e);
                    if (vb && f[8 * NET_LDX] > 0.f) on |= 1u << (4 * n + 2 + e);
                }
            net_product<4, MLP_F / 16, NET_LD1>(acc, A, sm.net.w1 + c0 * NET_LD1, lane);
        }
        step_relu(H1, acc, sm.net.b1 + c0, t);
        step_put(h1t, out.H1, H1, c0, ra, rb, va, vb, g, t);
        step_sync(group);  // H1 is whole; the feature tile has been read and takes the next one
        if (q + step < tiles) step_fetch(buf, X, (q + step) * 16, M, wide, w, lane);
        uint32_t A[MLP_H / 16][4];
#pragma unroll
        for (int k = 0; k < MLP_H / 16; ++k) net_lda(A[k], h1t, k, lane);
        net_product<4, MLP_H / 16, NET_LD2>(acc, A, sm.net.w2 + c0 * NET_LD2, lane);
        step_relu(H2, acc, sm.net.b2 + c0, t);
        step_put(h2t, out.H2, H2, c0, ra, rb, va, vb, g, t);
        step_sync(group);
#pragma unroll
        for (int k = 0; k < MLP_H / 16; ++k) net_lda(A[k], h2t, k, lane);
        float y[2][4];  // every warp forms all 16 outputs and their gradients
        net_product<2, MLP_H / 16, NET_LD2>(y, A, sm.net.w3, lane);
        uint32_t D3[4];
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const float2 bb = *reinterpret_cast<const float2*>(sm.net.b3 + n * 8 + 2 * t);
            float d[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float mask = (on >> (4 * n + e)) & 1u ? 1.f : 0.f;
                const float r = (e < 2 ? va : vb) ? mask * (y[n][e] + (e & 1 ? bb.y : bb.x) - tg[n][e]) : 0.f;
                if (w == 0) l += (double)r * (double)r;
                d[e] = 2.f * r / fm;
            }
            D3[2 * n] = pack_bf16(d[0], d[1]);
            D3[2 * n + 1] = pack_bf16(d[2], d[3]);
            if (w == 0) {
                const int c = n * 8 + 2 * t;
                if (va) {
                    if (KEEP) *reinterpret_cast<uint32_t*>(out.D3 + ra * MLP_S + c) = D3[2 * n];
                    *reinterpret_cast<float2*>(out.F3 + ra * MLP_S + c) = make_float2(d[0], d[1]);
                }
                if (vb) {
                    if (KEEP) *reinterpret_cast<uint32_t*>(out.D3 + rb * MLP_S + c) = D3[2 * n + 1];
                    *reinterpret_cast<float2*>(out.F3 + rb * MLP_S + c) = make_float2(d[2], d[3]);
                }
            }
        }
        // D2 = D3 W3 through H2's mask, D1 = D2 W2 through H1's
#pragma unroll
        for (int n = 0; n < 4; n += 2) {
            uint32_t b[4];
            net_ldb_t<NET_LD2>(b, sm.net.w3 + c0 + n * 8, lane);
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[n][e] = acc[n + 1][e] = 0.f;
            mma_bf16(acc[n], D3[0], D3[1], D3[2], D3[3], b[0], b[1]);
            mma_bf16(acc[n + 1], D3[0], D3[1], D3[2], D3[3], b[2], b[3]);
        }
        step_mask(D, acc, H2, out.F2, c0, ra, rb, va, vb, t);
        step_put<KEEP>(h1t, out.D2, D, c0, ra, rb, va, vb, g, t);  // over H1: every warp has read it
        step_sync(group);
#pragma unroll
        for (int k = 0; k < MLP_H / 16; ++k) net_lda(A[k], h1t, k, lane);
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll
        for (int k = 0; k < MLP_H / 16; ++k)
#pragma unroll
            for (int n = 0; n < 4; n += 2) {
                uint32_t b[4];
                net_ldb_t<NET_LD2>(b, sm.net.w2 + k * 16 * NET_LD2 + c0 + n * 8, lane);
                mma_bf16(acc[n], A[k][0], A[k][1], A[k][2], A[k][3], b[0], b[1]);
                mma_bf16(acc[n + 1], A[k][0], A[k][1], A[k][2], A[k][3], b[2], b[3]);
            }
        step_mask(D, acc, H1, out.F1, c0, ra, rb, va, vb, t);
        if (KEEP) step_put(nullptr, out.D1, D, c0, ra, rb, va, vb, g, t);
        // the next tile's H1 goes over D2 after the barrier at its start
    }
    if (w == 0) {
        l = warp_sum(l);
        if (lane == 0) s_loss[group] = l;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int i = 0; i < STEP_GROUPS; ++i) v += s_loss[i];
        atomicAdd(out.loss, v / (double)M);
    }
}

// Weight and bias gradients of all layers in one launch.  Weights: G[n][k] += sum_m D[m][n] X[m][k]
// (D: the rounded gradient at the layer's output, X: its input, features rounded here), block (x, y)
// taking rows [x rows, +rows) and, by y, a slab of 32 outputs of layer 2 (y = 0..3) or 1 (4..7), or
// layer 3 (8).  Both operands are staged row-major in shared memory, WG_MC rows at a time, and
// ldmatrix transposes them into fragments (the products run along the rows).  A chain of products
// covers WG_MC rows and its FP32 sums are then added up in registers: the tensor pipe's own sums
// truncate, and chains of 2304 rows showed it (2.5e-6 of a gradient against 3e-7).  The block's sums
// go to G in pairs with atomics.  Biases (y >= 9): the column sums of the unrounded gradients.
constexpr int WG_MC = 256, WG_WARPS = 8, WG_WJOBS = 9, WG_JOBS = WG_WJOBS + 3;
constexpr int WG_LDD = 32 + 8, WG_LDX = MLP_H + 8;
constexpr size_t WG_SMEM = sizeof(__nv_bfloat16) * WG_MC * (WG_LDD + WG_LDX);

__device__ __forceinline__ void ldmatrix_t(uint32_t (&f)[4], const __nv_bfloat16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
// cnt rows of C columns (a multiple of 8, from column c0 of LDG) into rows of LDS; zeros to WG_MC rows
template <int C, int LDG, int LDS>
__device__ __forceinline__ void wg_stage(__nv_bfloat16* s, const __nv_bfloat16* __restrict__ src, int c0, int64_t m0,
                                         int cnt) {
    constexpr int Q = C / 8;
#pragma unroll
    for (int e = threadIdx.x; e < WG_MC * Q; e += WG_WARPS * 32) {
        const int r = e / Q, c = 8 * (e - r * Q);
        if (r < cnt)
            net_cp16(s + r * LDS + c, src + (m0 + r) * LDG + c0 + c);
        else
            *reinterpret_cast<uint4*>(s + r * LDS + c) = make_uint4(0u, 0u, 0u, 0u);
    }
}
// the same from FP32, rounded here
template <int C, int LDG, int LDS>
__device__ __forceinline__ void wg_stage(__nv_bfloat16* s, const float* __restrict__ src, int c0, int64_t m0, int cnt) {
    constexpr int Q = C / 4;
#pragma unroll
    for (int e = threadIdx.x; e < WG_MC * Q; e += WG_WARPS * 32) {
        const int r = e / Q, c = 4 * (e - r * Q);
        uint2 v = make_uint2(0u, 0u);
        if (r < cnt) {
            const float4 f = *reinterpret_cast<const float4*>(src + (m0 + r) * LDG + c0 + c);
            v = make_uint2(pack_bf16(f.x, f.y), pack_bf16(f.z, f.w));
        }
        *reinterpret_cast<uint2*>(s + r * LDS + c) = v;
    }
}
// the warp's tile of MT m16 (all of the slab) x 2 n8 outputs, k columns from kc
template <int MT>
__device__ __forceinline__ void wg_tile(const __nv_bfloat16* sD, const __nv_bfloat16* sX, int kc, int lane,
                                        float (&sum)[2][2][4]) {
    const int r = lane & 7, s1 = (lane >> 3) & 1, s2 = lane >> 4;
    float acc[MT][2][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][n][e] = 0.f;
#pragma unroll 4
    for (int mm = 0; mm < WG_MC; mm += 16) {
        uint32_t b[4];
        ldmatrix_t(b, sX + (mm + r + 8 * s1) * WG_LDX + kc + 8 * s2);
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            uint32_t a[4];
            ldmatrix_t(a, sD + (mm + r + 8 * s2) * WG_LDD + 16 * i + 8 * s1);
            mma_bf16(acc[i][0], a[0], a[1], a[2], a[3], b[0], b[1]);
            mma_bf16(acc[i][1], a[0], a[1], a[2], a[3], b[2], b[3]);
        }
    }
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) sum[i][n][e] += acc[i][n][e];
}
__device__ __forceinline__ void wg_red2(float* p, float x, float y) {
    asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(x), "f"(y) : "memory");
}
// G[n] = sum_m D[m][n] for the eight columns from n0, by the block: 256 partial sums over the rows
// r, r + 256, ..., a butterfly over each 32 of them, then the eight in order
__device__ __forceinline__ void wg_colsum8(float* s, int64_t M, int N, int n0, const float* __restrict__ D,
                                           float* __restrict__ G) {
    const int r = threadIdx.x >> 3, c = threadIdx.x & 7, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = 0.f;
    const float* p = D + n0 + c;
    int64_t m0 = 0;
#pragma unroll 2
    for (; m0 + 256 <= M; m0 += 256)
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] += p[(m0 + 32 * k + r) * N];
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (m0 + 32 * k + r < M) v[k] += p[(m0 + 32 * k + r) * N];
#pragma unroll
    for (int k = 0; k < 8; ++k) s[(k * 8 + c) * 33 + r] = v[k];
    __syncthreads();
    float mine = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {  // the warp adds up its 32 partial sums of column q
        float x = s[(warp * 8 + q) * 33 + lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == q) mine = x;
    }
    __syncthreads();
    if (lane < 8) s[warp * 8 + lane] = mine;
    __syncthreads();
    if (threadIdx.x < 8) {
        float tot = 0.f;
        for (int w = 0; w < 8; ++w) tot += s[w * 8 + threadIdx.x];
        G[n0 + threadIdx.x] = tot;
    }
    __syncthreads();
}
template <bool KEEP>
__global__ void __launch_bounds__(WG_WARPS * 32, 2)
    k_mlp_wgrad(int64_t M, int64_t rows, const float* __restrict__ X, const StepOut in) {
    pdl_begin();
    extern __shared__ __align__(16) unsigned char wg_raw[];
    const int job = blockIdx.y;
    if (job >= WG_WJOBS) {
        constexpr int NG = (2 * MLP_H + MLP_S) / 8;
        for (int q = (job - WG_WJOBS) * gridDim.x + blockIdx.x; q < NG; q += (WG_JOBS - WG_WJOBS) * gridDim.x) {
            float* s = reinterpret_cast<float*>(wg_raw);
            if (q < MLP_H / 8)
                wg_colsum8(s, M, MLP_H, 8 * q, in.F1, in.G + OFF_B1);
            else if (q < 2 * MLP_H / 8)
                wg_colsum8(s, M, MLP_H, 8 * q - MLP_H, in.F2, in.G + OFF_B2);
            else
                wg_colsum8(s, M, MLP_S, 8 * q - 2 * MLP_H, in.F3, in.G + OFF_B3);
        }
        return;
    }
    __nv_bfloat16* sD = reinterpret_cast<__nv_bfloat16*>(wg_raw);
    __nv_bfloat16* sX = sD + WG_MC * WG_LDD;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, kc = 16 * warp;
    const int64_t m_begin = (int64_t)blockIdx.x * rows;
    const int64_t m_end = m_begin + rows < M ? m_begin + rows : M;
    const int K = job >= 4 && job < 8 ? MLP_F : MLP_H;
    float sum[2][2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) sum[i][n][e] = 0.f;
    for (int64_t m0 = m_begin; m0 < m_end; m0 += WG_MC) {
        const int cnt = (int)(m_end - m0 < WG_MC ? m_end - m0 : WG_MC);
        if (job < 4) {
            if constexpr (KEEP) wg_stage<32, MLP_H, WG_LDD>(sD, in.D2, 32 * job, m0, cnt);
            else wg_stage<32, MLP_H, WG_LDD>(sD, in.F2, 32 * job, m0, cnt);
            wg_stage<MLP_H, MLP_H, WG_LDX>(sX, in.H1, 0, m0, cnt);
        } else if (job < 8) {
            if constexpr (KEEP) wg_stage<32, MLP_H, WG_LDD>(sD, in.D1, 32 * (job - 4), m0, cnt);
            else wg_stage<32, MLP_H, WG_LDD>(sD, in.F1, 32 * (job - 4), m0, cnt);
            constexpr int Q = MLP_F / 2;
#pragma unroll 14
            for (int e = threadIdx.x; e < WG_MC * Q; e += WG_WARPS * 32) {
                const int r = e / Q, c = 2 * (e - r * Q);
                *reinterpret_cast<uint32_t*>(sX + r * WG_LDX + c) = r < cnt ? load_pair(X + (m0 + r) * MLP_F + c) : 0u;
            }
        } else {
            if constexpr (KEEP) wg_stage<MLP_S, MLP_S, WG_LDD>(sD, in.D3, 0, m0, cnt);
            else wg_stage<MLP_S, MLP_S, WG_LDD>(sD, in.F3, 0, m0, cnt);
            wg_stage<MLP_H, MLP_H, WG_LDX>(sX, in.H2, 0, m0, cnt);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (kc < K) {
            if (job < 8)
                wg_tile<2>(sD, sX, kc, lane, sum);
            else
                wg_tile<1>(sD, sX, kc, lane, sum);
        }
        __syncthreads();
    }
    if (kc >= K) return;
    float* G = in.G + (job < 4 ? OFF_W2 + (int64_t)32 * job * MLP_H : job < 8 ? OFF_W1 + (int64_t)32 * (job - 4) * MLP_F : OFF_W3);
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (i == 0 || job < 8)
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                float* p = G + (16 * i + g) * K + kc + 8 * n + 2 * t;
                wg_red2(p, sum[i][n][0], sum[i][n][1]);
                wg_red2(p + 8 * K, sum[i][n][2], sum[i][n][3]);
            }
}

// Adam (bias-corrected), then the bf16 copy of the weights; G is cleared for the next batch.
__global__ void k_adam(float* __restrict__ P, float* __restrict__ G, float* __restrict__ Mo,
                       float* __restrict__ Vo, __nv_bfloat16* __restrict__ Wb, float lr, float c1, float c2) {
    pdl_begin();
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= NPARAM) return;
    const float g = G[q];
    G[q] = 0.f;
    const float m = 0.9f * Mo[q] + 0.1f * g;
    const float v = 0.999f * Vo[q] + 0.001f * g * g;
    Mo[q] = m;
    Vo[q] = v;
    const float p = P[q] - lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
    P[q] = p;
    const int64_t b = bf_index(q);
    if (b >= 0) Wb[b] = __float2bfloat16_rn(p);
}

// ------------------------------------------------------------------ the model object
struct Model {
    DevBuf<float> P, G, Mo, Vo;
    DevBuf<__nv_bfloat16> Wb;
    int t = 0;
};

Model* mlp_create(uint64_t seed, cudaStream_t s) {
    AllocStream as_(s);
    auto* m = new Model();
    m->P.alloc(NPARAM);
    m->G.alloc(NPARAM);
    m->Mo.alloc(NPARAM);
    m->Vo.alloc(NPARAM);
    m->Wb.alloc(NBF);
    BAMG_CK(cudaMemsetAsync(m->Wb.get(), 0, sizeof(__nv_bfloat16) * NBF, s));  // the rows' padding
    BAMG_LAUNCH(k_mlp_init, blocks_for(NPARAM, 256), 256, 0, s, seed, m->P.get());
    BAMG_LAUNCH(k_mlp_to_bf16, blocks_for(NPARAM, 256), 256, 0, s, m->P.get(), m->Wb.get());
    BAMG_CK(cudaMemsetAsync(m->Mo.get(), 0, sizeof(float) * NPARAM, s));
    BAMG_CK(cudaMemsetAsync(m->Vo.get(), 0, sizeof(float) * NPARAM, s));
    return m;
}
void mlp_destroy(Model* m) { delete m; }

void mlp_set(Model* m, const float* h_params, cudaStream_t s) {
    BAMG_CK(cudaMemcpyAsync(m->P.get(), h_params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, s));
    BAMG_LAUNCH(k_mlp_to_bf16, blocks_for(NPARAM, 256), 256, 0, s, m->P.get(), m->Wb.get());
    BAMG_CK(cudaMemsetAsync(m->Mo.get(), 0, sizeof(float) * NPARAM, s));
    BAMG_CK(cudaMemsetAsync(m->Vo.get(), 0, sizeof(float) * NPARAM, s));
    m->t = 0;
}
void mlp_get(const Model* m, float* h_params, cudaStream_t s) {
    BAMG_CK(cudaMemcpyAsync(h_params, m->P.get(), sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, s));
    BAMG_CK(cudaStreamSynchronize(s));
}

// Activations and gradients (rounded and not) of one batch of rows, and the loss sum: 2144 bytes a row up to
// KEEP_ROWS (0.6 GB).  A larger batch leaves the rounded gradients out, 1600 bytes a row, and k_mlp_wgrad
// rounds the others as it reads them: the same bits, and no more traffic (what the step kernel does not
// write, k_mlp_wgrad reads).  4,000,000 rows took 8160 MiB and 21.6 ms with them, 6080 MiB and 20.3 ms without;
// 262,145 rows 1.19 ms and 1.09.  (Slices of 262,144 rows instead: 600 MiB, but 25.1 ms.)
constexpr int64_t KEEP_ROWS = 1 << 18;
struct MlpWork {
    DevBuf<__nv_bfloat16> H1, H2, D1, D2, D3;
    DevBuf<float> F1, F2, F3;
    DevBuf<double> loss;
    bool keep;  // the rounded gradients have a place of their own
    explicit MlpWork(int64_t rows) : keep(rows <= KEEP_ROWS) {
        H1.alloc(rows * MLP_H);
        H2.alloc(rows * MLP_H);
        if (keep) {
            D1.alloc(rows * MLP_H);
            D2.alloc(rows * MLP_H);
            D3.alloc(rows * MLP_S);
        }
        F1.alloc(rows * MLP_H);
        F2.alloc(rows * MLP_H);
        F3.alloc(rows * MLP_S);
        loss.alloc(1);
    }
};

// Dynamic shared memory beyond 48 KB for a kernel, allowed once per device (idempotent across
// threads); returns the device's SM count.
template <typename K>
static int net_device(K kernel, size_t smem, std::atomic<bool> (&allowed)[256]) {
    int dev = 0, nsm = 0;
    BAMG_CK(cudaGetDevice(&dev));
    BAMG_REQUIRE(dev >= 0 && dev < 256, BAMG_EINVAL, "device ordinal out of range");
    if (!allowed[dev]) {
        BAMG_CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        allowed[dev] = true;
    }
    BAMG_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    return nsm > 0 ? nsm : 1;
}
// k_mlp_net: weights and one feature tile a warp
constexpr size_t NET_BYTES = sizeof(NetSmem) + sizeof(float) * NET_WARPS * 16 * NET_LDX;
static_assert(NET_BYTES <= 227 * 1024, "shared memory");

void mlp_forward(const Model* m, int64_t rows, const float* feat, float* Y, cudaStream_t s) {
    if (rows <= 0) return;
    static std::atomic<bool> allowed[256] = {};
    const int nsm = net_device(k_mlp_net, NET_BYTES, allowed);
    BAMG_LAUNCH(k_mlp_net, (unsigned)std::min<int64_t>(nsm, (rows + 15) / 16), NET_WARPS * 32, NET_BYTES, s, rows,
                feat, (const __nv_bfloat16*)m->Wb.get(), (const float*)m->P.get(), Y);
}

// Gradients of the batch loss added to m->G; the loss sum into w.loss.
template <bool KEEP>
static void gradients_as(Model* m, int64_t rows, const float* feat, const float* target, MlpWork& w, bool early,
                         cudaStream_t s) {
    static std::atomic<bool> allowed[256] = {}, allowed_w[256] = {};
    const int nsm = net_device(k_mlp_step<KEEP>, sizeof(StepSmem), allowed);
    net_device(k_mlp_wgrad<KEEP>, WG_SMEM, allowed_w);
    const StepOut out{w.H1.get(), w.H2.get(), w.D1.get(), w.D2.get(), w.D3.get(),
                      w.F1.get(), w.F2.get(), w.F3.get(), m->G.get(), w.loss.get()};
    BAMG_LAUNCH(k_mlp_step<KEEP>, (unsigned)std::min<int64_t>(nsm, (rows + 15) / 16), STEP_WARPS * 32, sizeof(StepSmem),
                s, rows, feat, target, (const __nv_bfloat16*)m->Wb.get(), (const float*)m->P.get(), out, early);
    // up to two blocks per SM over the jobs, in whole chunks of rows
    const int64_t chunks = (rows + WG_MC - 1) / WG_MC, per = (chunks * WG_JOBS + 2 * nsm - 1) / (2 * nsm);
    const int64_t br = per * WG_MC;
    BAMG_LAUNCH(k_mlp_wgrad<KEEP>, dim3((unsigned)((rows + br - 1) / br), WG_JOBS), WG_WARPS * 32, WG_SMEM, s, rows, br,
                feat, out);
}
static void gradients(Model* m, int64_t rows, const float* feat, const float* target, MlpWork& w, bool early,
                      cudaStream_t s) {
    (w.keep ? gradients_as<true> : gradients_as<false>)(m, rows, feat, target, w, early, s);
}

double mlp_gradients(Model* m, int64_t rows, const float* feat, const float* target, float* h_grad, cudaStream_t s) {
    BAMG_REQUIRE(rows > 0, BAMG_EINVAL, "mlp_gradients: no rows");
    AllocStream as_(s);
    MlpWork w(rows);
    BAMG_CK(cudaMemsetAsync(w.loss.get(), 0, sizeof(double), s));
    BAMG_CK(cudaMemsetAsync(m->G.get(), 0, sizeof(float) * NPARAM, s));
    gradients(m, rows, feat, target, w, false, s);
    double l = 0.0;
    BAMG_CK(cudaMemcpyAsync(&l, w.loss.get(), sizeof(double), cudaMemcpyDeviceToHost, s));
    if (h_grad) BAMG_CK(cudaMemcpyAsync(h_grad, m->G.get(), sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, s));
    BAMG_CK(cudaStreamSynchronize(s));
    return l;
}

void mlp_train(Model* m, int64_t rows, const float* feat, const float* target, int epochs, int batch, double lr,
               double* h_loss, cudaStream_t s) {
    BAMG_REQUIRE(rows > 0 && epochs >= 0 && batch > 0, BAMG_EINVAL, "mlp_train: bad sizes");
    AllocStream as_(s);
    MlpWork w(std::min<int64_t>(rows, batch));
    BAMG_CK(cudaMemsetAsync(m->G.get(), 0, sizeof(float) * NPARAM, s));
    for (int e = 0; e < epochs; ++e) {
        BAMG_CK(cudaMemsetAsync(w.loss.get(), 0, sizeof(double), s));
        int64_t nb = 0;
        for (int64_t r0 = 0; r0 < rows; r0 += batch, ++nb) {
            const int64_t br = std::min<int64_t>(batch, rows - r0);
            gradients(m, br, feat + r0 * MLP_F, target + r0 * MLP_S, w, e > 0 || r0 > 0, s);
            m->t += 1;
            const float c1 = (float)(1.0 - std::pow(0.9, m->t)), c2 = (float)(1.0 - std::pow(0.999, m->t));
            BAMG_LAUNCH(k_adam, blocks_for(NPARAM, 256), 256, 0, s, m->P.get(), m->G.get(),
                        m->Mo.get(), m->Vo.get(), m->Wb.get(), (float)lr, c1, c2);
        }
        if (h_loss) {
            double l = 0.0;
            BAMG_CK(cudaMemcpyAsync(&l, w.loss.get(), sizeof(double), cudaMemcpyDeviceToHost, s));
            BAMG_CK(cudaStreamSynchronize(s));
            h_loss[e] = l / (double)nb;  // mean of the batch losses
        }
    }
    BAMG_CK(cudaStreamSynchronize(s));
}

}  // namespace bamg
