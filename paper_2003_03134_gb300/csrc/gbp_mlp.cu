// gbp_mlp.cu -- training of the per-factor damping network on BF16 tensor
// cores (forward and backward GEMMs with mma.sync m16n8k16, FP32
// accumulation), FP32 master weights and Adam (Kingma and Ba 2015), and the
// C ABI of the gbp_mlp object.
//
// One training step over a batch of B samples:
//   mlp_grad_kernel    one warp (a block) per 32 samples: forward, backward,
//                      this warp's partial gradient and loss;
//   mlp_reduce_kernel  the partials added in a fixed order (deterministic),
//                      then optionally Adam and the new weights' BF16
//                      B-operand fragments.
// mlp_pack_kernel packs the fragments and FP32 biases from master weights set
// by the caller.
#include "gbp_mlp.cuh"
#include "gbp_internal.h"
#include "../../include/gbp.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

namespace gbp {

static_assert(MLP_NPARAM == GBP_MLP_NPARAM && MLP_IN == GBP_MLP_NFEAT, "parameter layout");

constexpr int MLP_BLOCK = 128;               // samples per block
constexpr int MLP_WARPS = MLP_BLOCK / 32;
constexpr int GRAD_WAVE = 2048;              // warps of mlp_grad_kernel that run at once (14 on each of 152 SMs, rounded down)
constexpr int MLP_PART = MLP_NPARAM + 3;     // a warp's partial gradient, its loss, pad to an even count (8-byte rows)
static_assert(MLP_PART % 2 == 0, "float2 stores");

// ------------------------------------------------------------------------
// packing: fragment tile t, lane l holds B[2q..2q+1][g] and B[2q+8..2q+9][g]
// of the tile's 16 x 8 sub-matrix of B (K x N).

__device__ __forceinline__ float mlp_b_elem(const float* W, int t, int k, int n) {
    if (t < FT_L2) return W[MLP_OFF_W1 + k * MLP_H + 8 * t + n];                 // W1[k][n]
    if (t < FT_L3) {
        const int ks = (t - FT_L2) / 8, nt = (t - FT_L2) % 8;
        return W[MLP_OFF_W2 + (16 * ks + k) * MLP_H + 8 * nt + n];               // W2[k][n]
    }
    if (t < FT_W2T) {
        const int ks = t - FT_L3;
        return n == 0 ? W[MLP_OFF_W3 + 16 * ks + k] : 0.0f;                      // W3 in column 0
    }
    const int ks = (t - FT_W2T) / 8, nt = (t - FT_W2T) % 8;
    return W[MLP_OFF_W2 + (8 * nt + n) * MLP_H + 16 * ks + k];                   // W2^T[k][n]
}

__global__ void mlp_pack_kernel(const float* __restrict__ W, uint32_t* __restrict__ frag, float* __restrict__ bias) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < FT_N * 32) {
        const int t = i / 32, lane = i % 32, g = lane >> 2, q = lane & 3;
        frag[2 * i] = pack_bf16(mlp_b_elem(W, t, 2 * q, g), mlp_b_elem(W, t, 2 * q + 1, g));
        frag[2 * i + 1] = pack_bf16(mlp_b_elem(W, t, 2 * q + 8, g), mlp_b_elem(W, t, 2 * q + 9, g));
    }
    if (i < MLP_H) {
        bias[i] = W[MLP_OFF_B1 + i];
        bias[MLP_H + i] = W[MLP_OFF_B2 + i];
        bias[2 * MLP_H + 2 + i] = W[MLP_OFF_W3 + i];   // W3 in FP32 for the backward pass
    }
    if (i == 0) bias[2 * MLP_H] = W[MLP_OFF_B3];
}


// ------------------------------------------------------------------------
// forward over samples (inference)
//
// A warp walks 16-row tiles with every weight in registers: the 44 B-operand
// fragments are 88 registers a lane, loaded once per warp, and the
// activations stay in registers between the layers (mlp_forward_regs' scheme,
// the same roundings and the same mma order, so the same bits).  Rows are
// read straight into A fragments: a lane's four float2 cover whole 32-byte
// sectors over the warp, and the next tile's are in flight while this one is
// evaluated.  Shared memory holds only the biases.  4 million rows: 129 us
// (the mma pipe 60 % busy, which 4 or 5 blocks per SM with part of the
// weights in shared memory do not raise: 137-139 us), 340 us for a block per
// 128 rows that copied the weights to shared memory first and kept the
// activations there (its shared-memory pipe was 94 % busy); reading the rows
// once takes 40 us.

// relu of a rounded BF16 pair (rounding keeps the sign, so relu may follow it:
// one packed maximum for two); a NaN becomes 0
__device__ __forceinline__ uint32_t pack_relu(float lo, float hi) {
    uint32_t v = pack_bf16(lo, hi);
    asm("max.bf16x2 %0, %0, %1;" : "+r"(v) : "r"(0u));
    return v;
}

// A fragment of rows [r0, r0 + 16) of X; rows past n read as zero.
template <bool PAIRS>
__device__ __forceinline__ void load_rows(const float* __restrict__ X, int n, int r0, int lane, float2 (&v)[4]) {
    const int g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int r = r0 + g + 8 * (h & 1);
        const float* p = X + (size_t)r * MLP_IN + 2 * q + 8 * (h >> 1);
        if (r >= n) v[h] = make_float2(0.f, 0.f);
        else if constexpr (PAIRS) v[h] = __ldcs(reinterpret_cast<const float2*>(p));
        else v[h] = make_float2(p[0], p[1]);
    }
}

template <bool PAIRS>
__global__ void __launch_bounds__(MLP_BLOCK, 3) mlp_forward_kernel(const uint32_t* __restrict__ frag_g,
                                                                   const float* __restrict__ bias_g,
                                                                   const float* __restrict__ X, int n,
                                                                   float* __restrict__ y) {
    __shared__ __align__(16) float bias[MLP_BIAS_WORDS];
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int n_tiles = (n + 15) / 16, stride = gridDim.x * MLP_WARPS;
    int tile = blockIdx.x * MLP_WARPS + (threadIdx.x >> 5);
    float2 v[4];
    load_rows<PAIRS>(X, n, tile < n_tiles ? 16 * tile : n, lane, v);
    uint2 w[FT_W2T];
#pragma unroll
    for (int t = 0; t < FT_W2T; ++t) w[t] = reinterpret_cast<const uint2*>(frag_g)[t * 32 + lane];
    for (int i = threadIdx.x; i < MLP_BIAS_WORDS; i += MLP_BLOCK) bias[i] = bias_g[i];
    __syncthreads();
    for (; tile < n_tiles; tile += stride) {
        const uint32_t x0 = pack_bf16(v[0].x, v[0].y), x1 = pack_bf16(v[1].x, v[1].y);
        const uint32_t x2 = pack_bf16(v[2].x, v[2].y), x3 = pack_bf16(v[3].x, v[3].y);
        load_rows<PAIRS>(X, n, tile + stride < n_tiles ? 16 * (tile + stride) : n, lane, v);
        uint32_t a[4][4];
        float d[8][4];
        // layer 1: h1 = relu(X W1 + b1) -> A fragments of layer 2
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
            mma_bf16(d[nt], x0, x1, x2, x3, w[FT_L1 + nt].x, w[FT_L1 + nt].y);
        }
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const float2 b = *reinterpret_cast<const float2*>(bias + 8 * nt + 2 * q);
            a[nt >> 1][(nt & 1) ? 2 : 0] = pack_relu(d[nt][0] + b.x, d[nt][1] + b.y);
            a[nt >> 1][(nt & 1) ? 3 : 1] = pack_relu(d[nt][2] + b.x, d[nt][3] + b.y);
        }
        // layer 2: h2 = relu(h1 W2 + b2) -> A fragments of layer 3
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int nt = 0; nt < 8; ++nt)
                mma_bf16(d[nt], a[ks][0], a[ks][1], a[ks][2], a[ks][3], w[FT_L2 + ks * 8 + nt].x,
                         w[FT_L2 + ks * 8 + nt].y);
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const float2 b = *reinterpret_cast<const float2*>(bias + MLP_H + 8 * nt + 2 * q);
            a[nt >> 1][(nt & 1) ? 2 : 0] = pack_relu(d[nt][0] + b.x, d[nt][1] + b.y);
            a[nt >> 1][(nt & 1) ? 3 : 1] = pack_relu(d[nt][2] + b.x, d[nt][3] + b.y);
        }
        // layer 3: z3 = h2 W3 + b3 (column 0 of the output tile: lanes with q = 0)
        float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
            mma_bf16(z, a[ks][0], a[ks][1], a[ks][2], a[ks][3], w[FT_L3 + ks].x, w[FT_L3 + ks].y);
        if (q == 0) {
            const int r = 16 * tile + g;
            const float b3 = bias[2 * MLP_H];
            if (r < n) y[r] = mlp_output(z[0] + b3);
            if (r + 8 < n) y[r + 8] = mlp_output(z[2] + b3);
        }
    }
}

// ------------------------------------------------------------------------
// forward + backward of a minibatch: one warp per block, 32 samples
//
// A training minibatch is 4096 rows, so the step is a latency chain, not a
// throughput problem: a warp per 32 rows spreads it over 128 blocks (a block
// of 4 warps left 120 SMs idle).  Weights are read from L2 as B fragments by
// the warp that uses them (each once: 76 loads in flight at will), with no
// copy to shared memory; the activations and dz2 stay in registers as the A
// fragments of the next product, and go to shared memory only for the
// products over samples (dW2 = h1^T dz2, dW1 = x^T dz1), whose transposed
// operands ldmatrix.trans reads 8 x 8 blocks at a time.  Each warp writes its
// own partial gradient; mlp_reduce_kernel adds them.
//
// GROUPED (more rows than one wave of warps takes): a warp works the four 32s
// of 128 samples and adds them up in its partial, in the same order, so the
// partials take no more memory than one per 128 samples.
//
// A step at 4096 rows: 11.3 us for both launches (30.6 us with 32 blocks of 4
// warps, shared-memory weights and accumulators, and a third launch to pack).

struct GradSmem {
    alignas(16) __nv_bfloat16 x[32 * XS];
    alignas(16) __nv_bfloat16 h1[32 * HS];
    alignas(16) __nv_bfloat16 h2[32 * HS];   // h2, later dz1
    alignas(16) __nv_bfloat16 dz[32 * HS];   // dz2
    float dz3[32];
};

// four transposed 8 x 8 blocks; lane l gives the address of row l % 8 of block l / 8
__device__ __forceinline__ void ldmatrix_t(const __nv_bfloat16* p, uint32_t (&r)[4]) {
    const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}

__device__ __forceinline__ uint2 load_frag(const uint32_t* __restrict__ frag, int tile, int lane) {
    return *reinterpret_cast<const uint2*>(frag + (tile * 32 + lane) * 2);
}

// a value kept where the activation it belongs to (a BF16 half) is positive
__device__ __forceinline__ float where_pos(uint32_t h, bool upper, float v) {
    const uint32_t b = upper ? h >> 16 : h & 0xffffu;
    return b - 1u < 0x7f80u ? v : 0.f;   // (0, inf] by its bits
}

__device__ __forceinline__ void pdl_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// a warp's (or group's) partial: stored by its first 32 samples, added to by
// the others
__device__ __forceinline__ void put2(float* o, bool first, float a, float b) {
    if (!first) {
        const float2 v = *reinterpret_cast<const float2*>(o);
        a = v.x + a;
        b = v.y + b;
    }
    *reinterpret_cast<float2*>(o) = make_float2(a, b);
}
__device__ __forceinline__ void put1(float* o, bool first, float a) { *o = first ? a : *o + a; }

template <bool GROUPED>
__global__ void __launch_bounds__(32) mlp_grad_kernel(const uint32_t* __restrict__ frag, const float* __restrict__ bias,
                                                      const float* __restrict__ X, const float* __restrict__ T,
                                                      const int32_t* __restrict__ idx, int n, float inv_batch,
                                                      float* __restrict__ partials) {
    __shared__ GradSmem S;
    const int lane = threadIdx.x, g = lane >> 2, q = lane & 3;
    pdl_wait_previous();
    for (int sub = 0; sub < (GROUPED ? 4 : 1); ++sub) {
    const int si = (GROUPED ? 4 * int(blockIdx.x) + sub : int(blockIdx.x)) * 32 + lane;   // this lane's sample slot
    const bool valid = si < n;
    const int sample = valid ? (idx ? idx[si] : si) : 0;
    const bool first = !GROUPED || sub == 0;
    if (GROUPED) __syncwarp();   // the tiles are rewritten
    {
        float x[MLP_IN];
        const float* row = X + (size_t)sample * MLP_IN;
        if (!valid) {
#pragma unroll
            for (int j = 0; j < MLP_IN; ++j) x[j] = 0.f;
        } else if (reinterpret_cast<uintptr_t>(X) % 16 == 0) {
#pragma unroll
            for (int j = 0; j < MLP_IN / 4; ++j) {
                const float4 v = reinterpret_cast<const float4*>(row)[j];
                x[4 * j] = v.x; x[4 * j + 1] = v.y; x[4 * j + 2] = v.z; x[4 * j + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < MLP_IN; ++j) x[j] = row[j];
        }
        uint32_t p[MLP_IN / 2];
#pragma unroll
        for (int j = 0; j < MLP_IN / 2; ++j) p[j] = pack_bf16(x[2 * j], x[2 * j + 1]);
        uint4* out = reinterpret_cast<uint4*>(S.x + lane * XS);
        out[0] = make_uint4(p[0], p[1], p[2], p[3]);
        out[1] = make_uint4(p[4], p[5], p[6], p[7]);
    }
    const float target = valid ? T[sample] : 0.f;
    __syncwarp();

    // forward: h1, h2 as A fragments of the next layer and as rows in shared memory
    uint32_t a1[2][4][4], a2[2][4][4];
    {
        uint32_t x0[4], x1[4];
        load_a(S.x, XS, 0, 0, lane, x0[0], x0[1], x0[2], x0[3]);
        load_a(S.x, XS, 16, 0, lane, x1[0], x1[1], x1[2], x1[3]);
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const uint2 w = load_frag(frag, FT_L1 + nt, lane);
            const float b0 = bias[8 * nt + 2 * q], b1 = bias[8 * nt + 2 * q + 1];
            float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(d0, x0[0], x0[1], x0[2], x0[3], w.x, w.y);
            mma_bf16(d1, x1[0], x1[1], x1[2], x1[3], w.x, w.y);
            const int ks = nt >> 1, o = (nt & 1) * 2;
            a1[0][ks][o] = pack_relu(d0[0] + b0, d0[1] + b1);
            a1[0][ks][o + 1] = pack_relu(d0[2] + b0, d0[3] + b1);
            a1[1][ks][o] = pack_relu(d1[0] + b0, d1[1] + b1);
            a1[1][ks][o + 1] = pack_relu(d1[2] + b0, d1[3] + b1);
        }
    }
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const float b0 = bias[MLP_H + 8 * nt + 2 * q], b1 = bias[MLP_H + 8 * nt + 2 * q + 1];
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            const uint2 w = load_frag(frag, FT_L2 + ks * 8 + nt, lane);
            mma_bf16(d0, a1[0][ks][0], a1[0][ks][1], a1[0][ks][2], a1[0][ks][3], w.x, w.y);
            mma_bf16(d1, a1[1][ks][0], a1[1][ks][1], a1[1][ks][2], a1[1][ks][3], w.x, w.y);
        }
        const int ks = nt >> 1, o = (nt & 1) * 2;
        a2[0][ks][o] = pack_relu(d0[0] + b0, d0[1] + b1);
        a2[0][ks][o + 1] = pack_relu(d0[2] + b0, d0[3] + b1);
        a2[1][ks][o] = pack_relu(d1[0] + b0, d1[1] + b1);
        a2[1][ks][o + 1] = pack_relu(d1[2] + b0, d1[3] + b1);
    }
    float z[2][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) z[mt][0] = z[mt][1] = z[mt][2] = z[mt][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        const uint2 w = load_frag(frag, FT_L3 + ks, lane);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) mma_bf16(z[mt], a2[mt][ks][0], a2[mt][ks][1], a2[mt][ks][2], a2[mt][ks][3], w.x, w.y);
    }
    // row r = lane of column 0: held by lane 4 (r % 8) of m-tile r / 16
    float z3;
    {
        const int src = (lane & 7) << 2;
        const float v00 = __shfl_sync(0xffffffffu, z[0][0], src), v01 = __shfl_sync(0xffffffffu, z[0][2], src);
        const float v10 = __shfl_sync(0xffffffffu, z[1][0], src), v11 = __shfl_sync(0xffffffffu, z[1][2], src);
        z3 = ((lane < 16) ? ((lane & 8) ? v01 : v00) : ((lane & 8) ? v11 : v10)) + bias[2 * MLP_H];
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int at = (16 * mt + g + 8 * (h & 1)) * HS + 16 * ks + 2 * q + 8 * (h >> 1);
                *reinterpret_cast<uint32_t*>(S.h1 + at) = a1[mt][ks][h];
                *reinterpret_cast<uint32_t*>(S.h2 + at) = a2[mt][ks][h];
            }
    const float sg = 1.0f / (1.0f + __expf(-z3));
    const float y = MLP_DMAX * sg;
    const float r = valid ? y - target : 0.f;
    // loss = mean r^2 ; dL/dz3 = 2 r / B * 0.9 s (1 - s)
    const float dz3 = 2.0f * r * inv_batch * MLP_DMAX * sg * (1.0f - sg);
    S.dz3[lane] = dz3;
    float r2 = r * r * inv_batch;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_down_sync(0xffffffffu, r2, o);
    float pb3 = dz3;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pb3 += __shfl_down_sync(0xffffffffu, pb3, o);

    // dz2[s][j] = dz3[s] W3[j] [h2 > 0] in h2's fragment positions (in place of it), as BF16
    const float* W3 = bias + 2 * MLP_H + 2;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        const float r0 = __shfl_sync(0xffffffffu, dz3, 16 * mt + g), r1 = __shfl_sync(0xffffffffu, dz3, 16 * mt + g + 8);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int c = 16 * ks + 2 * q + 8 * (h >> 1);
                const float d = (h & 1) ? r1 : r0;
                const uint32_t v = pack_bf16(where_pos(a2[mt][ks][h], false, d * W3[c]),
                                             where_pos(a2[mt][ks][h], true, d * W3[c + 1]));
                a2[mt][ks][h] = v;
                *reinterpret_cast<uint32_t*>(S.dz + (16 * mt + g + 8 * (h & 1)) * HS + c) = v;
            }
    }
    __syncwarp();
    // vector partials: dW3[j] = sum_s h2[s][j] dz3[s], db2[j] = sum_s dz2[s][j],
    // db3 = sum_s dz3[s], in sample order (lane takes j = 2 lane, 2 lane + 1)
    float pW3[2] = {0.f, 0.f}, pb2[2] = {0.f, 0.f};
#pragma unroll 8
    for (int s = 0; s < 32; ++s) {
        const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(S.h2 + s * HS + 2 * lane);
        const __nv_bfloat162 d = *reinterpret_cast<const __nv_bfloat162*>(S.dz + s * HS + 2 * lane);
        const float ds = S.dz3[s];
        pW3[0] = fmaf(__bfloat162float(h.x), ds, pW3[0]);
        pW3[1] = fmaf(__bfloat162float(h.y), ds, pW3[1]);
        pb2[0] += __bfloat162float(d.x);
        pb2[1] += __bfloat162float(d.y);
    }
    __syncwarp();

    // dh1 = dz2 W2^T ; dz1 = dh1 [h1 > 0]  -> BF16 into the h2 tile
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        float d[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) d[mt][0] = d[mt][1] = d[mt][2] = d[mt][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            const uint2 w = load_frag(frag, FT_W2T + ks * 8 + nt, lane);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
                mma_bf16(d[mt], a2[mt][ks][0], a2[mt][ks][1], a2[mt][ks][2], a2[mt][ks][3], w.x, w.y);
        }
        // the ReLU mask of layer 1: h1 fragment (nt >> 1) holds columns 8 nt + 2q of both rows
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const uint32_t m0 = a1[mt][nt >> 1][(nt & 1) * 2], m1 = a1[mt][nt >> 1][(nt & 1) * 2 + 1];
            const int at = (16 * mt + g) * HS + 8 * nt + 2 * q;
            *reinterpret_cast<uint32_t*>(S.h2 + at) =
                pack_bf16(where_pos(m0, false, d[mt][0]), where_pos(m0, true, d[mt][1]));
            *reinterpret_cast<uint32_t*>(S.h2 + at + 8 * HS) =
                pack_bf16(where_pos(m1, false, d[mt][2]), where_pos(m1, true, d[mt][3]));
        }
    }
    __syncwarp();
    if (!GROUPED) pdl_launch_next();
    float pb1[2] = {0.f, 0.f};
#pragma unroll 8
    for (int s = 0; s < 32; ++s) {
        const __nv_bfloat162 d = *reinterpret_cast<const __nv_bfloat162*>(S.h2 + s * HS + 2 * lane);
        pb1[0] += __bfloat162float(d.x);
        pb1[1] += __bfloat162float(d.y);
    }

    // weight-gradient products over the 32 samples (K = samples): dW2 =
    // h1^T dz2 (64 x 64), dW1 = x^T dz1 (16 x 64), straight to this warp's
    // partial gradient in the flat parameter layout
    float* out = partials + (size_t)blockIdx.x * MLP_PART;
    const int lr = lane & 7, lb = lane >> 3;
    {
        uint32_t bz[2][8][2];   // B fragments of dz2: [k-step][n-tile]
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
            for (int nt = 0; nt < 8; nt += 2) {
                uint32_t v[4];
                ldmatrix_t(S.dz + (16 * ks + (lb & 1) * 8 + lr) * HS + 8 * (nt + (lb >> 1)), v);
                bz[ks][nt][0] = v[0]; bz[ks][nt][1] = v[1];
                bz[ks][nt + 1][0] = v[2]; bz[ks][nt + 1][1] = v[3];
            }
#pragma unroll
        for (int mt = 0; mt < 4; ++mt) {
            float d[8][4];
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                uint32_t a[4];   // rows of A = h1 units
                ldmatrix_t(S.h1 + (16 * ks + (lb >> 1) * 8 + lr) * HS + 16 * mt + (lb & 1) * 8, a);
#pragma unroll
                for (int nt = 0; nt < 8; ++nt) mma_bf16(d[nt], a[0], a[1], a[2], a[3], bz[ks][nt][0], bz[ks][nt][1]);
            }
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                float* o = out + MLP_OFF_W2 + (16 * mt + g) * MLP_H + 8 * nt + 2 * q;
                put2(o, first, d[nt][0], d[nt][1]);
                put2(o + 8 * MLP_H, first, d[nt][2], d[nt][3]);
            }
        }
    }
    {
        float d[8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
            uint32_t a[4];       // rows of A = input features
            ldmatrix_t(S.x + (16 * ks + (lb >> 1) * 8 + lr) * XS + (lb & 1) * 8, a);
#pragma unroll
            for (int nt = 0; nt < 8; nt += 2) {
                uint32_t v[4];
                ldmatrix_t(S.h2 + (16 * ks + (lb & 1) * 8 + lr) * HS + 8 * (nt + (lb >> 1)), v);
                mma_bf16(d[nt], a[0], a[1], a[2], a[3], v[0], v[1]);
                mma_bf16(d[nt + 1], a[0], a[1], a[2], a[3], v[2], v[3]);
            }
        }
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            float* o = out + MLP_OFF_W1 + g * MLP_H + 8 * nt + 2 * q;
            put2(o, first, d[nt][0], d[nt][1]);
            put2(o + 8 * MLP_H, first, d[nt][2], d[nt][3]);
        }
    }
    put2(out + MLP_OFF_B1 + 2 * lane, first, pb1[0], pb1[1]);
    put2(out + MLP_OFF_B2 + 2 * lane, first, pb2[0], pb2[1]);
    put2(out + MLP_OFF_W3 + 2 * lane, first, pW3[0], pW3[1]);
    if (lane == 0) {
        put1(out + MLP_OFF_B3, first, pb3);
        put1(out + MLP_NPARAM, first, r2);
    }
    }
}

// The updated parameter's places in the packed fragments and the side buffer
// (what mlp_pack_kernel writes for it).
__device__ __forceinline__ void pack_param(int p, float w, uint32_t* __restrict__ frag, float* __restrict__ bias) {
    auto put = [&](int tile, int k, int n) {   // element [k][n] of a 16 x 8 B tile
        const int word = (tile * 32 + n * 4 + ((k & 7) >> 1)) * 2 + (k >> 3);
        reinterpret_cast<__nv_bfloat16*>(frag)[2 * word + (k & 1)] = __float2bfloat16_rn(w);
    };
    if (p < MLP_OFF_B1) {
        const int k = p / MLP_H, n = p % MLP_H;
        put(FT_L1 + n / 8, k, n % 8);
    } else if (p < MLP_OFF_W2) {
        bias[p - MLP_OFF_B1] = w;
    } else if (p < MLP_OFF_B2) {
        const int k = (p - MLP_OFF_W2) / MLP_H, n = (p - MLP_OFF_W2) % MLP_H;
        put(FT_L2 + (k / 16) * 8 + n / 8, k % 16, n % 8);
        put(FT_W2T + (n / 16) * 8 + k / 8, n % 16, k % 8);
    } else if (p < MLP_OFF_W3) {
        bias[MLP_H + p - MLP_OFF_B2] = w;
    } else if (p < MLP_OFF_B3) {
        const int k = p - MLP_OFF_W3;
        put(FT_L3 + k / 16, k % 16, 0);
        bias[2 * MLP_H + 2 + k] = w;
    } else {
        bias[2 * MLP_H] = w;
    }
}

// Sum of the partials in a fixed order -- the four warps of each 128 samples
// first (PER = 4; PER = 1: the partials are these groups' already), then
// those sums in order -- and optionally an Adam step
// (step >= 1) with the packing of the new weights.  A block takes 32
// parameters; its 8 warps load RED_GROUPS groups of 128 samples at a time
// (16 loads of a lane in flight), one warp adds them up.  grad_out (nullable)
// receives the gradient, loss_out the loss.
constexpr int RED_WARPS = 8, RED_PER_WARP = 4, RED_GROUPS = RED_WARPS * RED_PER_WARP;

template <int PER>
__global__ void __launch_bounds__(RED_WARPS * 32) mlp_reduce_kernel(const float* __restrict__ partials, int n_part,
                                                                    float* __restrict__ W, float* __restrict__ m,
                                                                    float* __restrict__ v, int step, float lr,
                                                                    float* __restrict__ grad_out,
                                                                    float* __restrict__ loss_out,
                                                                    uint32_t* __restrict__ frag,
                                                                    float* __restrict__ bias) {
    __shared__ float part[2][RED_GROUPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    const bool mine = p <= MLP_NPARAM;
    const int n_groups = (n_part + PER - 1) / PER;
    pdl_wait_previous();
    // the optimiser's state is needed only after the sum: in flight with the partials
    float w0 = 0.f, m0 = 0.f, v0 = 0.f;
    if (warp == 0 && step > 0 && p < MLP_NPARAM) {
        w0 = W[p];
        m0 = m[p];
        v0 = v[p];
    }
    float gsum = 0.f;
    for (int g0 = 0, buf = 0; g0 < n_groups; g0 += RED_GROUPS, buf ^= 1) {
        float u[RED_PER_WARP][PER];
#pragma unroll
        for (int i = 0; i < RED_PER_WARP; ++i) {
            const int gr = g0 + warp + RED_WARPS * i;
#pragma unroll
            for (int j = 0; j < PER; ++j)
                u[i][j] = mine && PER * gr + j < n_part ? __ldcg(partials + (size_t)(PER * gr + j) * MLP_PART + p) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < RED_PER_WARP; ++i) {
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < PER; ++j) sum += u[i][j];
            part[buf][warp + RED_WARPS * i][lane] = sum;
        }
        __syncthreads();   // the other buffer is free once every warp has passed here
        if (warp == 0) {
            const int k = min(RED_GROUPS, n_groups - g0);
            if (k == RED_GROUPS) {
#pragma unroll
                for (int i = 0; i < RED_GROUPS; ++i) gsum += part[buf][i][lane];
            } else {
                for (int i = 0; i < k; ++i) gsum += part[buf][i][lane];
            }
        }
    }
    pdl_launch_next();
    if (warp != 0 || !mine) return;
    if (p == MLP_NPARAM) {
        if (loss_out) *loss_out = gsum;
        return;
    }
    if (grad_out) grad_out[p] = gsum;
    if (step > 0) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float mm = b1 * m0 + (1.f - b1) * gsum;
        const float vv = b2 * v0 + (1.f - b2) * gsum * gsum;
        m[p] = mm;
        v[p] = vv;
        const float mh = mm / (1.f - powf(b1, float(step)));
        const float vh = vv / (1.f - powf(b2, float(step)));
        const float w = w0 - lr * mh / (sqrtf(vh) + eps);
        W[p] = w;
        pack_param(p, w, frag, bias);
    }
}

}  // namespace gbp

// ==========================================================================
// C ABI

using namespace gbp;

struct gbp_mlp {
    cudaStream_t stream = nullptr;
    float* W = nullptr;         // master weights (FP32)
    float* m = nullptr;         // Adam moments
    float* v = nullptr;
    uint32_t* frag = nullptr;   // packed BF16 fragments
    float* bias = nullptr;      // b1, b2, b3, pad, W3 (FP32)
    float* partials = nullptr;
    int cap_warps = 0;
    float* d_loss = nullptr;
    float* d_grad = nullptr;
    int step = 0;
};

namespace {

gbp_status mlp_pack(gbp_mlp* n) {
    mlp_pack_kernel<<<(FT_N * 32 + 127) / 128, 128, 0, n->stream>>>(n->W, n->frag, n->bias);
    return cudaGetLastError() == cudaSuccess ? GBP_OK : GBP_ECUDA;
}

gbp_status mlp_grad(gbp_mlp* n, const float* X, const float* T, const int32_t* idx, int count, int step, float lr,
                    float* grad_out) {
    if (count <= 0) return GBP_EINVAL;
    // a warp per 32 rows while one wave of warps takes them (142 registers
    // and 15.5 KB a warp: 14 per SM), else a warp per 128
    const int warps = (count + 31) / 32;
    const bool grouped = warps > GRAD_WAVE;
    const int nw = grouped ? (count + 127) / 128 : warps;   // partials; a block each
    if (nw > n->cap_warps) {
        if (n->partials) cudaFree(n->partials);
        n->partials = nullptr;
        n->cap_warps = 0;
        if (cudaMalloc(reinterpret_cast<void**>(&n->partials), sizeof(float) * (size_t)nw * MLP_PART) != cudaSuccess)
            return GBP_ENOMEM;
        n->cap_warps = nw;
    }
    // programmatic dependent launch: each kernel's launch overlaps the end of
    // the one before it, whose results it waits for before it reads anything
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = n->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(nw);
    cfg.blockDim = dim3(32);
    cudaError_t e = cudaLaunchKernelEx(&cfg, grouped ? mlp_grad_kernel<true> : mlp_grad_kernel<false>, (const uint32_t*)n->frag, (const float*)n->bias, X, T, idx,
                                       count, 1.0f / count, n->partials);
    cfg.gridDim = dim3((MLP_NPARAM + 1 + 31) / 32);
    cfg.blockDim = dim3(RED_WARPS * 32);
    if (e == cudaSuccess)
        e = cudaLaunchKernelEx(&cfg, grouped ? mlp_reduce_kernel<1> : mlp_reduce_kernel<4>, (const float*)n->partials, nw, n->W, n->m, n->v, step, lr,
                               grad_out, n->d_loss, n->frag, n->bias);
    return e == cudaSuccess ? GBP_OK : GBP_ECUDA;
}

}  // namespace

extern "C" {

gbp_status gbp_mlp_create(const float* params, void* cuda_stream, gbp_mlp** out) {
    if (!out || !params) return GBP_EINVAL;
    *out = nullptr;
    for (int i = 0; i < MLP_NPARAM; ++i)
        if (!std::isfinite(params[i])) return GBP_EINVAL;
    gbp_mlp* n = new (std::nothrow) gbp_mlp();
    if (!n) return GBP_ENOMEM;
    n->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&n->W), sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->m), sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->v), sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->frag), sizeof(uint32_t) * FRAG_WORDS);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->bias), sizeof(float) * MLP_BIAS_WORDS);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->d_loss), sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->d_grad), sizeof(float) * MLP_NPARAM);
    if (e == cudaSuccess) e = cudaMemcpyAsync(n->W, params, sizeof(float) * MLP_NPARAM, cudaMemcpyHostToDevice, n->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->m, 0, sizeof(float) * MLP_NPARAM, n->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->v, 0, sizeof(float) * MLP_NPARAM, n->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);   // params is the caller's
    if (e != cudaSuccess || mlp_pack(n) != GBP_OK) {
        gbp_mlp_destroy(n);
        return GBP_ECUDA;
    }
    *out = n;
    return GBP_OK;
}

void gbp_mlp_destroy(gbp_mlp* n) {
    if (!n) return;
    void* ptrs[] = {n->W, n->m, n->v, n->frag, n->bias, n->partials, n->d_loss, n->d_grad};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete n;
}

gbp_status gbp_mlp_set_params(gbp_mlp* n, const float* params) {
    if (!n || !params) return GBP_EINVAL;
    for (int i = 0; i < MLP_NPARAM; ++i)
        if (!std::isfinite(params[i])) return GBP_EINVAL;
    if (cudaMemcpyAsync(n->W, params, sizeof(float) * MLP_NPARAM, cudaMemcpyHostToDevice, n->stream) != cudaSuccess ||
        cudaMemsetAsync(n->m, 0, sizeof(float) * MLP_NPARAM, n->stream) != cudaSuccess ||
        cudaMemsetAsync(n->v, 0, sizeof(float) * MLP_NPARAM, n->stream) != cudaSuccess)
        return GBP_ECUDA;
    n->step = 0;
    // the host buffer may be reused by the caller as soon as we return
    if (cudaStreamSynchronize(n->stream) != cudaSuccess) return GBP_ECUDA;
    return mlp_pack(n);
}

gbp_status gbp_mlp_get_params(const gbp_mlp* n, float* params) {
    if (!n || !params) return GBP_EINVAL;
    if (cudaMemcpyAsync(params, n->W, sizeof(float) * MLP_NPARAM, cudaMemcpyDeviceToHost, n->stream) != cudaSuccess ||
        cudaStreamSynchronize(n->stream) != cudaSuccess)
        return GBP_ECUDA;
    return GBP_OK;
}

gbp_status gbp_mlp_forward(gbp_mlp* n, const float* X, int32_t count, float* y) {
    if (!n || count < 0 || (count && (!X || !y))) return GBP_EINVAL;
    if (count == 0) return GBP_OK;
    // resident blocks walk the tiles (three per SM, the register budget); X may
    // be aligned to a float only
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return GBP_ECUDA;
    const int tiles = (count + 15) / 16;
    const int blocks = std::min((tiles + MLP_WARPS - 1) / MLP_WARPS, 3 * sms);
    if (reinterpret_cast<uintptr_t>(X) % 8 == 0)
        mlp_forward_kernel<true><<<blocks, MLP_BLOCK, 0, n->stream>>>(n->frag, n->bias, X, count, y);
    else
        mlp_forward_kernel<false><<<blocks, MLP_BLOCK, 0, n->stream>>>(n->frag, n->bias, X, count, y);
    return cudaGetLastError() == cudaSuccess ? GBP_OK : GBP_ECUDA;
}

gbp_status gbp_mlp_gradient(gbp_mlp* n, const float* X, const float* target, int32_t count, float* grad,
                            double* loss) {
    if (!n || !X || !target || !grad || count <= 0) return GBP_EINVAL;
    gbp_status st = mlp_grad(n, X, target, nullptr, count, 0, 0.f, n->d_grad);
    if (st != GBP_OK) return st;
    float l = 0.f;
    if (cudaMemcpyAsync(grad, n->d_grad, sizeof(float) * MLP_NPARAM, cudaMemcpyDeviceToHost, n->stream) != cudaSuccess ||
        cudaMemcpyAsync(&l, n->d_loss, sizeof(float), cudaMemcpyDeviceToHost, n->stream) != cudaSuccess ||
        cudaStreamSynchronize(n->stream) != cudaSuccess)
        return GBP_ECUDA;
    if (loss) *loss = l;
    return GBP_OK;
}

gbp_status gbp_mlp_train_step(gbp_mlp* n, const float* X, const float* target, const int32_t* idx, int32_t count,
                              float lr, float* loss_out) {
    if (!n || !X || !target || count <= 0 || !(lr > 0.f)) return GBP_EINVAL;
    n->step += 1;
    gbp_status st = mlp_grad(n, X, target, idx, count, n->step, lr, nullptr);
    if (st != GBP_OK) return st;
    if (loss_out) {
        if (cudaMemcpyAsync(loss_out, n->d_loss, sizeof(float), cudaMemcpyDeviceToHost, n->stream) != cudaSuccess ||
            cudaStreamSynchronize(n->stream) != cudaSuccess)
            return GBP_ECUDA;
    }
    return GBP_OK;
}

}  // extern "C"

namespace gbp {
cudaError_t mlp_copy_packed(const gbp_mlp* n, uint32_t* frag, float* bias, cudaStream_t s) {
    // the network's own stream may still be packing its latest weights
    cudaError_t e = cudaStreamSynchronize(n->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(frag, n->frag, sizeof(uint32_t) * FWD_FRAG_WORDS, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(bias, n->bias, sizeof(float) * MLP_BIAS_WORDS, cudaMemcpyDeviceToDevice, s);
    return e;
}
}  // namespace gbp
