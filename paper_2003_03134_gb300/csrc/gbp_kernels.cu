// gbp_kernels.cu -- CUDA kernels (sm_103a) of one synchronous GBP iteration
// for bundle adjustment (Ortiz et al., "Bundle Adjustment on a Graph
// Processor", CVPR 2020), templated on the storage/arithmetic type R
// (float: the fast path with an FP64 fallback; double: a full-precision
// mode).
//
// Iteration t (Sec. 5, synchronous schedule):
//   factor kernel  -- a warp per tile of whole landmarks, a lane per factor:
//                     both incoming messages, the relinearisation test
//                     (Sec. 5, Sec. 8), the Jacobian and residual at the
//                     factor's linearisation point, the Huber weight
//                     (Sec. 6), both factor-to-variable messages (eqs.
//                     messageeta, messagelambda), damping of eta (Sec. 5,
//                     Sec. 8); the beliefs of the landmarks inside the tile.
//   belief kernel  -- a block (small graphs) or a warp per keyframe: a
//                     fixed-order reduction of its messages, expanded from
//                     their compact form: prior(t+1) + sum of messages
//                     (eqs. beliefeta, belieflambda), its Cholesky factor
//                     and mean.
// No atomics touch floating-point sums: every reduction has a fixed order,
// so results are bitwise reproducible.
#include "gbp_device.cuh"

#include <algorithm>
#include <utility>

namespace gbp {

// ------------------------------------------------------------------------
// Two-kernel iteration (the launch-per-phase path).

// Programmatic dependent launch: the per-phase kernels let the next kernel
// in the stream launch once all of their blocks are past their main work
// (so only one kernel waits ahead), and wait for the previous kernel's
// completion (and its memory) before they read anything it writes.  Without
// the launch attribute both are no-ops.
__device__ __forceinline__ void pdl_allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_prev() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename R, int MODE, int NT, bool DEFER>
__device__ __forceinline__ void factor_body(const DevGraph<R>& g, const KParams<R>& P) {
    __shared__ __align__(16) MlpSmem<MODE> S;
    mlp_load_async<MODE>(P, S);   // network weights do not change between iterations
    pdl_wait_prev();
    const int lane = threadIdx.x & 31;
    const int tile = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
    const int t = g.ctl[CTL_ITER];
    float dmu = 0.0f;
    if (tile < g.n_tiles)   // uniform per warp
        if constexpr (DEFER) dmu = tile_work_deferring(g, P, g.tile_off + tile, t, lane);
        else dmu = tile_work<R, MODE, false>(g, P, g.tile_off + tile, t, lane, S, MODE == DAMP_LEARNED);
    else if constexpr (MODE == DAMP_LEARNED) mlp_load_wait();   // the block's barrier, for warps without a tile
    pdl_allow_next();
    dmu = warp_max(dmu);
    if (lane == 0 && dmu > 0.0f) dmu_atomic_max_slot(g.ctl, dmu_slot(t), dmu);
    // the belief kernel of this iteration reads t from CTL_ITER_B: the belief
    // kernel of t - 1 has finished and that of t starts after this kernel
    if (blockIdx.x == 0 && threadIdx.x == 0) g.ctl[CTL_ITER_B] = t;
}

// NT threads per block, and at least MINB blocks per SM (the register budget
// per thread; 1 = no constraint).  Each warp does one tile whatever the
// shape, so every shape gives bitwise identical results; the FP32 fixed
// schedule is instantiated in several shapes for the autotuner.
template <typename R, int MODE, int NT, int MINB, bool DEFER = false>
__global__ void __launch_bounds__(NT, MINB) factor_kernel(const __grid_constant__ DevGraph<R> g,
                                                          const __grid_constant__ KParams<R> P) {
    factor_body<R, MODE, NT, DEFER>(g, P);
}

// The tiles that factor_kernel<..., DEFER = true> left in this iteration
// (a factor of theirs needs the FP64 redo), worked with it: warps walk the
// list.  No store of theirs happened before, so they see the same state.
// The last block to finish clears the list for the next use of its slot.
template <typename R>
__global__ void __launch_bounds__(FACTOR_BLOCK) factor_deferred_kernel(const __grid_constant__ DevGraph<R> g,
                                                                       const __grid_constant__ KParams<R> P) {
    constexpr int WPB = FACTOR_BLOCK / 32;
    MlpSmem<DAMP_FIXED> S;
    pdl_wait_prev();
    const int lane = threadIdx.x & 31;
    const int t = g.ctl[CTL_ITER];
    const int slot = CTL_DEFER_N0 + (t & 1);
    const int n = min(g.ctl[slot], g.n_tiles);
    float dmu = 0.0f;
    for (int i = blockIdx.x * WPB + (threadIdx.x >> 5); i < n; i += gridDim.x * WPB)
        dmu = fmaxf(dmu, tile_work<R, DAMP_FIXED, false>(g, P, g.deferred[i], t, lane, S));
    pdl_allow_next();
    dmu = warp_max(dmu);
    if (lane == 0 && dmu > 0.0f) dmu_atomic_max_slot(g.ctl, dmu_slot(t), dmu);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&g.ctl[CTL_DEFER_DONE], 1) == int(gridDim.x) - 1) {
            g.ctl[slot] = 0;
            g.ctl[CTL_DEFER_DONE] = 0;
        }
    }
}

// BW = g.b_warps (warps per belief item), one instantiation per mapping
template <typename R, int BW>
__global__ void __launch_bounds__(FACTOR_BLOCK) belief_kernel(DevGraph<R> g, KParams<R> P) {
    pdl_wait_prev();
    const int t = g.ctl[CTL_ITER_B];
    // close the iteration from one thread: the factor kernel of t has
    // finished and that of t + 1 starts only after this kernel, so the
    // counter it reads and the |dmu| slot it fills are free to set now
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g.ctl[CTL_ITER] = t + 1;
        g.ctl[dmu_slot(t + 1)] = 0;
    }
    float dmu = 0.0f;
    const int item = phase_b_item_of(BW, blockIdx.x);
    if (item < phase_b_items(g)) dmu = phase_b_item<R, BW, false>(g, P, item, t);   // uniform per group
    pdl_allow_next();
    // max is order independent: the atomic on non-negative float bits is deterministic
    if (dmu > 0.0f) dmu_atomic_max_slot(g.ctl, dmu_slot(t), dmu);
}

// ------------------------------------------------------------------------
// Persistent iteration kernel: one cooperative launch runs up to n_iters
// iterations; the two phases are separated by a grid barrier.  The barrier's
// wait is bounded: after ~1 s without progress the block records a timeout
// (CTL_ERR = 2) and every block leaves the loop.

constexpr long long BARRIER_SPIN_LIMIT = 10000000;   // x ~100 ns sleeps

__device__ __forceinline__ bool grid_barrier(int32_t* ctl, int nblocks, int* flag_sh) {
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int32_t* vgen = ctl + CTL_BAR_GEN;
        volatile int32_t* verr = ctl + CTL_ERR;
        const int gen = *vgen;
        __threadfence();
        const int arrived = atomicAdd(&ctl[CTL_BAR_COUNT], 1);
        int ok = 1;
        if (arrived == nblocks - 1) {
            atomicExch(&ctl[CTL_BAR_COUNT], 0);
            __threadfence();
            atomicAdd(&ctl[CTL_BAR_GEN], 1);
        } else {
            long long spins = 0;
            while (*vgen == gen) {
                if (*verr == 2 || ++spins > BARRIER_SPIN_LIMIT) {
                    atomicCAS(&ctl[CTL_ERR], 0, 2);
                    ok = 0;
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
        *flag_sh = ok && (*verr != 2);
    }
    __syncthreads();
    return *flag_sh;
}

// BW = g.b_warps (warps per belief item): a separate instantiation per
// mapping, so that the block mapping's barriers and shared-memory reduction
// do not weigh on the register allocation of the warp mapping's kernel.
// MINB: at least this many blocks per SM (the register budget; 1 = none),
// a launch shape the autotuner chooses for the FP32 fixed schedule.
template <typename R, int MODE, int BW, int MINB>
__global__ void __launch_bounds__(FACTOR_BLOCK, MINB)
    persistent_kernel(const __grid_constant__ DevGraph<R> g, const __grid_constant__ KParams<R> P, int n_iters,
                      float conv_tol, int check_every) {
    __shared__ int flag_sh;
    __shared__ __align__(16) MlpSmem<MODE> S;
    mlp_load<MODE>(P, S);
    constexpr int WPB = FACTOR_BLOCK / 32;
    const int lane = threadIdx.x & 31;
    const int gwarp = blockIdx.x * WPB + (threadIdx.x >> 5);
    const int nwarps = gridDim.x * WPB;
    const int nb = gridDim.x;
    const int t0 = __ldcg(&g.ctl[CTL_ITER]);
    const int items = phase_b_items(g);
    int done = 0;
    float last = 0.0f;
    for (int it = 0; it < n_iters; ++it) {
        const int t = t0 + it;
        // phase A: factors and landmarks wholly inside a tile
        float dmu = 0.0f;
        for (int tile = gwarp; tile < g.n_tiles; tile += nwarps)
            dmu = fmaxf(dmu, tile_work<R, MODE, true>(g, P, g.tile_off + tile, t, lane, S));
        dmu = warp_max(dmu);
        if (lane == 0 && dmu > 0.0f) dmu_atomic_max_slot(g.ctl, dmu_slot(t), dmu);
        if (!grid_barrier(g.ctl, nb, &flag_sh)) break;
        // phase B: keyframes, split landmarks, orphans
        if (blockIdx.x == 0 && threadIdx.x == 0) g.ctl[dmu_slot(t + 1)] = 0;   // every block has read it
        float d2 = 0.0f;
        // a block per item, or a warp per item (see phase_b_item)
        constexpr bool per_block = BW == WPB;
        const int stride = per_block ? nb : nwarps;
        for (int item = per_block ? int(blockIdx.x) : gwarp; item < items; item += stride)
            d2 = fmaxf(d2, phase_b_item<R, BW, true>(g, P, item, t));
        if (d2 > 0.0f) dmu_atomic_max_slot(g.ctl, dmu_slot(t), d2);   // groups' first threads
        if (!grid_barrier(g.ctl, nb, &flag_sh)) break;
        done = it + 1;
        last = __int_as_float(__ldcg(&g.ctl[dmu_slot(t)]));
        if (conv_tol > 0.0f && done % check_every == 0 && last < conv_tol) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g.ctl[CTL_ITER] = t0 + done;
        g.ctl[CTL_DMU_LAST] = __float_as_int(last);
        g.ctl[CTL_ITERS_RUN] = done;
    }
}

// The tile entries (gbp_internal.h) from the tiles' factors: a thread per lane.
// The lanes of a landmark that lies in one tile (at most 32 factors) follow
// one another in factor order.
template <typename R>
__global__ void __launch_bounds__(128) tile_index_kernel(DevGraph<R> g, int n_tiles, int4* __restrict__ tidx) {
    const size_t i = (size_t)blockIdx.x * 128 + threadIdx.x;
    if (i >= (size_t)n_tiles * 32) return;
    const int lane = threadIdx.x & 31, f = g.tf[i];
    int4 e = make_int4(-1, 0, -1, lane | (lane << 8));
    if (f >= 0) {
        e.x = g.fk[f];
        e.y = g.kpos[f];
        e.z = g.fm[f];
        const int lo = g.lm_off[e.z], n = g.lm_off[e.z + 1] - lo, first = lane - (f - lo);
        if (n <= 32) e.w = first | ((first + n - 1) << 8) | TIDX_WHOLE;
    }
    tidx[i] = e;
}

// Beliefs of iteration 0: b^0 = prior(0) (+ anchor), mean 0.
template <typename R>
__global__ void init_beliefs_kernel(DevGraph<R> g, KParams<R> P) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    const R isig2 = P.inv_sigma2;
    if (v < g.n_kf) {
        const R s = kf_prior_scale(g, P, v, g.kf_birth[v]);
        R p[6], out[KBEL];
#pragma unroll
        for (int i = 0; i < 6; ++i) p[i] = (s * g.kf_D[v * 6 + i] + P.anchor_scale * g.kf_A[v * 6 + i]) * isig2;
        kf_prior_record<R>(p, out);
        store_rec<R, KBEL>(g.kf_bel + (size_t)v * KBEL, out);
    } else if (v < g.n_kf + g.n_lm) {
        const int m = v - g.n_kf;
        const R s = lm_prior_scale(g, P, m, g.lm_birth[m]);
        R out[LBEL];
#pragma unroll
        for (int j = 0; j < LBEL; ++j) out[j] = R(0);
#pragma unroll
        for (int i = 0; i < 3; ++i) out[pk(i, i)] = s * g.lm_D[m * 3 + i] * isig2;
        store_rec<R, LBEL>(g.lm_bel + (size_t)m * LBEL, out);
    }
}

// Beliefs of variables added to a graph: prior(0) alone, mean 0.  The factor
// of a keyframe's record is rounded from FP64.
template <typename R>
__global__ void init_new_kernel(DevGraph<R> g, KParams<R> P, int k0, int l0) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    const int nk = g.n_kf - k0, nl = g.n_lm - l0;
    const R s0 = prior_scale(P, 0), isig2 = P.inv_sigma2;
    if (v < nk) {
        const int k = k0 + v;
        R p[6], out[KBEL];
        for (int i = 0; i < 6; ++i) p[i] = mul_rn(mul_rn(s0, g.kf_D[k * 6 + i]), isig2);
        kf_prior_record<R>(p, out);
        for (int i = 0; i < 6; ++i) out[KB_L + pk(i, i)] = R(1.0 / sqrt(double(p[i])));
        store_rec<R, KBEL>(g.kf_bel + (size_t)k * KBEL, out);
    } else if (v < nk + nl) {
        const size_t m = l0 + (v - nk);
        R out[LBEL];
        for (int j = 0; j < LBEL; ++j) out[j] = R(0);
        for (int i = 0; i < 3; ++i) out[pk(i, i)] = mul_rn(mul_rn(s0, g.lm_D[m * 3 + i]), isig2);
        store_rec<R, LBEL>(g.lm_bel + m * LBEL, out);
    }
}

// ------------------------------------------------------------------------
// prior generation (Sec. 4 / Sec. 8): per-variable mean over its factors of
// diag(J_v^T J_v) at the factors' linearisation points (the references, at
// creation) with Huber weight 1 and sigma = 1.

template <typename R>
__global__ void __launch_bounds__(FACTOR_BLOCK) prior_factor_kernel(DevGraph<R> g, KParams<R> P, R* tmp_k, R* tmp_l) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= g.n_f) return;
    const int k = g.fk[f], m = g.fm[f];
    KParams<R> Q = P;
    Q.huber_n = R(0);
    Q.inv_sigma2 = R(1);
    Q.inv_sigma = R(1);
    R x0[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) x0[i] = g.x0[(size_t)i * g.n_f + f];
    Lin<R> L;
    linearise<R>(Q, g.kf_R + (size_t)k * 9, g.kf_c + (size_t)k * 3, g.lm_ref + (size_t)m * 3, x0,
                 g.z[2 * (size_t)f], g.z[2 * (size_t)f + 1], L);
#pragma unroll
    for (int j = 0; j < 6; ++j) tmp_k[(size_t)j * g.n_f + f] = L.W * (L.Jk[0][j] * L.Jk[0][j] + L.Jk[1][j] * L.Jk[1][j]);
#pragma unroll
    for (int j = 0; j < 3; ++j) tmp_l[(size_t)j * g.n_f + f] = L.W * (L.Jl[0][j] * L.Jl[0][j] + L.Jl[1][j] * L.Jl[1][j]);
}

template <typename R, int n>
__device__ __forceinline__ void finish_prior(R* D, int deg) {
    R mx = R(0);
#pragma unroll
    for (int i = 0; i < n; ++i) {
        if (deg > 0) D[i] /= R(deg);
        mx = fmax(mx, D[i]);
    }
#pragma unroll
    for (int i = 0; i < n; ++i) {
        if (mx <= R(0)) D[i] = R(1);
        else if (D[i] < R(1e-9) * mx) D[i] = R(1e-9) * mx;
    }
}

template <typename R>
__global__ void prior_reduce_kernel(DevGraph<R> g, const R* tmp_k, const R* tmp_l, R* kf_D, R* kf_A, const R* anc,
                                    R* lm_D) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < g.n_kf) {
        R D[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
        const int b0 = g.kf_off[v], b1 = g.kf_off[v + 1];
        for (int i = b0; i < b1; ++i) {
            const int f = g.kf_list[i];
#pragma unroll
            for (int j = 0; j < 6; ++j) D[j] += tmp_k[(size_t)j * g.n_f + f];
        }
        finish_prior<R, 6>(D, b1 - b0);
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            kf_D[v * 6 + j] = D[j];
            kf_A[v * 6 + j] = anc[v * 6 + j] * D[j];
        }
    } else if (v < g.n_kf + g.n_lm) {
        const int m = v - g.n_kf;
        R D[3] = {R(0), R(0), R(0)};
        const int b0 = g.lm_off[m], b1 = g.lm_off[m + 1];
        for (int f = b0; f < b1; ++f) {
#pragma unroll
            for (int j = 0; j < 3; ++j) D[j] += tmp_l[(size_t)j * g.n_f + f];
        }
        finish_prior<R, 3>(D, b1 - b0);
#pragma unroll
        for (int j = 0; j < 3; ++j) lm_D[m * 3 + j] = D[j];
    }
}

// ------------------------------------------------------------------------
// metrics: average reprojection error (Sec. 9.1) at the current means, its
// distance to reference projections, Huber-regime count.  Two-pass fixed
// order reduction through per-block partials.
//
// Bound: the FP64 pipe (a warp instruction per 16 cycles and SM).  The
// references come rounded to R from the host (kf_Rr, f_dlc: the same roundings
// as rounding them here), counts are integers, and what is left in FP64 per
// factor is the square root of |r|^2 and the sum.  900k factors: 61 -> 38 us
// (metrics_kernel), 45 -> 23 us (residual_kernel), and 192 -> 8 us for the
// final sum by a block instead of one thread (kernel times under ncu).

// |z - h(mu)|^2 of factor f at the current means; false where the point is
// closer than z_min to its camera.
template <typename R>
__device__ __forceinline__ bool error2_at_means(const DevGraph<R>& g, const KParams<R>& P, int f, R zu, R zv, R& r2) {
    const size_t n_f = g.n_f;
    const int k = g.fk[f], m = g.fm[f];
    const R* kb = g.kf_bel + (size_t)k * KBEL;
    const R* lb = g.lm_bel + (size_t)m * LBEL;
    const R x[9] = {kb[KB_MU], kb[KB_MU + 1], kb[KB_MU + 2], kb[KB_MU + 3], kb[KB_MU + 4], kb[KB_MU + 5],
                    lb[9], lb[10], lb[11]};
    KParams<R> Q = P;
    Q.huber_n = R(0);
    Lin<R> L;
    const R dlc[3] = {g.f_dlc[f], g.f_dlc[n_f + f], g.f_dlc[2 * n_f + f]};
    R Rr[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) Rr[i] = g.kf_Rr[(size_t)k * 9 + i];
    linearise_ref<R>(Q, Rr, dlc, x, zu, zv, L);
    r2 = L.r2;
    return L.W > R(0);
}

// Sums of a block: one double (tree over the threads) and up to three counts.
template <int NC>
__device__ __forceinline__ double block_metrics(double v, int (&n)[NC]) {
    __shared__ double red[METRIC_BLOCK];
    __shared__ int cnt[NC];
    const int tid = threadIdx.x;
    red[tid] = v;
    if (tid < NC) cnt[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        n[j] = __reduce_add_sync(0xffffffffu, n[j]);
        if ((tid & 31) == 0 && n[j]) atomicAdd(&cnt[j], n[j]);
    }
    for (int st = METRIC_BLOCK / 2; st > 0; st >>= 1) {
        if (tid < st) red[tid] += red[tid + st];
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < NC; ++j) n[j] = cnt[j];
    return red[0];
}

template <typename R>
__global__ void __launch_bounds__(METRIC_BLOCK) metrics_kernel(DevGraph<R> g, KParams<R> P, double* partials) {
    double v = 0.0;
    int n[2] = {0, 0};   // counted, in the Huber regime
    for (int f = blockIdx.x * METRIC_BLOCK + threadIdx.x; f < g.n_f; f += gridDim.x * METRIC_BLOCK) {
        R r2;
        if (error2_at_means<R>(g, P, f, g.z[2 * (size_t)f], g.z[2 * (size_t)f + 1], r2)) {
            const double e = sqrt(double(r2));
            v += e;
            ++n[0];
            if (P.huber_n > R(0) && e * double(P.inv_sigma) > double(P.huber_n)) ++n[1];
        }
    }
    const double s = block_metrics<2>(v, n);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = s;
        partials[2 * (size_t)gridDim.x + blockIdx.x] = double(n[0]);
        partials[3 * (size_t)gridDim.x + blockIdx.x] = double(n[1]);
    }
}

// reference-projection distance needs the residual vector, not only |r|:
// recompute h(mu) per factor (with z = reference pixel the residual is ref - h(mu))
template <typename R>
__global__ void __launch_bounds__(METRIC_BLOCK) metrics_ref_kernel(DevGraph<R> g, KParams<R> P, double* partials) {
    double v = 0.0;
    int n[1] = {0};
    for (int f = blockIdx.x * METRIC_BLOCK + threadIdx.x; f < g.n_f; f += gridDim.x * METRIC_BLOCK) {
        const R ru = g.uv_ref[2 * (size_t)f], rv = g.uv_ref[2 * (size_t)f + 1];
        R r2;
        if (error2_at_means<R>(g, P, f, ru, rv, r2) && isfinite(ru)) {
            v += sqrt(double(r2));
            ++n[0];
        }
    }
    const double s = block_metrics<1>(v, n);
    if (threadIdx.x == 0) {
        partials[4 * (size_t)gridDim.x + blockIdx.x] = s;
        partials[5 * (size_t)gridDim.x + blockIdx.x] = double(n[0]);
    }
}

// Per-problem reprojection statistics of a batch: one block per problem
// over its contiguous factor range, fixed-order block reduction.
// out[3p] = sum of errors, out[3p+1] = count, out[3p+2] = Huber-regime count.
template <typename R>
__global__ void __launch_bounds__(METRIC_BLOCK) problem_metrics_kernel(DevGraph<R> g, KParams<R> P,
                                                                       const int32_t* prob_f0, double* out) {
    const int p = blockIdx.x;
    double v = 0.0;
    int n[2] = {0, 0};
    for (int f = prob_f0[p] + threadIdx.x; f < prob_f0[p + 1]; f += METRIC_BLOCK) {
        R r2;
        if (error2_at_means<R>(g, P, f, g.z[2 * (size_t)f], g.z[2 * (size_t)f + 1], r2)) {
            const double e = sqrt(double(r2));
            v += e;
            ++n[0];
            if (P.huber_n > R(0) && e * double(P.inv_sigma) > double(P.huber_n)) ++n[1];
        }
    }
    const double s = block_metrics<2>(v, n);
    if (threadIdx.x == 0) {
        out[3 * (size_t)p] = s;
        out[3 * (size_t)p + 1] = double(n[0]);
        out[3 * (size_t)p + 2] = double(n[1]);
    }
}

// Per-factor reprojection error |z - h(mu)| at the current means (Sec. 9.1),
// -1 for a point closer than z_min to its camera; to its place in the
// caller's order.
template <typename R>
__global__ void __launch_bounds__(METRIC_BLOCK) residual_kernel(DevGraph<R> g, KParams<R> P,
                                                                const int32_t* __restrict__ obs_index, double* out) {
    const int f = blockIdx.x * METRIC_BLOCK + threadIdx.x;
    if (f >= g.n_f) return;
    R r2;
    const bool ok = error2_at_means<R>(g, P, f, g.z[2 * (size_t)f], g.z[2 * (size_t)f + 1], r2);
    out[obs_index[f]] = ok ? sqrt(double(r2)) : -1.0;
}

// The current means for the caller, in double, so that they leave the device
// as the arrays the caller asked for (a copy of 120 bytes a keyframe and
// point, no pass over the belief records on the host): chart means (n x 6,
// n x 3), or world poses Exp(dw) Rref | t and points.
__device__ __forceinline__ void so3_exp_double(const double w[3], double E[9]) {
    const double th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    double a, b;
    if (th2 < 1e-12) {
        a = 1.0 - th2 / 6.0;
        b = 0.5 - th2 / 24.0;
    } else {
        const double th = sqrt(th2), sh = sin(0.5 * th);
        a = sin(th) / th;
        b = 2.0 * sh * sh / th2;
    }
    const double W[9] = {0, -w[2], w[1], w[2], 0, -w[0], -w[1], w[0], 0};
    const double W2[9] = {w[0] * w[0] - th2, w[0] * w[1], w[0] * w[2], w[1] * w[0], w[1] * w[1] - th2, w[1] * w[2],
                          w[2] * w[0], w[2] * w[1], w[2] * w[2] - th2};
    for (int i = 0; i < 9; ++i) E[i] = a * W[i] + b * W2[i];
    E[0] += 1.0; E[4] += 1.0; E[8] += 1.0;
}

template <typename R>
__global__ void __launch_bounds__(128) means_kernel(DevGraph<R> g, int world, double* __restrict__ kf,
                                                    double* __restrict__ lm, int32_t* __restrict__ ctl_out) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (ctl_out && blockIdx.x == 0 && threadIdx.x < CTL_N) ctl_out[threadIdx.x] = g.ctl[threadIdx.x];
    if (v < g.n_kf) {
        const R* kb = g.kf_bel + (size_t)v * KBEL + KB_MU;
        double mu[6];
        for (int i = 0; i < 6; ++i) mu[i] = double(kb[i]);
        if (!world) {
            for (int i = 0; i < 6; ++i) kf[6 * (size_t)v + i] = mu[i];
            return;
        }
        double E[9], Rm[9], c[3];
        so3_exp_double(mu + 3, E);
        const double* Rr = g.kf_R + 9 * (size_t)v;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j)
                Rm[3 * i + j] = E[3 * i] * Rr[j] + E[3 * i + 1] * Rr[3 + j] + E[3 * i + 2] * Rr[6 + j];
        for (int i = 0; i < 3; ++i) c[i] = g.kf_c[3 * (size_t)v + i] + mu[i];
        double* o = kf + 12 * (size_t)v;
        for (int i = 0; i < 9; ++i) o[i] = Rm[i];
        for (int i = 0; i < 3; ++i) o[9 + i] = -(Rm[3 * i] * c[0] + Rm[3 * i + 1] * c[1] + Rm[3 * i + 2] * c[2]);
    } else if (v < g.n_kf + g.n_lm) {
        const size_t m = v - g.n_kf;
        for (int i = 0; i < 3; ++i) {
            const double d = double(g.lm_bel[m * LBEL + 9 + i]);
            lm[3 * m + i] = world ? g.lm_ref[3 * m + i] + d : d;
        }
    }
}

// The blocks' partials added up by one block, in a fixed order (a thread's
// own in block order, then a tree).
__global__ void __launch_bounds__(METRIC_BLOCK) metrics_finish_kernel(const double* partials, int nb, int with_ref,
                                                                      double* out) {
    __shared__ double red[6][METRIC_BLOCK];
    const int tid = threadIdx.x, rows = with_ref ? 6 : 4;   // rows: error, -, counted, Huber, ref error, ref counted
    for (int j = 0; j < rows; ++j) {
        double s = 0.0;
        if (j != 1)
            for (int b = tid; b < nb; b += METRIC_BLOCK) s += partials[(size_t)j * nb + b];
        red[j][tid] = s;
    }
    __syncthreads();
    for (int st = METRIC_BLOCK / 2; st > 0; st >>= 1) {
        if (tid < st)
            for (int j = 0; j < rows; ++j) red[j][tid] += red[j][tid + st];
        __syncthreads();
    }
    if (tid != 0) return;
    out[MET_N_ARE] = red[2][0];
    out[MET_ARE] = red[2][0] > 0 ? red[0][0] / red[2][0] : 0.0;
    out[MET_HUBER] = red[3][0];
    out[MET_ARE_REF] = with_ref ? (red[5][0] > 0 ? red[4][0] / red[5][0] : 0.0) : -1.0;
}

// ------------------------------------------------------------------------
// launchers

int metrics_blocks(int n_f) {
    int b = (n_f + METRIC_BLOCK - 1) / METRIC_BLOCK;
    if (b < 1) b = 1;
    if (b > 1024) b = 1024;
    return b;
}

// One launch, with programmatic stream serialisation when pdl is set.
template <typename... KArgs, typename... Args>
cudaError_t launch_ex(void (*kernel)(KArgs...), int blocks, int threads, cudaStream_t s, bool pdl, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename R, int MODE, int NT, int MINB, bool DEFER = false>
cudaError_t launch_factor_shape(const DevGraph<R>& g, const KParams<R>& p, cudaStream_t s, bool pdl) {
    constexpr int wpb = NT / 32;
    const int blocks = std::max(1, (g.n_tiles + wpb - 1) / wpb);   // >= 1: it also publishes the iteration index
    cudaError_t e = launch_ex(factor_kernel<R, MODE, NT, MINB, DEFER>, blocks, NT, s, pdl, g, p);
    if constexpr (DEFER) {
        // deferred tiles are rare: a few hundred warps walk the list
        constexpr int wpd = FACTOR_BLOCK / 32;
        const int nb = std::max(1, std::min((g.n_tiles + wpd - 1) / wpd, 608));
        if (e == cudaSuccess) e = launch_ex(factor_deferred_kernel<R>, nb, FACTOR_BLOCK, s, pdl, g, p);
    }
    return e;
}

template <typename R>
cudaError_t launch_factor(const DevGraph<R>& g, const KParams<R>& p, cudaStream_t s, int mode, bool pdl, int shape) {
    if (mode == DAMP_LEARNED) return launch_factor_shape<R, DAMP_LEARNED, 128, 1>(g, p, s, pdl);
    if (mode == DAMP_RECORD) return launch_factor_shape<R, DAMP_RECORD, 128, 1>(g, p, s, pdl);
    if constexpr (sizeof(R) == 4) {
        switch (shape) {
            case 1: return launch_factor_shape<R, DAMP_FIXED, 128, 3>(g, p, s, pdl);
            case 2: return launch_factor_shape<R, DAMP_FIXED, 128, 4>(g, p, s, pdl);
            case 3: return launch_factor_shape<R, DAMP_FIXED, 64, 1>(g, p, s, pdl);
            case 4: return launch_factor_shape<R, DAMP_FIXED, 128, 4, true>(g, p, s, pdl);
            case 5: return launch_factor_shape<R, DAMP_FIXED, 128, 3, true>(g, p, s, pdl);
            default: break;
        }
    }
    return launch_factor_shape<R, DAMP_FIXED, 128, 1>(g, p, s, pdl);
}

template <typename R>
cudaError_t launch_belief(const DevGraph<R>& g, const KParams<R>& p, cudaStream_t s, bool pdl) {
    int blocks = phase_b_blocks(g);
    if (blocks < 1) blocks = 1;
    if (g.b_warps == FACTOR_BLOCK / 32)
        return launch_ex(belief_kernel<R, FACTOR_BLOCK / 32>, blocks, FACTOR_BLOCK, s, pdl, g, p);
    return launch_ex(belief_kernel<R, 1>, blocks, FACTOR_BLOCK, s, pdl, g, p);
}

// the persistent kernel for this graph's belief mapping and damping
// schedule (one launch shape)
template <typename R, int BW>
const void* persistent_fn_bw(int mode, int) {
    if (mode == DAMP_LEARNED) return reinterpret_cast<const void*>(persistent_kernel<R, DAMP_LEARNED, BW, 1>);
    return reinterpret_cast<const void*>(persistent_kernel<R, DAMP_FIXED, BW, 1>);
}

template <typename R>
const void* persistent_fn(const DevGraph<R>& g, int mode, int shape) {
    constexpr int WPB = FACTOR_BLOCK / 32;
    return g.b_warps == WPB ? persistent_fn_bw<R, WPB>(mode, shape) : persistent_fn_bw<R, 1>(mode, shape);
}

template <typename R>
int persistent_grid(const DevGraph<R>& g, int mode, int shape) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    const cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, persistent_fn(g, mode, shape), FACTOR_BLOCK, 0);
    if (e != cudaSuccess || per_sm <= 0) return 0;
    constexpr int wpb = FACTOR_BLOCK / 32;
    const int cap = sms * per_sm;
    const int want = std::max((g.n_tiles + wpb - 1) / wpb, phase_b_blocks(g));
    return std::max(1, std::min(cap, want));
}

template <typename R>
cudaError_t launch_persistent(const DevGraph<R>& g, const KParams<R>& p, int n_iters, float conv_tol,
                              int check_every, int grid, cudaStream_t s, int mode, int shape) {
    DevGraph<R> gg = g;
    KParams<R> pp = p;
    void* args[] = {&gg, &pp, &n_iters, &conv_tol, &check_every};
    return cudaLaunchCooperativeKernel(persistent_fn(g, mode, shape), dim3(grid), dim3(FACTOR_BLOCK), args, 0, s);
}

// The current messages' eta in factor order (keyframe side 6, landmark side
// 3; SoA 9 x n_f): the reference of the record schedule's damping targets.
// Both messages of a factor are in the basis of its current Jacobian, whose
// keyframe block the slot's kj record holds (the landmark block is minus its
// first three columns).
template <typename R>
__global__ void capture_messages_kernel(DevGraph<R> g, const R* __restrict__ mk_cur, R* __restrict__ eta_inf) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= g.n_f) return;
    const size_t n_f = g.n_f;
    const R* rec = mk_cur + (size_t)g.kpos[f] * KREC;
    const R* jr = g.kj + (size_t)g.kpos[f] * KJ;
    const R J[2][6] = {{jr[0], jr[1], jr[2], jr[3], jr[4], jr[5]}, {jr[6], jr[7], jr[8], jr[9], jr[10], jr[11]}};
    const R Jl[2][3] = {{-jr[0], -jr[1], -jr[2]}, {-jr[6], -jr[7], -jr[8]}};
    R ek[6], el[3];
    msg_eta<R, 6>(J, rec[3], rec[4], ek);
    msg_eta<R, 3>(Jl, g.ml[3 * n_f + f], g.ml[4 * n_f + f], el);
#pragma unroll
    for (int i = 0; i < 6; ++i) eta_inf[i * n_f + f] = ek[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) eta_inf[(6 + i) * n_f + f] = el[i];
}

template <typename R>
cudaError_t launch_capture_messages(const DevGraph<R>& g, int t, R* eta_inf, cudaStream_t s) {
    if (g.n_f == 0) return cudaSuccess;
    // after t completed iterations the current messages m^t are in buffer t & 1
    const R* mk_cur = (t & 1) ? g.mk2 : g.mk;
    capture_messages_kernel<R><<<(g.n_f + 255) / 256, 256, 0, s>>>(g, mk_cur, eta_inf);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_init_new(const DevGraph<R>& g, const KParams<R>& p, int k0, int l0, cudaStream_t s) {
    const int n = (g.n_kf - k0) + (g.n_lm - l0);
    if (n > 0) init_new_kernel<R><<<(n + 127) / 128, 128, 0, s>>>(g, p, k0, l0);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_tile_index(const DevGraph<R>& g, int n_tiles, int4* tidx, cudaStream_t s) {
    if (n_tiles > 0) tile_index_kernel<R><<<(n_tiles + 3) / 4, 128, 0, s>>>(g, n_tiles, tidx);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_init(const DevGraph<R>& g, const KParams<R>& p, cudaStream_t s) {
    int nv = g.n_kf + g.n_lm;
    if (nv > 0) init_beliefs_kernel<R><<<(nv + 127) / 128, 128, 0, s>>>(g, p);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_prior(const DevGraph<R>& g, const KParams<R>& p, R* tmp_k, R* tmp_l, R* kf_D, R* kf_A,
                         const R* anc, R* lm_D, cudaStream_t s) {
    if (g.n_f > 0) prior_factor_kernel<R><<<(g.n_f + FACTOR_BLOCK - 1) / FACTOR_BLOCK, FACTOR_BLOCK, 0, s>>>(g, p, tmp_k, tmp_l);
    int nv = g.n_kf + g.n_lm;
    if (nv > 0) prior_reduce_kernel<R><<<(nv + 127) / 128, 128, 0, s>>>(g, tmp_k, tmp_l, kf_D, kf_A, anc, lm_D);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_metrics(const DevGraph<R>& g, const KParams<R>& p, double* partials, int nb, double* out,
                           cudaStream_t s) {
    metrics_kernel<R><<<nb, METRIC_BLOCK, 0, s>>>(g, p, partials);
    if (g.uv_ref) metrics_ref_kernel<R><<<nb, METRIC_BLOCK, 0, s>>>(g, p, partials);
    metrics_finish_kernel<<<1, METRIC_BLOCK, 0, s>>>(partials, nb, g.uv_ref != nullptr, out);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_problem_metrics(const DevGraph<R>& g, const KParams<R>& p, const int32_t* prob_f0, int n_problems,
                                   double* out, cudaStream_t s) {
    if (n_problems > 0) problem_metrics_kernel<R><<<n_problems, METRIC_BLOCK, 0, s>>>(g, p, prob_f0, out);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_residuals(const DevGraph<R>& g, const KParams<R>& p, const int32_t* obs_index, double* out,
                             cudaStream_t s) {
    if (g.n_f > 0)
        residual_kernel<R><<<(g.n_f + METRIC_BLOCK - 1) / METRIC_BLOCK, METRIC_BLOCK, 0, s>>>(g, p, obs_index, out);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_means(const DevGraph<R>& g, bool world, double* kf, double* lm, int32_t* ctl_out, cudaStream_t s) {
    static_assert(CTL_N <= 128, "a thread per control word");
    const int nv = std::max(g.n_kf + g.n_lm, 1);
    means_kernel<R><<<(nv + 127) / 128, 128, 0, s>>>(g, world ? 1 : 0, kf, lm, ctl_out);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------
// One graph split across ranks: the records a rank exchanges between the
// phases of an iteration.  Message records (kind 0), per factor: its
// compact message to the keyframe of iteration t+1 (KREC) and its staged
// Jacobian block (KJ) -- what the keyframe's owner needs to sum it.
// Keyframe records (kind 1): the belief record (KBEL).

constexpr int SPLIT_MSG = KREC + KJ;

template <typename R>
__global__ void split_records_kernel(DevGraph<R> g, int kind, int put, int n, const int32_t* __restrict__ idx,
                                     float* io) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (kind == 0) {
        const int t = g.ctl[CTL_ITER];
        const size_t slot = (size_t)g.kpos[idx[i]];
        R* rec = mk_write(g, t) + slot * KREC;
        R* jr = g.kjs + slot * KJ;
        float* o = io + (size_t)i * SPLIT_MSG;
        for (int j = 0; j < KREC; ++j) {
            if (put) rec[j] = R(o[j]);
            else o[j] = float(rec[j]);
        }
        for (int j = 0; j < KJ; ++j) {
            if (put) jr[j] = R(o[KREC + j]);
            else o[KREC + j] = float(jr[j]);
        }
    } else {
        R* rec = g.kf_bel + (size_t)idx[i] * KBEL;
        float* o = io + (size_t)i * KBEL;
        for (int j = 0; j < KBEL; ++j) {
            if (put) rec[j] = R(o[j]);
            else o[j] = float(rec[j]);
        }
    }
}

template <typename R>
cudaError_t launch_split_records(const DevGraph<R>& g, int kind, int put, int n, const int32_t* idx, float* io,
                                 cudaStream_t s) {
    if (n > 0) split_records_kernel<R><<<(n + 127) / 128, 128, 0, s>>>(g, kind, put, n, idx, io);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------
// Re-layout after a keyframe is added (incremental SLAM): the per-factor
// state of the grown graph gathered on the device from the previous
// layout's buffers.  src_f[f]: the previous internal index of the new
// layout's factor f, or -1 for a factor of the new keyframe.
//   phase 0: linearisation points -- kept, or for a new factor the current
//            means (its keyframe's chart origin and its landmark's mean,
//            or 0 for a new landmark);
//   phase 1: t_lin, the stored linearisation, the landmark message, the
//            learned schedule's history, and by keyframe slot the Jacobian
//            block and both message buffers -- kept, or empty and t_lin = t.

template <typename R>
__global__ void relayout_kernel(DevGraph<R> nw, RelayoutSrc<R> o, int phase) {
    const int F1 = nw.n_f, F0 = o.n_f;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < F1; f += gridDim.x * blockDim.x) {
        const int src = o.src_f[f];
        if (phase == 0) {
            if (src >= 0) {
                for (int i = 0; i < 9; ++i) nw.x0[(size_t)i * F1 + f] = o.x0[(size_t)i * F0 + src];
            } else {
                const int m = nw.fm[f];
                for (int i = 0; i < 6; ++i) nw.x0[(size_t)i * F1 + f] = R(0);
                for (int i = 0; i < 3; ++i)
                    nw.x0[(size_t)(6 + i) * F1 + f] = m < o.n_lm ? o.lm_bel[(size_t)m * LBEL + 9 + i] : R(0);
            }
            continue;
        }
        const int slot = nw.kpos[f];
        R* mk_cur = (o.t & 1) ? nw.mk2 : nw.mk;
        R* mk_oth = (o.t & 1) ? nw.mk : nw.mk2;
        if (src >= 0) {
            const int os = o.kpos[src];
            nw.tlin[f] = o.tlin[src];
            for (int i = 0; i < NML; ++i) nw.ml[(size_t)i * F1 + f] = o.ml[(size_t)i * F0 + src];
            for (int i = 0; i < NLIN; ++i) nw.lin[(size_t)i * F1 + f] = o.lin[(size_t)i * F0 + src];
            for (int i = 0; i < HIST; ++i) nw.hist[(size_t)i * F1 + f] = o.hist[(size_t)i * F0 + src];
            for (int i = 0; i < KJ; ++i) nw.kj[(size_t)slot * KJ + i] = o.kj[(size_t)os * KJ + i];
            for (int i = 0; i < KREC; ++i) {
                mk_cur[(size_t)slot * KREC + i] = o.mk_cur[(size_t)os * KREC + i];
                mk_oth[(size_t)slot * KREC + i] = o.mk_oth[(size_t)os * KREC + i];
            }
        } else {
            nw.tlin[f] = o.t;
            for (int i = 0; i < NML; ++i) nw.ml[(size_t)i * F1 + f] = R(0);
            for (int i = 0; i < NLIN; ++i) nw.lin[(size_t)i * F1 + f] = R(0);
            for (int i = 0; i < HIST; ++i) nw.hist[(size_t)i * F1 + f] = 0.0f;
            for (int i = 0; i < KJ; ++i) nw.kj[(size_t)slot * KJ + i] = R(0);
            for (int i = 0; i < KREC; ++i) {
                mk_cur[(size_t)slot * KREC + i] = R(0);
                mk_oth[(size_t)slot * KREC + i] = R(0);
            }
        }
    }
}

template <typename R>
cudaError_t launch_relayout(const DevGraph<R>& nw, const RelayoutSrc<R>& o, int phase, cudaStream_t s) {
    const int blocks = std::max(1, std::min((nw.n_f + 255) / 256, 1024));
    relayout_kernel<R><<<blocks, 256, 0, s>>>(nw, o, phase);
    return cudaGetLastError();
}

#define GBP_INSTANTIATE(R)                                                                                 \
    template cudaError_t launch_factor<R>(const DevGraph<R>&, const KParams<R>&, cudaStream_t, int, bool, int); \
    template cudaError_t launch_capture_messages<R>(const DevGraph<R>&, int, R*, cudaStream_t);            \
    template cudaError_t launch_tile_index<R>(const DevGraph<R>&, int, int4*, cudaStream_t);               \
    template cudaError_t launch_init<R>(const DevGraph<R>&, const KParams<R>&, cudaStream_t);              \
    template cudaError_t launch_belief<R>(const DevGraph<R>&, const KParams<R>&, cudaStream_t, bool);      \
    template cudaError_t launch_problem_metrics<R>(const DevGraph<R>&, const KParams<R>&, const int32_t*, int, double*, cudaStream_t); \
    template int persistent_grid<R>(const DevGraph<R>&, int, int);                                         \
    template cudaError_t launch_persistent<R>(const DevGraph<R>&, const KParams<R>&, int, float, int, int, cudaStream_t, int, int); \
    template cudaError_t launch_prior<R>(const DevGraph<R>&, const KParams<R>&, R*, R*, R*, R*, const R*, R*, cudaStream_t); \
    template cudaError_t launch_init_new<R>(const DevGraph<R>&, const KParams<R>&, int, int, cudaStream_t); \
    template cudaError_t launch_metrics<R>(const DevGraph<R>&, const KParams<R>&, double*, int, double*, cudaStream_t); \
    template cudaError_t launch_residuals<R>(const DevGraph<R>&, const KParams<R>&, const int32_t*, double*, cudaStream_t); \
    template cudaError_t launch_means<R>(const DevGraph<R>&, bool, double*, double*, int32_t*, cudaStream_t); \
    template cudaError_t launch_split_records<R>(const DevGraph<R>&, int, int, int, const int32_t*, float*, cudaStream_t); \
    template cudaError_t launch_relayout<R>(const DevGraph<R>&, const RelayoutSrc<R>&, int, cudaStream_t);

GBP_INSTANTIATE(float)
GBP_INSTANTIATE(double)

}  // namespace gbp
