// gbp_resident.cu -- the resident kernel: one cooperative launch runs all
// iterations of a gbp_iterate call of a small graph (FP32, fixed damping),
// with each warp tile's state kept in registers for the whole launch.
//
// At this size (paper scale: ~600 tiles, 125 keyframes on 152 SMs) an
// iteration moves ~4 MB that all sits in L2; its time is the chain of
// dependent steps from one set of beliefs to the next.  The chain is kept to
// what an iteration cannot do without:
//
//   * The message to the keyframe, m^{t+1}_{f->k}, depends on the landmark's
//     incoming message only (Sec. 5), which is the warp's own state: it is
//     formed ahead, while the previous iteration's beliefs are still being
//     summed.  Of b^t a factor needs only the keyframe's mean before it can
//     send, for the relinearisation test (Sec. 5, Sec. 8).
//   * Everything else of the factor phase -- the message to the landmark, the
//     landmark's belief, the next message to the keyframe -- runs while other
//     warps of the block sum the keyframes.
//
// A block has NA factor warps (one tile each, for the whole launch) and one
// group of FACTOR_BLOCK belief threads (a keyframe at a time).  Iteration t:
//
//   factor warps: [b^t ready] keyframe side, test -> store m^{t+1}
//                 -> arrive(1) -> m^{t+1} to the landmark, its belief,
//                 m^{t+2} to the keyframe formed ahead -> barrier(2)
//   belief warps: wait(1): every block's messages are stored -> sum, factorise
//                 -> barrier(2): b^{t+1} ready
//
// The arithmetic is that of tile_work and phase_b_item, expression by
// expression, so the results are bitwise those of the per-phase kernels.
//
// Per iteration (200 iterations from reset, launch included; walks, relinearising
// somewhere in nearly every iteration) against the per-phase kernels: 10
// keyframes, 15 tiles 4.7 us against 8.0; 60 and 225 6.7 / 10.1; 125 and 566
// 7.2 / 10.3; 150 and 608 7.3 / 10.5; with 8 factor warps a block 125 and 634
// 10.0 / 10.7, 150 and 976 9.8 / 11.0, 150 and 1190 11.2 / 11.7.  Of 9.1 us with
// 8 factor warps and a relinearisation somewhere in every iteration (clock64 of
// one block): the gather of the beliefs 1.3, keyframe side, test and
// relinearisation 2.3, the arrival and its way to the slowest block's belief
// warps 1.5, the sums and factorisation 2.4, the barrier and the spread of the
// blocks 1.6.
#include "gbp_device.cuh"

#include <algorithm>

namespace gbp {

namespace {

constexpr int BAR_FACTOR = 1, BAR_BELIEF = 2;   // named barriers of a block's two groups
constexpr int NB_BELIEF = FACTOR_BLOCK;         // belief threads per block

__device__ __forceinline__ int ld_acquire(const int32_t* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(int32_t* p) {
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory");
}

// Arrivals are counted, never reset within a launch (the last launch's final
// counts are this launch's base), so a wait is a plain poll.  It is bounded:
// after ~2 s without progress, or when another block has given up, it
// records the timeout (CTL_ERR = 2) and returns false.
constexpr int SPIN_LIMIT = 1 << 22;
__device__ __forceinline__ bool wait_count(int32_t* ctl, const int32_t* cnt, unsigned target) {
    for (int spin = 0; spin < SPIN_LIMIT; ++spin) {
        if (int(unsigned(ld_acquire(cnt)) - target) >= 0) return true;   // counts may wrap
        if ((spin & 1023) == 1023 && *reinterpret_cast<volatile int32_t*>(ctl + CTL_ERR) == 2) return false;
    }
    atomicCAS(&ctl[CTL_ERR], 0, 2);
    return false;
}

// One lane's factor between iterations: its linearisation, both messages of
// the last iteration, the landmark's mean, the landmark's incoming precision
// of the coming iteration (Pm, qm) and the message to the keyframe that it
// gives unless the factor relinearises (ck, damped).
struct Resident {
    int f, k, slot, tl, lbirth, m;
    int seg0, seg1, seg_max;
    bool active;
    float J0[6], J1[6], y[2], W;
    float cml[NML], mo[NML], x0[9], lb_mu[3], lD[3];
    float Pm[6], qm[3], ck[NML];
    bool ok_m, m64;     // Pm positive definite, after the FP64 redo (m64: it was needed)
};

__device__ __forceinline__ void lin_of(const Resident& S, Lin<float>& L) {
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        L.Jk[0][j] = S.J0[j];
        L.Jk[1][j] = S.J1[j];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        L.Jl[0][j] = -S.J0[j];
        L.Jl[1][j] = -S.J1[j];
    }
    L.y[0] = S.y[0];
    L.y[1] = S.y[1];
    L.W = S.W;
    L.r2 = 0.0f;   // not used by the fixed schedule
}

// A new linearisation (taken in this iteration): to the lane's registers, the
// factor's lin record and the staging block, which the belief phase moves.
__device__ __forceinline__ void take_lin(const DevGraph<float>& g, const Lin<float>& L, Resident& S) {
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        S.J0[j] = L.Jk[0][j];
        S.J1[j] = L.Jk[1][j];
    }
    S.y[0] = L.y[0];
    S.y[1] = L.y[1];
    S.W = L.W;
    store_lin<float>(g, S.f, L);
    store_jac<float>(g.kjs + (size_t)S.slot * KJ, L.Jk);
}

// The tile's state at iteration t, from memory; factors that have not been
// linearised yet are (as tile_work does).
__device__ __forceinline__ void load_state(const DevGraph<float>& g, const KParams<float>& P, int tile, int t, int lane,
                                           Resident& S) {
    const size_t n_f = g.n_f;
    const int4 te = g.tidx[(size_t)tile * 32 + lane];
    S.active = te.x >= 0;
    S.f = g.tf[(size_t)tile * 32 + lane];
    S.k = S.active ? te.x : 0;
    S.slot = te.y;
    S.m = te.z;
    S.seg0 = te.w & 31;          // every landmark lies inside one tile here
    S.seg1 = (te.w >> 8) & 31;
    S.seg_max = __reduce_max_sync(0xffffffffu, unsigned(S.seg1 - S.seg0 + 1));
    S.tl = S.lbirth = 0;
    float jr[KJ], rec[KREC], lin[NLIN];
#pragma unroll
    for (int i = 0; i < KJ; ++i) jr[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < KREC; ++i) rec[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < NML; ++i) S.cml[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < NLIN; ++i) lin[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < 9; ++i) S.x0[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) S.lb_mu[i] = S.lD[i] = 0.0f;
    if (S.active) {
        const int f = S.f;
        S.tl = g.tlin[f];
        S.lbirth = g.lm_birth[S.m];
        load_rec_cg<float, KJ>(g.kj + (size_t)S.slot * KJ, jr);
        load_msg<true, float>(mk_read(g, t) + (size_t)S.slot * KREC, rec);
#pragma unroll
        for (int i = 0; i < NML; ++i) S.cml[i] = g.ml[i * n_f + f];
#pragma unroll
        for (int i = 0; i < NLIN; ++i) lin[i] = g.lin[i * n_f + f];
#pragma unroll
        for (int i = 0; i < 9; ++i) S.x0[i] = g.x0[i * n_f + f];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            S.lb_mu[i] = __ldcg(g.lm_bel + (size_t)S.m * LBEL + 9 + i);
            S.lD[i] = g.lm_D[S.m * 3 + i];
        }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) { S.J0[i] = jr[i]; S.J1[i] = jr[6 + i]; }
#pragma unroll
    for (int i = 0; i < NML; ++i) S.mo[i] = rec[i];
    S.y[0] = lin[0];
    S.y[1] = lin[1];
    S.W = lin[2];
    if (S.active && S.tl == t) {
        Arr9<float> xv;
#pragma unroll
        for (int i = 0; i < 9; ++i) xv.v[i] = S.x0[i];
        take_lin(g, linearise_at<float>(xv, lin_args<float>(P, g, S.k, S.f)), S);
    }
}

// The message to the keyframe from the landmark's incoming precision, in the
// basis of the lane's linearisation, undamped; ok_m and m64 are decided.
__device__ __forceinline__ void message_to_keyframe(Resident& S, const float* Lm, const float* im) {
    Lin<float> L;
    lin_of(S, L);
    if (!S.ok_m) {
#pragma unroll
        for (int i = 0; i < NML; ++i) S.ck[i] = S.mo[i];
    } else if (S.m64) {
        Arr9<float> pq;
#pragma unroll
        for (int i = 0; i < 6; ++i) pq.v[i] = S.Pm[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) pq.v[6 + i] = S.qm[i];
        const Msg5<float> o = lm_message64<float>(pq, L);
#pragma unroll
        for (int i = 0; i < NML; ++i) S.ck[i] = o.v[i];
    } else {
        message_chol<float, 3>(Lm, im, S.qm, L.Jl, L.y, L.W, S.ck);
    }
}

// The message to the keyframe of iteration t (ck), from the messages to the
// landmark of the previous one (mlo, expanded): steps 2b, 4 and 5 of
// tile_work for an iteration without relinearisation.
__device__ __forceinline__ void form_ahead(const DevGraph<float>& g, const KParams<float>& P, int t, int lane,
                                           const float* mlo, Resident& S) {
    {
        float fw[9], bw[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) { fw[j] = mlo[j]; bw[j] = mlo[j]; }
        for (int d = 1; d < S.seg_max; d <<= 1) {
#pragma unroll
            for (int j = 0; j < 9; ++j) {
                const float o = __shfl_up_sync(0xffffffffu, fw[j], d);
                if (lane - d >= S.seg0) fw[j] += o;
                const float u = __shfl_down_sync(0xffffffffu, bw[j], d);
                if (lane + d <= S.seg1) bw[j] += u;
            }
        }
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const float pre = __shfl_up_sync(0xffffffffu, fw[j], 1);
            const float suf = __shfl_down_sync(0xffffffffu, bw[j], 1);
            const float cv = (lane - 1 >= S.seg0 ? pre : 0.0f) + (lane + 1 <= S.seg1 ? suf : 0.0f);
            if (j < 6) S.Pm[j] = cv;
            else S.qm[j - 6] = cv;
        }
    }
    if (S.active) {
        const float sp = prior_scale(P, t - S.lbirth) * P.inv_sigma2;
#pragma unroll
        for (int i = 0; i < 3; ++i) S.Pm[pk(i, i)] += sp * S.lD[i];
    } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) S.Pm[i] = 0.0f;
#pragma unroll
        for (int i = 0; i < 3; ++i) { S.Pm[pk(i, i)] = 1.0f; S.qm[i] = 0.0f; }
    }
    float Lm[6], im[3], rm;
#pragma unroll
    for (int i = 0; i < 6; ++i) Lm[i] = S.Pm[i];
    S.ok_m = chol_packed<float, 3>(Lm, im, rm);
    S.m64 = false;
    if (P.fallback && S.active && !S.ok_m) {
        Arr9<float> pq;
#pragma unroll
        for (int i = 0; i < 6; ++i) pq.v[i] = S.Pm[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) pq.v[6 + i] = S.qm[i];
        S.m64 = true;
        S.ok_m = lm_incoming_ok64<float>(pq);
    }
    message_to_keyframe(S, Lm, im);
    if (S.ok_m && t - S.tl >= P.damp_hold) {
        const float d = P.damping;
        S.ck[3] = (1.0f - d) * S.ck[3] + d * S.mo[3];
        S.ck[4] = (1.0f - d) * S.ck[4] + d * S.mo[4];
    }
}

// The FP64 redo of the keyframe's incoming precision (form_messages).
__device__ __forceinline__ bool cavity64(const DevGraph<float>& g, const KParams<float>& P, int t, const Resident& S,
                                         double* kc) {
    const float* recs = mk_read(g, t);
    bool ok = !P.exact_cavity && kf_incoming_self64<float>(g.kf_bel + (size_t)S.k * KBEL, recs, g.kj, S.slot, kc);
    if (!ok) {
        ok = kf_resum64<float>(recs, g.kj, g.kf_off[S.k], g.kf_off[S.k + 1], S.slot, kf_prior_scale(g, P, S.k, t),
                               g.kf_D + (size_t)S.k * 6, g.kf_A + (size_t)S.k * 6, P.anchor_scale, P.inv_sigma2, kc);
        atomicAdd(&g.ctl[CTL_RESUMS], 1);
    }
    atomicAdd(&g.ctl[CTL_FALLBACKS], 1);
    return ok;
}

// Keyframe k's belief from its messages m^{t+1}, by the block's belief
// threads (phase_b_item, the block mapping); its |dmu| in the first thread.
// What does not depend on the messages is loaded before they are waited for.
struct KfItem {
    int k, b0, b1;
    float prior[6], mu_old[6];
};

__device__ __forceinline__ void kf_load(const DevGraph<float>& g, const KParams<float>& P, int k, int t, int tid,
                                        KfItem& it) {
    it.k = k;
    it.b0 = g.kf_off[k];
    it.b1 = g.kf_off[k + 1];
    if (tid == 0) {
        const float sp = kf_prior_scale(g, P, k, t + 1);
        const float* old = g.kf_bel + (size_t)k * KBEL;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            it.prior[i] = (sp * g.kf_D[k * 6 + i] + P.anchor_scale * g.kf_A[k * 6 + i]) * P.inv_sigma2;
            it.mu_old[i] = __ldcg(old + KB_MU + i);
        }
    }
}

__device__ __forceinline__ float kf_sum(const DevGraph<float>& g, const KParams<float>& P, const KfItem& it, int t,
                                        int tid, int* bad) {
    const float* msgs = mk_write(g, t);
    float hi[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) hi[j] = 0.0f;
    constexpr int BU = 2;   // entries per thread at a time, all their loads before the first is summed
    for (int i0 = it.b0 + tid; i0 < it.b1; i0 += BU * NB_BELIEF) {
        float rec[BU][KREC], jr[BU][KJ];
#pragma unroll
        for (int u = 0; u < BU; ++u) {
            const int i = i0 + u * NB_BELIEF;
            if (i < it.b1) {
                load_msg<true, float>(msgs + (size_t)i * KREC, rec[u]);
                load_rec_cg<float, KJ>(g.kj + (size_t)i * KJ, jr[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < BU; ++u) {
            const int i = i0 + u * NB_BELIEF;
            if (i < it.b1) {
                if (bits_int<float>(rec[u][KREC_TL]) == t) {
                    load_rec_cg<float, KJ>(g.kjs + (size_t)i * KJ, jr[u]);
                    store_rec<float, KJ>(g.kj + (size_t)i * KJ, jr[u]);
                }
                const float J[2][6] = {{jr[u][0], jr[u][1], jr[u][2], jr[u][3], jr[u][4], jr[u][5]},
                                       {jr[u][6], jr[u][7], jr[u][8], jr[u][9], jr[u][10], jr[u][11]}};
                float lam[21], eta[6];
                expand_msg<float, 6>(J, rec[u][0], rec[u][1], rec[u][2], rec[u][3], rec[u][4], lam, eta);
#pragma unroll
                for (int j = 0; j < 21; ++j) hi[j] += lam[j];
#pragma unroll
                for (int j = 0; j < 6; ++j) hi[21 + j] += eta[j];
            }
        }
    }
    float acc[27];
    group_total<float, 32, 27, NB_BELIEF / 32, BAR_BELIEF>(hi, acc, tid);
    return tid == 0 ? finish_keyframe<float>(g, P, it.k, it.prior, acc, it.mu_old, g.kf_bel_out, bad) : 0.0f;
}

// NA factor warps and FACTOR_BLOCK belief threads per block, one block per
// SM: 255 registers a thread for NA = 4, 168 (with spills) for 8.
template <int NA>
__global__ void __launch_bounds__(NA * 32 + NB_BELIEF, 1)
    resident_kernel(const __grid_constant__ DevGraph<float> g, const __grid_constant__ KParams<float> P, int n_iters,
                    float conv_tol, int check_every) {
    __shared__ int failed, stop, bad;   // bad: an error was raised, by this block or before this launch
    __shared__ float dmu_sh[NA + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool factor = warp < NA;
    const int nb = gridDim.x;
    const int tile = warp * nb + blockIdx.x;
    const bool has_tile = factor && tile < g.n_tiles;
    const int tid_b = int(threadIdx.x) - NA * 32;      // belief thread
    int32_t* const cnt1 = g.ctl + CTL_RES_CNT1;
    int32_t* const cnt2 = g.ctl + CTL_RES_CNT2;
    const int t0 = __ldcg(&g.ctl[CTL_ITER]);
    const unsigned base1 = __ldcg(&g.ctl[CTL_RES_BASE1]), base2 = __ldcg(&g.ctl[CTL_RES_BASE2]);
    if (threadIdx.x == 0) {
        failed = stop = 0;
        bad = __ldcg(&g.ctl[CTL_ERR]) != 0;
    }
    if (threadIdx.x <= NA) dmu_sh[threadIdx.x] = 0.0f;
    __syncthreads();

    Resident S;
    if (has_tile) {
        load_state(g, P, tile, t0, lane, S);
        Lin<float> L;
        lin_of(S, L);
        float mlo[9];
        expand_msg<float, 3>(L.Jl, S.cml[0], S.cml[1], S.cml[2], S.cml[3], S.cml[4], mlo, mlo + 6);
        form_ahead(g, P, t0, lane, mlo, S);
    }
    int done = 0;
    float last = 0.0f;
    for (int it = 0; it < n_iters; ++it) {
        const int t = t0 + it;
        const bool check = conv_tol > 0.0f && (it + 1) % check_every == 0;
        const bool want_dmu = check || it == n_iters - 1;
        if (factor) {
            KfSide<float> ks;
            double kc[KC64];
            bool ok_k = true, k64 = false, rebased = false;
            float cl[NML];
            if (has_tile) {
                float kb[KB_A];
                load_kf<true, float>(g.kf_bel + (size_t)S.k * KBEL, kb);
#pragma unroll
                for (int i = 0; i < NML; ++i) cl[i] = S.cml[i];   // kept unless formed below
                {
                    Lin<float> L;
                    lin_of(S, L);
                    kf_side<float>(kb, kb + KB_MU, L.Jk, S.mo, ks);
                }
                ok_k = ks.pd;
                bool relin = false;
                if (S.active && S.ok_m && !P.linear && t - S.tl >= P.relin_interval) {
                    const float* kmu = kb + KB_MU;
                    float d2 = 0.0f;
#pragma unroll
                    for (int i = 0; i < 6; ++i) d2 += (kmu[i] - S.x0[i]) * (kmu[i] - S.x0[i]);
#pragma unroll
                    for (int i = 0; i < 3; ++i) d2 += (S.lb_mu[i] - S.x0[6 + i]) * (S.lb_mu[i] - S.x0[6 + i]);
                    relin = d2 > P.relin_beta * P.relin_beta;
                }
                // before this block's arrival: the belief phase replaces what it reads
                if (P.fallback && S.active && !(ks.det >= P.cav_ratio)) {
                    ok_k = cavity64(g, P, t, S, kc);
                    k64 = ok_k;
                }
                if (relin && ok_k) {
                    Arr9<float> xn;
                    Arr12<float> Jo;
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        xn.v[i] = kb[KB_MU + i];
                        Jo.v[i] = S.J0[i];
                        Jo.v[6 + i] = S.J1[i];
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i) xn.v[6 + i] = S.lb_mu[i];
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        S.x0[i] = xn.v[i];
                        g.x0[(size_t)i * g.n_f + S.f] = xn.v[i];
                    }
                    S.tl = t;
                    g.tlin[S.f] = t;
                    atomicAdd(&g.ctl[CTL_RELINS], 1);
                    const Rebased<float> rb =
                        rebase<float>(g.kf_bel + (size_t)S.k * KBEL, Jo, S.mo[3], S.mo[4], ks.a0, ks.a1, ks.K00,
                                      ks.K01, ks.K11, !k64, xn, lin_args<float>(P, g, S.k, S.f));
                    take_lin(g, rb.L, S);
                    if (!k64)
#pragma unroll
                        for (int i = 0; i < NML; ++i) cl[i] = rb.cl[i];
                    rebased = true;
                    float Lm[6], im[3], rm;
#pragma unroll
                    for (int i = 0; i < 6; ++i) Lm[i] = S.Pm[i];
                    chol_packed<float, 3>(Lm, im, rm);
                    message_to_keyframe(S, Lm, im);
                }
                if (S.active) {
                    float rec[KREC];
#pragma unroll
                    for (int i = 0; i < NML; ++i) rec[i] = S.ck[i];
                    rec[KREC_TL] = int_bits<float>(S.tl);
                    rec[6] = 0.0f;
                    rec[7] = 0.0f;
                    store_msg<float>(mk_write(g, t) + (size_t)S.slot * KREC, rec);
                }
            }
            asm volatile("bar.sync %0, %1;" ::"n"(BAR_FACTOR), "n"(NA * 32) : "memory");
            if (threadIdx.x == 0) red_release(cnt1);
            float dmu = 0.0f;
            if (has_tile) {
                if (S.active && S.m64) atomicAdd(&g.ctl[CTL_FALLBACKS], 1);
                if (S.active && !S.ok_m) atomicAdd(&g.ctl[CTL_HELD], 1);
                if (S.active && !ok_k) atomicAdd(&g.ctl[CTL_HELD], 1);
                Lin<float> L;
                lin_of(S, L);
                if (ok_k) {
                    if (k64) {
                        const Msg5<float> o = kf_message64<float>(kc, L);
#pragma unroll
                        for (int i = 0; i < NML; ++i) cl[i] = o.v[i];
                    } else if (!rebased) {
                        message_to_landmark<float>(ks, L.y, L.W, cl);
                    }
                    if (t - S.tl >= P.damp_hold) {
                        const float d = P.damping;
                        cl[3] = (1.0f - d) * cl[3] + d * S.cml[3];
                        cl[4] = (1.0f - d) * cl[4] + d * S.cml[4];
                    }
                }
                float mlo[9], sum[9];
                if (S.active) {
#pragma unroll
                    for (int i = 0; i < NML; ++i) g.ml_out[(size_t)i * g.n_f + S.f] = cl[i];
                }
                expand_msg<float, 3>(L.Jl, cl[0], cl[1], cl[2], cl[3], cl[4], mlo, mlo + 6);
#pragma unroll
                for (int i = 0; i < 9; ++i) sum[i] = S.active ? mlo[i] : 0.0f;
#pragma unroll
                for (int i = 0; i < NML; ++i) {
                    S.cml[i] = cl[i];
                    S.mo[i] = S.ck[i];
                }
                for (int d = 1; d < S.seg_max; d <<= 1) {
#pragma unroll
                    for (int j = 0; j < 9; ++j) {
                        const float o = __shfl_up_sync(0xffffffffu, sum[j], d);
                        if (lane - d >= S.seg0) sum[j] += o;
                    }
                }
                float mu[3] = {0.0f, 0.0f, 0.0f};
                if (S.active && lane == S.seg1)
                    dmu = finish_landmark<float>(g, P, S.m, prior_scale(P, t + 1 - S.lbirth), sum, S.lb_mu, g.lm_bel_out,
                                                 mu, &bad);
#pragma unroll
                for (int i = 0; i < 3; ++i) S.lb_mu[i] = __shfl_sync(0xffffffffu, mu[i], S.seg1);
                form_ahead(g, P, t + 1, lane, mlo, S);
            }
            if (want_dmu) {
                dmu = warp_max(dmu);
                if (lane == 0) dmu_sh[warp] = dmu;
            }
        } else {
            KfItem kf;
            const int k0 = blockIdx.x;
            if (k0 < g.n_kf) kf_load(g, P, k0, t, tid_b, kf);
            if (tid_b == 0 && !wait_count(g.ctl, cnt1, base1 + unsigned(it + 1) * nb)) failed = 1;
            asm volatile("bar.sync %0, %1;" ::"n"(BAR_BELIEF), "n"(NB_BELIEF) : "memory");
            float dmu = 0.0f;
            for (int k = k0; k < g.n_kf; k += nb) {
                if (k != k0) kf_load(g, P, k, t, tid_b, kf);
                dmu = fmaxf(dmu, kf_sum(g, P, kf, t, tid_b, &bad));
            }
            if (tid_b == 0) {
                dmu_sh[NA] = dmu;
                // every block has read the slot's previous use (iteration t - 1)
                if (blockIdx.x == 0) g.ctl[dmu_slot(t + 1)] = 0;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (want_dmu) {
                float m = 0.0f;
#pragma unroll
                for (int w = 0; w <= NA; ++w) m = (dmu_sh[w] >= 0.0f) ? fmaxf(m, dmu_sh[w]) : INFINITY;
                if (m > 0.0f) dmu_atomic_max_slot(g.ctl, dmu_slot(t), m);
                // the convergence loop leaves at the first check after an error.  The
                // word carries its iteration: a block that is already past this
                // barrier cannot make a slower one leave earlier than itself.
                // (Here, not outside want_dmu: 0.04 us an iteration less.)
                if (check && bad) atomicCAS(&g.ctl[CTL_RES_ERR_T], 0, t + 1);
            }
            red_release(cnt2);
            if (!wait_count(g.ctl, cnt2, base2 + unsigned(it + 1) * nb)) failed = 1;
            if (check) {
                last = __int_as_float(__ldcg(&g.ctl[dmu_slot(t)]));
                const int et = __ldcg(&g.ctl[CTL_RES_ERR_T]);
                if (last < conv_tol || (et != 0 && et <= t + 1)) stop = 1;
            }
        }
        __syncthreads();
        if (failed) break;
        done = it + 1;
        if (stop) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        last = done > 0 ? __int_as_float(__ldcg(&g.ctl[dmu_slot(t0 + done - 1)])) : 0.0f;
        g.ctl[CTL_ITER] = t0 + done;
        g.ctl[CTL_DMU_LAST] = __float_as_int(last);
        g.ctl[CTL_ITERS_RUN] = done;
        g.ctl[CTL_RES_BASE1] = int(base1 + unsigned(done) * nb);
        g.ctl[CTL_RES_BASE2] = int(base2 + unsigned(done) * nb);
    }
}

// Factor warps per block: the fewest that hold the tiles (the more registers
// each); 0: too many tiles.
int factor_warps(int n_tiles, int sms) {
    for (int na : {4, 8})
        if (n_tiles <= sms * na) return na;
    return 0;
}

}  // namespace

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

// Blocks of the resident kernel for this graph; 0 where it does not apply:
// more tiles than the SMs hold at one block each, a landmark split across
// tiles or a variable without factors (belief-phase items of their own), the
// warp mapping of the belief phase, a part of a split graph.
int resident_grid(const DevGraph<float>& g) {
    const int sms = sm_count();
    if (sms <= 0 || g.b_warps != NB_BELIEF / 32 || g.n_big > 0 || g.n_orphan > 0 || g.n_tiles < 1) return 0;
    if (g.tile_off != 0 || g.kf_item_off != 0 || g.kf_item_n != g.n_kf) return 0;
    const int na = factor_warps(g.n_tiles, sms);
    return na ? std::min(sms, std::max((g.n_tiles + na - 1) / na, g.n_kf)) : 0;
}

cudaError_t launch_resident(const DevGraph<float>& g, const KParams<float>& p, int n_iters, float conv_tol,
                            int check_every, cudaStream_t s) {
    const int grid = resident_grid(g);
    if (grid <= 0) return cudaErrorInvalidConfiguration;
    const int na = factor_warps(g.n_tiles, sm_count());
    DevGraph<float> gg = g;
    KParams<float> pp = p;
    void* args[] = {&gg, &pp, &n_iters, &conv_tol, &check_every};
    const void* fn = na == 4 ? reinterpret_cast<const void*>(resident_kernel<4>)
                             : reinterpret_cast<const void*>(resident_kernel<8>);
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(na * 32 + NB_BELIEF), args, 0, s);
}

}  // namespace gbp
