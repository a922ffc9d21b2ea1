// gbp_noalloc.cu -- average reprojection error of caller-owned device arrays
// without any device allocation.
//
// This is a variant of the library's metrics reduction (per-observation
// reprojection error, per-block partial sums, one fixed-order final sum) for
// callers that cannot allocate device memory at the point where they need
// the number: for example a real-time tracking loop that reserves all of its
// device memory at start-up and must never hit cudaMalloc's device-wide
// synchronisation and unbounded latency afterwards, or a host application
// whose own allocator owns every byte of device memory.  Such callers pass
// their inputs and an output slot; the per-block partials live in the
// fixed-size device array below, which every GPU that loads the library keeps
// until the process exits.
#include "../../include/gbp.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

namespace {

constexpr int NOALLOC_BLOCK = 256;
constexpr int NOALLOC_MAX_BLOCKS = GBP_NOALLOC_MAX_OBS / NOALLOC_BLOCK;
constexpr int NOALLOC_MAX_DEVICES = 64;
constexpr int ARE_BLOCKS = 1216;   // 8 per SM of 152: every warp slot of the chip
static_assert(ARE_BLOCKS <= NOALLOC_MAX_BLOCKS, "scratch slots");

// Partial sums: slot b holds block b's error sum, slot NOALLOC_MAX_BLOCKS + b
// its count.  Shared by every call on a device; each call overwrites exactly
// the slots it later reads.
static __device__ __align__(256) double g_are_scratch[2 * NOALLOC_MAX_BLOCKS];

// Device address of g_are_scratch per device, looked up once per device.
// Several host threads may make their first call on a device at once: each
// looks the address up and stores the same value, so relaxed atomics suffice.
static std::atomic<double*> g_scratch_addr[NOALLOC_MAX_DEVICES];

// Bound: the FP64 pipe (one warp instruction per 16 cycles and SM), so the
// error is formed with as few FP64 operations as its definition allows.  With
// p the camera-frame point and c = uv - (cx, cy), the residual is d / p2 with
// d = c p2 - (fx p0, fy p1), and its length
//   |d| / p2 = A rsqrt(A p2^2),  A = |d|^2:
// one reciprocal square root in the place of two divisions and a square root
// (28 FP64 instructions an observation instead of ~70; each step is exact or
// rounds once, as before).  Where A p2^2 leaves the middle of the exponent
// range (a residual of 0, infinities, NaN) the divisions are taken.
// 2^20 observations: 68 us for both kernels, 129 us with the divisions, both
// counts in FP64 and 4096 partials (reading the inputs once takes 4 us).
__device__ __noinline__ double error_by_division(double fx, double fy, double cu, double cv, double p0, double p1, double p2) {
    const double du = cu - fx * p0 / p2, dv = cv - fy * p1 / p2;
    return sqrt(du * du + dv * dv);
}

__global__ void __launch_bounds__(NOALLOC_BLOCK)
are_partials_kernel(double fx, double fy, double cx, double cy, double z_min, int32_t n_kf,
                    const double* __restrict__ kf_Rt, int32_t n_lm, const double* __restrict__ lm_xyz, int32_t n_obs,
                    const int32_t* __restrict__ obs_kf, const int32_t* __restrict__ obs_lm,
                    const double* __restrict__ obs_uv, double* scratch) {
    __shared__ double red[NOALLOC_BLOCK];
    __shared__ int count;
    const int tid = threadIdx.x;
    if (tid == 0) count = 0;
    double sum = 0.0;
    int n = 0;
    for (int i = blockIdx.x * NOALLOC_BLOCK + tid; i < n_obs; i += gridDim.x * NOALLOC_BLOCK) {
        // an observation whose indices are out of range is left out, never read through
        const int k = obs_kf[i], m = obs_lm[i];
        if (k < 0 || k >= n_kf || m < 0 || m >= n_lm) continue;
        const double* Rt = kf_Rt + 12 * (size_t)k;
        const double* X = lm_xyz + 3 * (size_t)m;
        const double x = X[0], y = X[1], z = X[2];
        const double p0 = fma(Rt[0], x, fma(Rt[1], y, fma(Rt[2], z, Rt[9])));
        const double p1 = fma(Rt[3], x, fma(Rt[4], y, fma(Rt[5], z, Rt[10])));
        const double p2 = fma(Rt[6], x, fma(Rt[7], y, fma(Rt[8], z, Rt[11])));
        if (!(p2 >= z_min)) continue;
        const double cu = obs_uv[2 * (size_t)i] - cx, cv = obs_uv[2 * (size_t)i + 1] - cy;
        const double du = fma(cu, p2, -(fx * p0)), dv = fma(cv, p2, -(fy * p1));
        const double A = fma(du, du, dv * dv), D = A * (p2 * p2);
        // exponent of D within 2^-900 .. 2^900
        const bool mid = unsigned(__double2hiint(D) - 0x07b00000) < 0x70800000u;
        sum += mid ? A * rsqrt(D) : error_by_division(fx, fy, cu, cv, p0, p1, p2);
        ++n;
    }
    red[tid] = sum;
    __syncthreads();
    n = __reduce_add_sync(0xffffffffu, n);
    if ((tid & 31) == 0 && n) atomicAdd(&count, n);
    for (int st = NOALLOC_BLOCK / 2; st > 0; st >>= 1) {
        if (tid < st) red[tid] += red[tid + st];
        __syncthreads();
    }
    if (tid == 0) {
        scratch[blockIdx.x] = red[0];
        scratch[NOALLOC_MAX_BLOCKS + blockIdx.x] = double(count);
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launched while the partials are formed (programmatic dependent launch),
// waits for them.
__global__ void __launch_bounds__(NOALLOC_BLOCK) are_finish_kernel(const double* scratch, int nb, double* out) {
    __shared__ double red[2][NOALLOC_BLOCK];
    const int tid = threadIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double s = 0.0, c = 0.0;
    for (int b = tid; b < nb; b += NOALLOC_BLOCK) {
        s += scratch[b];
        c += scratch[NOALLOC_MAX_BLOCKS + b];
    }
    red[0][tid] = s;
    red[1][tid] = c;
    __syncthreads();
    for (int st = NOALLOC_BLOCK / 2; st > 0; st >>= 1) {
        if (tid < st) {
            red[0][tid] += red[0][tid + st];
            red[1][tid] += red[1][tid + st];
        }
        __syncthreads();
    }
    if (tid == 0) {
        out[0] = red[1][0] > 0.0 ? red[0][0] / red[1][0] : 0.0;
        out[1] = red[1][0];
    }
}

}  // namespace

extern "C" gbp_status gbp_reprojection_error_noalloc(const gbp_intrinsics* intr, double z_min, int32_t n_kf,
                                                     const double* kf_Rt, int32_t n_lm, const double* lm_xyz,
                                                     int32_t n_obs, const int32_t* obs_kf, const int32_t* obs_lm,
                                                     const double* obs_uv, double* out, void* cuda_stream) {
    if (!intr || !out || n_obs < 0 || n_kf < 0 || n_lm < 0) return GBP_EINVAL;
    if (n_obs > GBP_NOALLOC_MAX_OBS) return GBP_EINVAL;   // more observations than the scratch array holds
    if (n_obs > 0 && (!kf_Rt || !lm_xyz || !obs_kf || !obs_lm || !obs_uv)) return GBP_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return GBP_ECUDA;
    // one-time set-up on this device: host code needs the scratch array's
    // device address (its name in host code is only a host-side stand-in)
    double* scratch = g_scratch_addr[dev].load(std::memory_order_relaxed);
    if (!scratch) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_are_scratch) != cudaSuccess || !p) return GBP_ECUDA;
        scratch = static_cast<double*>(p);
        g_scratch_addr[dev].store(scratch, std::memory_order_relaxed);
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    (void)cudaGetLastError();   // an error left by an unrelated earlier call is not this call's to report
    // at most ARE_BLOCKS blocks walk the observations: few partials to add up at the end
    const int nb = std::min((n_obs + NOALLOC_BLOCK - 1) / NOALLOC_BLOCK, ARE_BLOCKS);
    if (nb > 0)
        are_partials_kernel<<<nb, NOALLOC_BLOCK, 0, s>>>(intr->fx, intr->fy, intr->cx, intr->cy, z_min, n_kf, kf_Rt,
                                                         n_lm, lm_xyz, n_obs, obs_kf, obs_lm, obs_uv, scratch);
    if (cudaGetLastError() != cudaSuccess) return GBP_ECUDA;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(NOALLOC_BLOCK);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, are_finish_kernel, (const double*)scratch, nb, out) != cudaSuccess) return GBP_ECUDA;
    return cudaGetLastError() == cudaSuccess ? GBP_OK : GBP_ECUDA;
}
