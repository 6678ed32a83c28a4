// Shared by the local GP kernels (gp_local.cu in FP64, gp_fixed.cu in fixed
// point): block reductions, the design of a location, and the MLE's outputs.
#pragma once
#include <cuda_runtime.h>

#include "device_util.cuh"
#include "lagp_internal.h"

// Status of a location that the fixed-point kernels leave to the FP64 ones.
// The MLE leaves FX_REDO - k where the first k iterations hold: d is then the
// point that they came to.
constexpr int FX_REDO = -1;

struct MleOut {
    double *llik, *dllik, *d2llik;
    int32_t *iters, *status;
};

// gp_fixed.cu.  counters: zeroed words, one a size class (at most 8); redo:
// zeroed word that counts the locations left (status FX_REDO or below, outputs
// not final).  ws: gp_fixed_workspace bytes (the MLE's squared
// distances, a CTA's own; less than the FP64 kernel's matrices).
bool gp_fixed_supported(lagp_ctx *ctx, const GpArgs &a, bool mle);
size_t gp_fixed_workspace(lagp_ctx *ctx, const GpArgs &a);
lagp_status launch_predict_fixed(lagp_ctx *ctx, const GpArgs &a, const double *d, double *mean, double *s2,
                                 double *df, int32_t *status, int *counters, int *redo);
lagp_status launch_mle_fixed(lagp_ctx *ctx, const GpArgs &a, double *d, double dmin, double dmax, int32_t max_iter,
                             const MleOut &o, unsigned long long *work, double *ws, int *counters, int *redo);

namespace {

constexpr int GP_THREADS = 128;
constexpr int GP_WARPS = GP_THREADS / 32;

struct Blk {
    int tid, lane, warp;
};

// Block sums of NV values at once: warp sums, then one warp adds the warps'
// partials (not every thread); three barriers for all NV.
template <int NV, int T = GP_THREADS>
__device__ void block_sums(double (&v)[NV], const Blk &b) {
    __shared__ double part[T / 32 * NV], tot[NV];
#pragma unroll
    for (int i = 0; i < NV; i++) v[i] = warp_sum(v[i]);
    __syncthreads();  // earlier readers of part / tot are done
    if (b.lane == 0)
#pragma unroll
        for (int i = 0; i < NV; i++) part[b.warp * NV + i] = v[i];
    __syncthreads();
    if (b.warp == 0 && b.lane < NV) {
        double t = 0.0;
        for (int w = 0; w < T / 32; w++) t += part[w * NV + b.lane];
        tot[b.lane] = t;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; i++) v[i] = tot[i];
}

// Validate a location and load its design; returns the per-location status.
template <int T = GP_THREADS>
__device__ int load_design(const GpArgs &a, int64_t loc, int nm, const double *dptr, double *xd,
                           double *y, int *flag, const Blk &b) {
    if (b.tid == 0) *flag = LAGP_OK;
    __syncthreads();
    const double d = dptr ? dptr[loc] : 1.0;
    if (b.tid == 0 && (nm < 1 || nm > a.nmax || !(d > 0.0) || !isfinite(d))) *flag = LAGP_EINVAL;
    __syncthreads();
    if (*flag != LAGP_OK) return *flag;
    const int32_t *s = a.sel + loc * a.nmax;
    for (int t = b.tid; t < nm; t += T) {
        int32_t r = s[t];
        if (r < 0 || r >= a.N) *flag = LAGP_EINVAL;
    }
    __syncthreads();
    if (*flag != LAGP_OK) return *flag;
    for (int e = b.tid; e < nm * a.p; e += T) {
        int t = e / a.p, i = e - t * a.p;
        xd[e] = load_coord64(a.X, s[t], a.p, i, a.dtype);
    }
    for (int t = b.tid; t < nm; t += T)
        y[t] = a.dtype == LAGP_F64 ? static_cast<const double *>(a.Y)[s[t]]
                                   : (double)static_cast<const float *>(a.Y)[s[t]];
    __syncthreads();
    return LAGP_OK;
}

__device__ double sqd(const double *u, const double *v, int p) {
    double s = 0.0;
    for (int i = 0; i < p; i++) {
        double df = u[i] - v[i];
        s = fma(df, df, s);
    }
    return s;
}

}  // namespace
