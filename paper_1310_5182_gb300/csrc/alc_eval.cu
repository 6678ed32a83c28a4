// The ALC criterion of Eq. (dxy) for many candidates at one location and a
// fixed design — the computation the paper times in Sec. 4.1 (one reference
// location, N' = 60,000 candidates, designs of n = 16..512).
//
// Given the design X_n and the location x:
//   prep   K_n = exp(-D/d) + g I, its Cholesky factor L (FP64), z = L^{-1} k_n(x),
//          1/diag(L); padded to a multiple of 32 rows with identity rows.
//   cands  per candidate c: u_c = L^{-1} k_n(x_c) by blocked forward
//          substitution, s_c = |u_c|^2 = k_c^T K_n^{-1} k_c,
//          q_c = z^T u_c = k_n(x)^T K_n^{-1} k_c, and
//          Delta_c = (K(x_c, x) - q_c)^2 / (1 + g - s_c)
//          (Eq. (dxy) with Eq. (piedef) after simplification).
// In FP64 the candidate kernel is one thread per candidate, 32-row blocks: the
// off-diagonal blocks L_IJ are staged in shared memory (read as broadcasts),
// the current block's 32 values live in registers, earlier solved blocks
// stream from a global panel W[i][c] (coalesced across the candidates).  Per
// candidate n^2/2 FP64 FMAs with every lane busy: the FP64 unit bounds it.
//
// For nuggets below 1 the substitution runs in 59-bit fixed point on the
// integer pipe instead (fx59.cuh): rows of L have norm < sqrt(2) and u_c is
// bounded by the same, so a product costs three multiply-adds, 12 cycles a
// warp instead of 64; the n exponentials of a candidate stay in FP64 and run
// beside them.  A candidate's covariances are scaled by the power of two that
// brings the largest near 1/8, so that far candidates keep their relative
// precision.  L comes from the fixed-point factorisation for n <= 128 (one
// CTA, 0.80 -> 0.23 ms at n = 128),
// else from the FP64 one.  What leaves the range is redone in FP64 by the
// conditional launches behind (one flag a candidate).  60,000 candidates,
// n = 128: 1.36 -> 0.48 ms, 2.16 -> 0.70 ms a call.
#include <cuda_runtime.h>

#include <algorithm>

#include "device_util.cuh"
#include "exp64.cuh"
#include "fx_chol.cuh"
#include "lagp_internal.h"

namespace {

constexpr int EV_THREADS = 128;  // candidates per CTA
constexpr int EV_B = 32;         // rows per block of the substitution
constexpr int PREP_THREADS = 256;

// One CTA: L (np x np, np = n rounded up to 32, identity padding), rd, z.
__global__ void __launch_bounds__(PREP_THREADS)
eval_prep_kernel(const void *X, int p, lagp_dtype dt, const double *x, const int32_t *design, int n,
                 int np, double d, double g, double *L, double *rd, double *z, int32_t *status,
                 const int *redo) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (redo && *redo == 0) return;  // (after the fixed-point kernels: nothing was left)
    double *xd = reinterpret_cast<double *>(smem_raw);  // n x p design coordinates
    double *kx = xd + (size_t)n * p;                    // np
    __shared__ int s_ok;
    __shared__ double etab[EXP64_TABLE_SIZE];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < EXP64_TABLE_SIZE; i += PREP_THREADS) etab[i] = exp64_table_g[i];
    if (tid == 0) s_ok = 1;
    for (int e = tid; e < n * p; e += PREP_THREADS) xd[e] = load_coord64(X, design[e / p], p, e % p, dt);
    __syncthreads();
    const double ninv_d = -1.0 / d;
    for (int e = tid; e < np * np; e += PREP_THREADS) {
        const int i = e / np, k = e - i * np;
        double v;
        if (i < n && k < n) {
            double s = 0.0;
            for (int t = 0; t < p; t++) {
                const double df = xd[(size_t)i * p + t] - xd[(size_t)k * p + t];
                s = fma(df, df, s);
            }
            v = exp64_tang(s * ninv_d, etab) + (i == k ? g : 0.0);
        } else {
            v = i == k ? 1.0 : 0.0;  // identity padding
        }
        L[(size_t)i * np + k] = v;
    }
    for (int i = tid; i < np; i += PREP_THREADS) {
        double s = 0.0;
        if (i < n)
            for (int t = 0; t < p; t++) {
                const double df = xd[(size_t)i * p + t] - x[t];
                s = fma(df, df, s);
            }
        kx[i] = i < n ? exp64_tang(s * ninv_d, etab) : 0.0;
    }
    __syncthreads();
    // in-place left-looking Cholesky of the lower triangle
    for (int c = 0; c < np; c++) {
        if (warp == 0) {
            double s = 0.0;
            for (int k = lane; k < c; k += 32) s = fma(L[(size_t)c * np + k], L[(size_t)c * np + k], s);
            s = warp_sum(s);
            if (lane == 0) {
                const double piv = L[(size_t)c * np + c] - s;
                if (!(piv > 0.0)) s_ok = 0;
                const double lcc = piv > 0.0 ? sqrt(piv) : 1.0;
                L[(size_t)c * np + c] = lcc;
                rd[c] = 1.0 / lcc;
            }
        }
        __syncthreads();
        const double rcc = rd[c];
        for (int i = c + 1 + tid; i < np; i += PREP_THREADS) {
            double s0 = L[(size_t)i * np + c], s1 = 0.0;
            int k = 0;
            for (; k + 2 <= c; k += 2) {
                s0 = fma(-L[(size_t)i * np + k], L[(size_t)c * np + k], s0);
                s1 = fma(-L[(size_t)i * np + k + 1], L[(size_t)c * np + k + 1], s1);
            }
            if (k < c) s0 = fma(-L[(size_t)i * np + k], L[(size_t)c * np + k], s0);
            L[(size_t)i * np + c] = (s0 + s1) * rcc;
        }
        __syncthreads();
    }
    // z = L^{-1} k_n(x)
    if (warp == 0) {
        for (int i = 0; i < np; i++) {
            double s = 0.0;
            for (int k = lane; k < i; k += 32) s = fma(L[(size_t)i * np + k], z[k], s);
            s = warp_sum(s);
            if (lane == 0) z[i] = (kx[i] - s) * rd[i];
            __syncwarp();
        }
    }
    if (tid == 0) *status = s_ok ? LAGP_OK : LAGP_ENOTPD;
}

__global__ void __launch_bounds__(EV_THREADS)
eval_cands_kernel(const void *X, int p, lagp_dtype dt, const double *x, const int32_t *design, int n,
                  int np, const int32_t *cands, int64_t Nc, double d, double g, const double *L,
                  const double *rd, const double *z, double *W, double *delta, const int32_t *status,
                  const int *redo, const int32_t *left) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *blk = reinterpret_cast<double *>(smem_raw);  // EV_B x EV_B block of L
    double *xd = blk + EV_B * EV_B;                       // n x p design coordinates
    double *xc = xd + (size_t)n * p;                      // EV_THREADS x p candidate coordinates
    __shared__ double etab[EXP64_TABLE_SIZE];
    const int tid = threadIdx.x;
    const int64_t c = (int64_t)blockIdx.x * EV_THREADS + tid;
    if (redo && *redo == 0) return;
    // after the fixed-point kernels: the candidates they left (all when the
    // factorisation itself left the range, and when it fails in FP64)
    const bool failed = *status != LAGP_OK;
    const bool write = c < Nc && (!left || left[c] != 0 || failed);
    if (left && !__syncthreads_or(write)) return;
    const bool live = c < Nc;
    if (failed) {  // the design's K_n was not positive definite
        if (write) delta[c] = CUDART_NAN;
        return;
    }
    for (int i = tid; i < EXP64_TABLE_SIZE; i += EV_THREADS) etab[i] = exp64_table_g[i];
    for (int e = tid; e < n * p; e += EV_THREADS) xd[e] = load_coord64(X, design[e / p], p, e % p, dt);
    const int32_t crow = live ? cands[c] : 0;
    for (int i = 0; i < p; i++) xc[(size_t)tid * p + i] = load_coord64(X, crow, p, i, dt);
    __syncthreads();
    const double ninv_d = -1.0 / d;
    const double *mx = xc + (size_t)tid * p;
    double s = 0.0, q = 0.0;
    const int nb = np / EV_B;
    for (int I = 0; I < nb; I++) {
        double acc[EV_B];
#pragma unroll
        for (int r = 0; r < EV_B; r++) {  // k_n(x_c) for rows of block I
            const int row = I * EV_B + r;
            double sd = 0.0;
            if (row < n)
                for (int t = 0; t < p; t++) {
                    const double df = mx[t] - xd[(size_t)row * p + t];
                    sd = fma(df, df, sd);
                }
            acc[r] = row < n ? exp64_tang(sd * ninv_d, etab) : 0.0;
        }
        for (int J = 0; J < I; J++) {  // acc -= L_IJ w_J
            __syncthreads();
            for (int e = tid; e < EV_B * EV_B; e += EV_THREADS)
                blk[e] = L[(size_t)(I * EV_B + e / EV_B) * np + J * EV_B + (e % EV_B)];
            __syncthreads();
            const double *Wj = W + (size_t)J * EV_B * Nc + c;
#pragma unroll 4
            for (int k = 0; k < EV_B; k++) {
                const double w = live ? Wj[(size_t)k * Nc] : 0.0;
#pragma unroll
                for (int r = 0; r < EV_B; r++) acc[r] = fma(-blk[r * EV_B + k], w, acc[r]);
            }
        }
        __syncthreads();
        for (int e = tid; e < EV_B * EV_B; e += EV_THREADS)
            blk[e] = L[(size_t)(I * EV_B + e / EV_B) * np + I * EV_B + (e % EV_B)];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < EV_B; r++) {  // the diagonal block, in place
            double t = acc[r];
#pragma unroll
            for (int k = 0; k < r; k++) t = fma(-blk[r * EV_B + k], acc[k], t);
            acc[r] = t * rd[I * EV_B + r];
            s = fma(acc[r], acc[r], s);
            q = fma(z[I * EV_B + r], acc[r], q);
        }
        if (live && I + 1 < nb) {
            double *Wi = W + (size_t)I * EV_B * Nc + c;
#pragma unroll
            for (int r = 0; r < EV_B; r++) Wi[(size_t)r * Nc] = acc[r];
        }
    }
    if (write) {
        double sk = 0.0;
        for (int t = 0; t < p; t++) {
            const double df = mx[t] - x[t];
            sk = fma(df, df, sk);
        }
        const double kap = exp64_tang(sk * ninv_d, etab);  // K(x_c, x)
        const double minv = (1.0 + g) - s;                  // m^{-1}(x_c), Eq. (piedef)
        const double r = kap - q;
        delta[c] = minv > 0.0 ? r * r / minv : CUDART_NAN;
    }
}

// ---------------------------------------------------------- fixed point

constexpr int EF_THREADS = 64;   // candidates per CTA
constexpr int EF_B = 16;         // rows per block of the substitution
constexpr int EF_K = 64;         // earlier rows staged at a time
constexpr int EF_HEAD = 3;       // covariances scaled to at most 2^-EF_HEAD: |u| up to 16 of them

// Shared memory of the fixed-point prep: the matrix, then y_at as fx_chol.cuh
// has it, then the design.
__host__ __device__ inline size_t ef_prep_smem(int n, int p) {
    return (size_t)fx_words(n, n + 1) * 16 + ((size_t)3 * n + (size_t)n * p) * 8;
}

// L (limbs, np x np row-major), 1 / diag (ry 2^(rt - 59)) and z = L^{-1} k_n(x)
// 2^-ws (limbs), np = n rounded up to EF_B with identity rows.  One CTA, n <=
// 128.  Out of range: *status = FX_REDO and *redo counts.
__global__ void __launch_bounds__(FXT)
eval_prep_fx_kernel(const void *X, int p, lagp_dtype dt, const double *x, const int32_t *design, int n, int np,
                    double d, double g, int2 *L, long long *ry, int *rt, int2 *z, int *ws, int32_t *status,
                    int *redo) {
    const int words = fx_words(n, n + 1), m = n + 1;
    const FxFactor F{words, n, m, words * 16, n};
    double *kx = fx_y(F), *xd = kx + 3 * n;  // (after the pivots)
    __shared__ int red[FXW];
    const Blk b{(int)threadIdx.x, (int)threadIdx.x & 31, (int)threadIdx.x >> 5};
    for (int e = b.tid; e < n * p; e += FXT) xd[e] = load_coord64(X, design[e / p], p, e % p, dt);
    __syncthreads();
    const double ninv_d = -1.0 / d;
    bool odd = false;  // a distance that is not finite
    for (int e = b.tid; e < n * (n + 1) / 2 + n; e += FXT) {
        int i, k;
        fx_tri(e, i, k);
        const bool cross = i >= n;
        const double D = sqd(cross ? x : xd + (size_t)i * p, xd + (size_t)k * p, p);
        odd |= !(D < CUDART_INF);
        const double E = exp64_tang(D * ninv_d, exp64_table_g);
        if (cross) kx[k] = E;
        else *fx_raw(F, 0, fx_slot(i, k, m)) = fx_from(i == k ? E + g : E);
    }
    const int ex = fx_exponent(kx, n, red, b);
    bool ok = !(__syncthreads_or(odd) || ex == INT32_MAX);
    if (ok) {
        for (int k = b.tid; k < n; k += FXT) *fx_raw(F, 0, fx_slot(n, k, m)) = fx_from(fx_shift(kx[k], -(ex + 2)));
        ok = !fx_factorise<1>(F, b);
    }
    if (ok) {
        bool big = false;  // |z|^2 >= 63 (entries are below 1: only beyond 64 rows)
        if (n >= 64 && b.tid < 32) {
            float s = 0.f;
            for (int i = b.tid; i < n; i += 32) {
                const float v = (float)fx_split(fx_load(F, 0, fx_slot(n, i, m))).h * 0x1p-29f;
                s = fmaf(v, v, s);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(LAGP_FULL_MASK, s, o);
            big = s >= 63.f;
        }
        ok = !__syncthreads_or(big);
    }
    if (!ok) {
        if (b.tid == 0) {
            *status = FX_REDO;
            *redo = 1;
        }
        return;
    }
    for (int e = b.tid; e < np * np; e += FXT) {
        const int i = e / np, k = e - i * np;
        Fx f{i == k ? 1 << 29 : 0, 0};
        if (i < n && k < n) f = k <= i ? fx_split(fx_load(F, 0, fx_slot(i, k, m))) : Fx{0, 0};
        L[e] = make_int2(f.h, f.l);
    }
    for (int i = b.tid; i < np; i += FXT) {
        ry[i] = i < n ? fx_ry(F)[i] : FX_ONE;
        rt[i] = i < n ? fx_rt(F)[i] : 0;
        const Fx f = i < n ? fx_split(fx_load(F, 0, fx_slot(n, i, m))) : Fx{0, 0};
        z[i] = make_int2(f.h, f.l);
    }
    if (b.tid == 0) {
        *ws = ex + 2;
        *status = LAGP_OK;
    }
}

// The same from the FP64 factor (n > 128): the limbs of its entries.  z is
// scaled by the power of two that brings its largest entry below 1/4 (every
// block finds it; |z^T u| then stays below 16): a location far from the design
// has a z as small as its covariances, and the same relative precision.
__global__ void eval_limbs_kernel(const double *L64, const double *rd, const double *z64, int np64, int n, int np,
                                  int2 *L, long long *ry, int *rt, int2 *z, int *ws, const int32_t *status,
                                  int *redo) {
    if (*status != LAGP_OK) return;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    __shared__ int s_top;
    if (threadIdx.x == 0) s_top = 0;
    __syncthreads();
    int top = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) top = max(top, (__double2hiint(z64[i]) >> 20) & 0x7ff);
    atomicMax(&s_top, top);
    __syncthreads();
    top = s_top;
    const int zs = top == 0 ? 0 : top - 1022 + 2;
    for (int e = tid; e < np * np; e += gridDim.x * blockDim.x) {
        const int i = e / np, k = e - i * np;
        const double v = i < n && k <= i ? L64[(size_t)i * np64 + k] : (i == k ? 1.0 : 0.0);
        const Fx f = fx_split(fx_from(v));
        L[e] = make_int2(f.h, f.l);
    }
    for (int i = tid; i < np; i += gridDim.x * blockDim.x) {
        // rd = y 2^t with y in [0.5, 1)
        const double r = i < n ? rd[i] : 1.0;
        const int ex = ((__double2hiint(r) >> 20) & 0x7ff) - 1022;
        if (ex < 0 || ex > 24) redo[0] = redo[1] = 1;  // (as fx_rsqrt's range)
        rt[i] = ex;
        ry[i] = fx_from(fx_shift(r, -ex));
        const Fx f = fx_split(fx_from(i < n && top < 0x7ff ? fx_shift(z64[i], -zs) : 0.0));
        z[i] = make_int2(f.h, f.l);
    }
    if (tid == 0) {
        *ws = zs;
        if (top == 0x7ff) redo[0] = redo[1] = 1;  // not finite
    }
}

__global__ void __launch_bounds__(EF_THREADS, 8)
eval_cands_fx_kernel(const void *X, int p, lagp_dtype dt, const double *x, const int32_t *design, int n, int np,
                     const int32_t *cands, int64_t Nc, double d, double g, const int2 *__restrict__ L,
                     const long long *__restrict__ ry, const int *__restrict__ rt, const int2 *__restrict__ z,
                     const int *__restrict__ wsp, int2 *W, double *delta, const int32_t *status, int *redo,
                     int32_t *left) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int4 *blk = reinterpret_cast<int4 *>(smem_raw);           // EF_K columns of EF_B rows (two rows a word)
    double *xd = reinterpret_cast<double *>(blk + EF_K * EF_B / 2);  // n x p design coordinates
    double *xc = xd + (size_t)n * p;                          // EF_THREADS x p candidate coordinates
    float *xf = reinterpret_cast<float *>(xc + (size_t)EF_THREADS * p);  // both in FP32, relative to x
    float *cf = xf + (size_t)n * p + (size_t)threadIdx.x * p;
    __shared__ int2 s_y[EF_B], s_z[EF_B];
    __shared__ int s_t[EF_B];
    const int tid = threadIdx.x;
    const int64_t c = (int64_t)blockIdx.x * EF_THREADS + tid;
    const bool live = c < Nc;
    const int32_t st = *status;
    if (st != LAGP_OK || redo[1] != 0) {  // (redo[1]: limbs out of range)
        if (live) {
            left[c] = st == LAGP_ENOTPD ? 0 : 1;
            if (st == LAGP_ENOTPD) delta[c] = CUDART_NAN;
        }
        return;
    }
    for (int e = tid; e < n * p; e += EF_THREADS) {
        xd[e] = load_coord64(X, design[e / p], p, e % p, dt);
        xf[e] = (float)(xd[e] - x[e % p]);
    }
    const int32_t crow = live ? cands[c] : cands[0];
    double *mx = xc + (size_t)tid * p;
    for (int i = 0; i < p; i++) {
        mx[i] = load_coord64(X, crow, p, i, dt);
        cf[i] = (float)(mx[i] - x[i]);
    }
    __syncthreads();
    const double ninv_d = -1.0 / d;
    // the scale: 2^e with max_i k_i 2^e near 2^-EF_HEAD, from the nearest design row in FP32
    float near = CUDART_INF_F;
    for (int r = 0; r < n; r++) {
        float s = 0.f;
        for (int t = 0; t < p; t++) {
            const float df = cf[t] - xf[r * p + t];
            s = fmaf(df, df, s);
        }
        near = fminf(near, s);
    }
    const int e2 = (int)fminf(near / (float)d * 1.4426950f, 900.f) - EF_HEAD;
    unsigned bad = !(near < CUDART_INF_F);
    long long sh = 0, sm = FX_HALF, qh = 0, qm = FX_HALF;  // |u|^2 and z^T u
    float norm2 = 0.f;                                     // |u|^2 in FP32: whether they hold
    const int nb = np / EF_B;
    for (int I = 0; I < nb; I++) {
        long long hi[EF_B], mid[EF_B];
#pragma unroll
        for (int r = 0; r < EF_B; r++) hi[r] = 0, mid[r] = FX_HALF;
        for (int k0 = 0; k0 < I * EF_B; k0 += EF_K) {
            const int kk = min(EF_K, I * EF_B - k0);
            __syncthreads();
            for (int e = tid; e < EF_B * kk; e += EF_THREADS) {
                const int r = e / kk, k = e - r * kk;
                reinterpret_cast<int2 *>(blk)[k * EF_B + r] = L[(size_t)(I * EF_B + r) * np + k0 + k];
            }
            __syncthreads();
            const int2 *Wk = W + (size_t)k0 * Nc + (live ? c : 0);
#pragma unroll 2
            for (int k = 0; k < kk; k++) {
                const int2 u = Wk[(size_t)k * Nc];
                const int4 *row = blk + k * (EF_B / 2);
#pragma unroll
                for (int r = 0; r < EF_B; r += 2) {
                    const int4 l = row[r / 2];
                    hi[r] = fx_mad(u.x, l.x, hi[r]);
                    mid[r] = fx_mad(u.y, l.x, fx_mad(u.x, l.y, mid[r]));
                    hi[r + 1] = fx_mad(u.x, l.z, hi[r + 1]);
                    mid[r + 1] = fx_mad(u.y, l.z, fx_mad(u.x, l.w, mid[r + 1]));
                }
            }
        }
        __syncthreads();
        for (int e = tid; e < EF_B * EF_B; e += EF_THREADS) {
            const int r = e / EF_B, k = e - r * EF_B;
            reinterpret_cast<int2 *>(blk)[k * EF_B + r] = L[(size_t)(I * EF_B + r) * np + I * EF_B + k];
        }
        if (tid < EF_B) {
            const Fx y = fx_split(ry[I * EF_B + tid]);
            s_y[tid] = make_int2(y.h, y.l);
            s_t[tid] = rt[I * EF_B + tid];
            s_z[tid] = z[I * EF_B + tid];
        }
        __syncthreads();
        int2 *Wi = W + (size_t)I * EF_B * Nc + c;
#pragma unroll
        for (int r = 0; r < EF_B; r++) {  // the diagonal block, in place
            const int row = I * EF_B + r;
            double kv = 0.0;
            if (row < n) {
                double sd = 0.0;
                for (int t = 0; t < p; t++) {
                    const double df = mx[t] - xd[(size_t)row * p + t];
                    sd = fma(df, df, sd);
                }
                kv = fx_shift(exp64_tang(sd * ninv_d, exp64_table_g), e2);
            }
            const int2 y2 = s_y[r], z2 = s_z[r];
            bad |= kv >= 1.0;
            const long long S = fx_from(kv >= 1.0 ? 0.0 : kv) - (hi[r] << 1) - (mid[r] >> 29);
            const Fx u = fx_split(fx_scaled(S, s_t[r], Fx{y2.x, y2.y}, bad));
            bad |= fx_beyond_h(u);
            const float uf = (float)u.h * 0x1p-29f;
            norm2 = fmaf(uf, uf, norm2);
            sh = fx_mad(u.h, 2 * u.h, sh);
            sm = fx_mid(sm, u, u);
            qh = fx_mad(u.h, 2 * z2.x, qh);
            qm = fx_mid(qm, u, Fx{z2.x, z2.y});
#pragma unroll
            for (int r2 = r + 1; r2 < EF_B; r2++) {
                const int2 l = reinterpret_cast<const int2 *>(blk)[r * EF_B + r2];
                hi[r2] = fx_mad(u.h, l.x, hi[r2]);
                mid[r2] = fx_mad(u.l, l.x, fx_mad(u.h, l.y, mid[r2]));
            }
            if (live && I + 1 < nb) Wi[(size_t)r * Nc] = make_int2(u.h, u.l);
        }
    }
    if (live) {
        double sk = 0.0;
        for (int t = 0; t < p; t++) {
            const double df = mx[t] - x[t];
            sk = fma(df, df, sk);
        }
        const double kap = exp64_tang(sk * ninv_d, exp64_table_g);  // K(x_c, x)
        // |u|^2 < 3.9 in its scale, so that neither sum has wrapped (they hold 16,
        // and |z| is at most 8).  The sum itself could not tell: 34 looks like 2.
        const long long sv = fx_sum(sh, sm), qv = fx_sum(qh, qm);
        bad |= !(norm2 < 3.9f);
        const double s = scalbn(fx_double(sv), -2 * e2), q = scalbn(fx_double(qv), *wsp - e2);
        const double minv = (1.0 + g) - s;  // m^{-1}(x_c), Eq. (piedef)
        const double r = kap - q;
        delta[c] = minv > 0.0 ? r * r / minv : CUDART_NAN;
        bad |= !(minv > 0.0);  // (for FP64 to decide)
        left[c] = bad ? 1 : 0;
        if (bad) atomicExch(redo, 1);
    }
}

}  // namespace

extern "C" lagp_status lagp_alc_eval(lagp_ctx *ctx, const void *X, int64_t N, int32_t p,
                                     lagp_dtype dtype, const double *x, const int32_t *design,
                                     int32_t n, const int32_t *cands, int64_t Nc, double d, double g,
                                     double *delta, int32_t *status) {
    if (!ctx) return LAGP_EINVAL;
    ctx->err.clear();
    if (!X || !x || !design || !status || (Nc > 0 && (!cands || !delta)))
        return lagp_fail(ctx, LAGP_EINVAL, "lagp_alc_eval: NULL required array");
    if (N < 1 || N >= (int64_t)INT32_MAX || p < 1 || p > 64 || (dtype != LAGP_F64 && dtype != LAGP_F32))
        return lagp_fail(ctx, LAGP_EINVAL, "lagp_alc_eval: need 1 <= N < 2^31, 1 <= p <= 64, dtype F64/F32");
    if (n < 1 || n > 1024 || Nc < 0 || !(d > 0.0) || !(g >= 0.0))
        return lagp_fail(ctx, LAGP_EINVAL, "lagp_alc_eval: need 1 <= n <= 1024, Nc >= 0, d > 0, g >= 0");
    LAGP_CUDA(ctx, cudaSetDevice(ctx->device));
    const int np = (n + EV_B - 1) / EV_B * EV_B;
    const int64_t nw = Nc > 0 ? Nc : 1;
    // FP64: L, 1 / diag, z, the panel of solved rows; fixed point: the same in
    // limbs (its panel in the same place), the exponents, the flags
    const size_t wbytes = (size_t)np * np * 8 + 2 * (size_t)np * 8 + (size_t)np * nw * 8;
    const size_t fbytes = (size_t)np * np * 8 + (size_t)np * 24 + (size_t)nw * 4 + 64;
    const bool fixed = g < 1.0;
    char *base = static_cast<char *>(lagp_ws(ctx, WS_ALC_STATE, wbytes + (fixed ? fbytes : 0) + 256));
    if (!base) return LAGP_ENOMEM;
    double *Lm = reinterpret_cast<double *>(base);
    double *rd = Lm + (size_t)np * np, *z = rd + np, *W = z + np;
    int2 *fL = reinterpret_cast<int2 *>(base + wbytes);
    long long *fry = reinterpret_cast<long long *>(fL + (size_t)np * np);
    int2 *fz = reinterpret_cast<int2 *>(fry + np);
    int *frt = reinterpret_cast<int *>(fz + np);
    int *words = frt + np;  // [0] the scale of z, [1] work is left to FP64, [2] all of it
    int32_t *left = words + 3;
    const size_t smem_prep = ((size_t)n * p + np) * 8;
    const size_t smem = ((size_t)EV_B * EV_B + (size_t)n * p + (size_t)EV_THREADS * p) * 8;
    if (smem_prep > ctx->smem_optin || (Nc > 0 && smem > ctx->smem_optin))
        return lagp_fail(ctx, LAGP_EINVAL, "lagp_alc_eval: n x p too large");
    cudaStream_t st = ctx->stream;
    const int nf = (n + EF_B - 1) / EF_B * EF_B;
    const size_t smem_fx = (size_t)EF_K * EF_B * 8 + ((size_t)n * p + (size_t)EF_THREADS * p) * 8 +
                           ((size_t)n + EF_THREADS) * p * 4;
    const bool fx = fixed && smem_fx <= lagp_smem_room(ctx, eval_cands_fx_kernel);
    const bool fx_prep = fx && n <= FX_NMAX && ef_prep_smem(n, p) <= lagp_smem_room(ctx, eval_prep_fx_kernel);
    auto prep64 = [&](const int *redo) {
        cudaFuncSetAttribute(eval_prep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_prep);
        eval_prep_kernel<<<1, PREP_THREADS, smem_prep, st>>>(X, p, dtype, x, design, n, np, d, g, Lm, rd, z, status,
                                                             redo);
        ctx->launches++;
    };
    if (fx) LAGP_CUDA(ctx, cudaMemsetAsync(words, 0, 12, st));
    if (fx_prep) {
        cudaFuncSetAttribute(eval_prep_fx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ef_prep_smem(n, p));
        eval_prep_fx_kernel<<<1, FXT, ef_prep_smem(n, p), st>>>(X, p, dtype, x, design, n, nf, d, g, fL, fry, frt, fz,
                                                                words, status, words + 1);
        ctx->launches++;
    } else {
        prep64(nullptr);
        if (fx && Nc > 0) {
            eval_limbs_kernel<<<ctx->num_sms, 256, 0, st>>>(Lm, rd, z, np, n, nf, fL, fry, frt, fz, words, status,
                                                            words + 1);
            ctx->launches++;
        }
    }
    LAGP_CUDA(ctx, cudaGetLastError());
    if (fx && Nc > 0) {
        cudaFuncSetAttribute(eval_cands_fx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_fx);
        eval_cands_fx_kernel<<<(unsigned)((Nc + EF_THREADS - 1) / EF_THREADS), EF_THREADS, smem_fx, st>>>(
            X, p, dtype, x, design, n, nf, cands, Nc, d, g, fL, fry, frt, fz, words, reinterpret_cast<int2 *>(W), delta,
            status, words + 1, left);
        ctx->launches++;
        LAGP_CUDA(ctx, cudaGetLastError());
    }
    // in FP64: everything, or what the fixed-point kernels left
    if (fx_prep) prep64(words + 1);
    if (Nc > 0) {
        cudaFuncSetAttribute(eval_cands_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        const int64_t grid = (Nc + EV_THREADS - 1) / EV_THREADS;
        eval_cands_kernel<<<(unsigned)grid, EV_THREADS, smem, st>>>(X, p, dtype, x, design, n, np, cands, Nc, d, g, Lm,
                                                                    rd, z, W, delta, status, fx ? words + 1 : nullptr,
                                                                    fx ? left : nullptr);
        ctx->launches++;
    }
    LAGP_CUDA(ctx, cudaGetLastError());
    return LAGP_OK;
}
