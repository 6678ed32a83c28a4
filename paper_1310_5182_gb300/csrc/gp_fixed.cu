// a7 (local prediction) and a8 (local Newton MLE of d) in 59-bit fixed point
// (fx59.cuh), for designs of up to 128 rows and nuggets below 1.
//
// One CTA of 128 threads per location (persistent, atomic work counter), all
// of its matrices in shared memory.
//   K_n is factorised as L L^T with the responses (and, for the prediction,
//   k_n(x)) as further rows: the rows below K_n's become z^T = (L^{-1} Y)^T
//   and w^T = (L^{-1} k)^T.  For the MLE the factorisation carries its first
//   and second derivatives in log d along (forward mode): with
//     M0 = K,  M1 = d K' = t e^-t,  M2 = d^2 K'' = (t^2 - 2t) e^-t,  t = D/d,
//   column c of L, L1 = d L', L2 = d^2 L'' comes from
//     S0 = M0 - sum L L^T,  S1 = M1 - sum (L1 L^T + L L1^T),
//     S2 = M2 - sum (L2 L^T + 2 L1 L1^T + L L2^T)            (sums over k < c)
//     l = sqrt(S0),  l1 = S1 / (2l),  l2 = (S2/2 - l1^2) / l   on the diagonal,
//     L = S0 / l,  L1 = (S1 - L l1) / l,  L2 = (S2 - 2 L1 l1 - L l2) / l  below,
//   and then log|K|, psi = |z|^2 and their derivatives are sums over the
//   diagonal and over the z row: six products a (row, column, k) triple, n^3
//   in all, with no inverse, no traces and no second pass.  All entries are
//   of order one (t e^-t <= 1/e, |t^2 - 2t| e^-t <= 0.47, |L| < sqrt(2)), which
//   is what fixed point asks for; z is scaled by a power of two.
//
// Bound: latency and instruction fetch between short barriers (MLE, n = 60, four
// CTAs an SM: issue 37%, barrier stalls 3.0 and no instruction 1.8 per issued
// instruction, ALU 34%, FP64 20%); the prediction's n^2/2 exponentials on the
// FP64 unit (62% busy at n = 60).
// Two columns a step: the sums run with a 2 x 2 tile of (rows, columns) a
// thread, so that a 16-byte shared-memory load (two k) feeds four products,
// and 4 to 16 lanes share a row's sum, so that the threads stay busy as the
// rows left shrink; meanwhile one warp makes the 2 x 2 diagonal block, and
// then one thread a row finishes the two columns.
//
// Measured against the FP64 kernels (gp_local.cu), whole calls: the MLE of
// 20,000 slab locations, n = 60, 4.1 evaluations each, 79.9 -> 29.7 ms; the
// prediction at 100 locations, n = 50, 112 -> 66 us.  Errors against 80-bit
// references over lengthscales from nearly diagonal to ill-conditioned K, n = 8
// and 60: medians as from the FP64 kernels (l'' up to five times smaller where
// K is ill-conditioned).  The line: above 128 rows the three matrices no longer fit in
// shared memory; from g = 1 on the factor's entries leave the range.
//
// A location whose values leave the fixed-point range (|x| < 2; 1 in the
// further rows) first widens the scale of z (K's own rounding times its
// condition number is then what counts, not that of the responses), then goes
// to the FP64 kernels of gp_local.cu: its status is FX_REDO or below when this
// kernel ends, and a second launch redoes it (returning at once when there is
// none).  So do locations with non-finite inputs or without a nonzero response,
// means of small responses beside large ones, and estimates at nearly diagonal K.
//
// Range of the sums: |S| holds 16 and wraps round at 32.  Rows of L have norms
// below sqrt(2) whatever the data, and z rows, with entries below 1, at most
// 11.4; the derivative rows' norms came to 1.7 and 5.1 (L1, L2) over kernels,
// dimensions, lengthscales and nuggets down to 1e-8 with every entry in range,
// so that S2 stays below 22, and 2^63 lies 17 standard deviations from the
// middle sums of a share (a quarter of the columns).
#include <cuda_runtime.h>

#include <algorithm>

#include "device_util.cuh"
#include "exp64.cuh"
#include "fx_chol.cuh"
#include "gp_common.cuh"
#include "lagp_internal.h"

namespace {

// z is scaled by 2^-FX_Z0 / max |y| (|z| up to 64 max |y| then fits), else by 2^-FX_Z1
constexpr int FX_Z0 = 6, FX_Z1 = 14;

struct FxLaunch {
    int cls_lo, cls_hi;   // this launch takes the locations with cls_lo < n <= cls_hi
    bool stray;           // and those whose n is out of range
    int words;            // matrix words for n = cls_hi
    int *counter, *redo;  // work counter; number of locations left to the FP64 kernels
    double *dist;         // per CTA: squared distances of the design (MLE)
};

__device__ __forceinline__ bool fx_mine(const FxLaunch &f, int nm, int nmax) {
    if (nm < 1 || nm > nmax) return f.stray;
    return nm > f.cls_lo && nm <= f.cls_hi;
}

// ------------------------------------------------------------------ predict

// Eight CTAs an SM (64 registers): a location's chain of diagonal blocks is
// latency, which the other CTAs fill.  10,000 locations, n = 14 / 50: 0.46 /
// 1.52 ms at 124 registers, 0.28 / 0.98 here (FP64 kernel: 0.43 / 2.44).
__global__ void __launch_bounds__(FXT, 8)
predict_fx_kernel(GpArgs a, FxLaunch f, const double *__restrict__ dv, double *mean, double *s2, double *df,
                  int32_t *status) {
    const int nmax = f.cls_hi, p = a.p;
    double *y = reinterpret_cast<double *>(fx_smem + f.words * 16);
    double *xd = y + 3 * nmax, *xq = xd + nmax * p, *kx = xq + p;  // (after y: the pivots)
    __shared__ int s_loc, s_flag, red[FXW];
    __shared__ float s_part[FXW];
    const Blk b{(int)threadIdx.x, (int)threadIdx.x & 31, (int)threadIdx.x >> 5};
    for (;;) {
        if (b.tid == 0) s_loc = atomicAdd(f.counter, 1);
        __syncthreads();
        const int64_t loc = s_loc;
        __syncthreads();
        if (loc >= a.M) break;
        const int nm = a.n ? a.n[loc] : a.nmax;
        if (!fx_mine(f, nm, a.nmax)) continue;
        int st = load_design(a, loc, nm, dv, xd, y, &s_flag, b);
        double mu = CUDART_NAN, sv = CUDART_NAN, dfv = CUDART_NAN;
        if (st == LAGP_OK) {
            const double d = dv[loc], g = a.g, ninv_d = -1.0 / d;
            for (int i = b.tid; i < p; i += FXT) xq[i] = load_coord64(a.Xref, loc, p, i, a.dtype);
            __syncthreads();
            const int m = nm + 2;
            const FxFactor F{f.words, nm, m, f.words * 16, nmax};
            st = FX_REDO;
            int zs = 0, ws = 0;
            // (responses that are all zero, or not finite, go to FP64 at once)
            const int ey = fx_exponent(y, nm, red, b);
            for (int wide = 0; wide < 2 && st != LAGP_OK && ey != INT32_MAX; wide++) {
                bool odd = false;  // a distance that is not finite
                for (int e = b.tid; e < nm * (nm + 1) / 2 + nm; e += FXT) {
                    int i, k;
                    fx_tri(e, i, k);
                    const bool cross = i >= nm;
                    const double D = sqd(cross ? xq : xd + (size_t)i * p, xd + (size_t)k * p, p);
                    odd |= !(D < CUDART_INF);
                    const double E = exp64_tang(D * ninv_d, exp64_table_g);
                    if (cross) kx[k] = E;
                    else *fx_raw(F, 0, fx_slot(i, k, m)) = fx_from(i == k ? E + g : E);
                }
                const int ex = fx_exponent(kx, nm, red, b);
                if (__syncthreads_or(odd) || ex == INT32_MAX) break;
                zs = ey + (wide ? FX_Z1 : FX_Z0);
                ws = ex + 2;
                for (int k = b.tid; k < nm; k += FXT) {
                    *fx_raw(F, 0, fx_slot(nm, k, m)) = fx_from(fx_shift(y[k], -zs));
                    *fx_raw(F, 0, fx_slot(nm + 1, k, m)) = fx_from(fx_shift(kx[k], -ws));
                }
                if (!fx_factorise<1>(F, b)) st = LAGP_OK;
            }
            if (st == LAGP_OK) {
                double v[3] = {0.0, 0.0, 0.0};
                float part = 0.f;  // |w|_1 + |z|_1 - 2^11 |w|^T |z| (from the high limbs)
                for (int i = b.tid; i < nm; i += FXT) {
                    const long long zf = fx_load(F, 0, fx_slot(nm, i, m)), wf = fx_load(F, 0, fx_slot(nm + 1, i, m));
                    const double z = fx_double(zf), w = fx_double(wf);
                    v[0] = fma(w, z, v[0]);
                    v[1] = fma(z, z, v[1]);
                    v[2] = fma(w, w, v[2]);
                    const float zh = fabsf((float)(int)(zf >> 30)) * 0x1p-29f, wh = fabsf((float)(int)(wf >> 30)) * 0x1p-29f;
                    part += zh + wh - 0x1p11f * (zh * wh);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(LAGP_FULL_MASK, part, o);
                if (b.lane == 0) s_part[b.warp] = part;
                block_sums<3>(v, b);  // (its barriers order s_part)
                part = 0.f;
                for (int q = 0; q < FXW; q++) part += s_part[q];
                // w and z are absolute (2^-59): a mean made of a few small responses
                // beside far larger ones has fewer bits than in FP64 (responses
                // over twelve decades, K nearly diagonal: relative 3e-9 against
                // 1e-14).  It goes there when 2^-58 (|w|_1 + |z|_1) exceeds both
                // 2^-47 of its terms' magnitudes and 2^-44 of itself and K is within
                // e^{-n/8} of its diagonal's determinant; with rows that are
                // coupled FP64's z carries the rounding of the largest entries too.
                bool few = 0x1p-14 * part > fabs(v[0]);
                if (few) {  // (block-uniform)
                    float ld = 0.f;  // log2 of det(K)^(-1/2)
                    for (int i = b.tid; i < nm; i += FXT)
                        ld += __log2f((float)(int)(fx_ry(F)[i] >> 30) * 0x1p-29f) + (float)fx_rt(F)[i];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) ld += __shfl_xor_sync(LAGP_FULL_MASK, ld, o);
                    __syncthreads();  // s_part was read
                    if (b.lane == 0) s_part[b.warp] = ld;
                    __syncthreads();
                    ld = 0.f;
                    for (int q = 0; q < FXW; q++) ld += s_part[q];
                    few = ld < nm * (0.09f - 0.5f * __log2f(1.f + (float)g));
                }
                if (few) {
                    st = FX_REDO;
                } else {
                    mu = scalbn(v[0], zs + ws);
                    const double psi = scalbn(v[1], 2 * zs), kk = scalbn(v[2], 2 * ws);
                    sv = psi * ((1.0 + g) - kk) / nm;
                    dfv = nm;
                }
            }
        }
        if (b.tid == 0) {
            if (st == FX_REDO) atomicAdd(f.redo, 1);
            mean[loc] = mu;
            s2[loc] = sv;
            df[loc] = dfv;
            status[loc] = st;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------- MLE

struct FxEval {
    double l, dl, d2l;
    int flag;  // fx_factorise's; 2: derivatives too small for a fixed point
};

// l, and with NM = 3 l' and l'', of Eq. (gpk) at d from the packed squared distances; zs: the
// power of two that z is scaled by; lgam: log Gamma(n/2) - (n/2) log 2 pi.
template <int NM, int T>
__device__ __noinline__ FxEval fx_llik(const FxFactor F, const double *dist, double d, double g, int zs,
                          double lgam, const Blk &b) {
    const int n = F.n, m = F.m;
    const double ninv_d = -1.0 / d;
    for (int e = b.tid; e < n * (n + 1) / 2; e += T) {
        int i, k;
        fx_tri(e, i, k);
        const double t = -(dist[e] * ninv_d);
        const double E = exp64_tang(-t, exp64_table_g);
        const double K1 = E > 0.0 ? t * E : 0.0, K2 = E > 0.0 ? K1 * (t - 2.0) : 0.0;
        const int s = fx_slot(i, k, m);
        *fx_raw(F, 0, s) = fx_from(i == k ? E + g : E);
        if constexpr (NM == 3) {
            *fx_raw(F, 1, s) = fx_from(K1);
            *fx_raw(F, 2, s) = fx_from(K2);
        }
    }
    for (int k = b.tid; k < n; k += T) {
        const int s = fx_slot(n, k, m);
        *fx_raw(F, 0, s) = fx_from(fx_shift(fx_y(F)[k], -zs));
        if constexpr (NM == 3) *fx_raw(F, 1, s) = *fx_raw(F, 2, s) = 0;
    }
    FxEval r;
    r.flag = fx_factorise<NM, T>(F, b);
    r.l = r.dl = r.d2l = CUDART_NAN;
    if (r.flag) return r;
    // log|K| = -2 log prod r, r = 1 / l = y 2^t with y in (0.7, 1.42]: the
    // product of a warp's y stays in range, one logarithm for all
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    double prod = 1.0;
    for (int i = b.tid; i < n; i += T) {
        const double yr = fx_double(fx_ry(F)[i]), ri = fx_shift(yr, fx_rt(F)[i]);
        prod *= yr;
        v[0] += fx_rt(F)[i];
        const int s = fx_slot(i, i, m), z = fx_slot(n, i, m);
        const double z0 = fx_double(fx_load(F, 0, z));
        v[3] = fma(z0, z0, v[3]);             // psi and its derivatives (scaled)
        if constexpr (NM == 3) {
            const double p1 = fx_double(fx_load(F, 1, s)) * ri, p2 = fx_double(fx_load(F, 2, s)) * ri;
            const double z1 = fx_double(fx_load(F, 1, z)), z2 = fx_double(fx_load(F, 2, z));
            v[1] += p1;                       // (d/dlog d) sum log l
            v[2] += fma(-p1, p1, p2);
            v[4] = fma(2.0 * z0, z1, v[4]);
            v[5] = fma(2.0 * z1, z1, fma(2.0 * z0, z2, v[5]));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) prod *= __shfl_xor_sync(LAGP_FULL_MASK, prod, o);
    __shared__ double s_prod[T / 32];
    if (b.lane == 0) s_prod[b.warp] = prod;
    block_sums<6, T>(v, b);  // (its barriers order s_prod)
    __shared__ FxEval s_r;
    if (b.warp == 0) {
        // the logarithms side by side, the other scalars on every lane
        double all = 1.0;
        for (int w = 0; w < T / 32; w += 2) all *= s_prod[w] * s_prod[w + 1];
        const double arg = b.lane == 0 ? all : (b.lane == 1 ? scalbn(v[3], 2 * zs) / 2.0 : 1.0 + g);
        const double lg = log(arg);
        const double half_logdet = -(__shfl_sync(LAGP_FULL_MASK, lg, 0) + v[0] * CUDART_LN2);
        const double logpsi = __shfl_sync(LAGP_FULL_MASK, lg, 1);
        const double logdiag = __shfl_sync(LAGP_FULL_MASK, lg, 2);
        const double hn = 0.5 * n, ipsi = 1.0 / v[3], id = -ninv_d, q1 = v[4] * ipsi;
        if (b.lane == 0) {
            s_r.l = lgam - half_logdet - hn * logpsi;
            s_r.dl = (-v[1] - hn * q1) * id;
            s_r.d2l = (-v[2] - hn * fma(-q1, q1, v[5] * ipsi)) * id * id;
            // K next to diagonal (|K| within e^{-n/8} of the diagonal's product):
            // the terms of d l' are small, and their errors absolute, about 2^-52
            // n: below n / 16 they would exceed FP64's.  (8-d, n = 60, d = 0.004:
            // l' off by a relative 1e-9.)  With terms below 2^-16 rounding would
            // decide the sign, and so the step, whatever K is.
            const double terms = fabs(v[1]) + hn * fabs(q1);
            const bool diagonal = half_logdet > hn * (logdiag - 0.125);
            s_r.flag = NM == 3 && n > 1 && !(terms >= 0x1p-16 && (!diagonal || terms >= 0.125 * hn)) ? 2 : 0;
        }
    }
    __syncthreads();
    return s_r;
}

// NM = 1: the likelihood at d alone (max_iter = 0, no derivative wanted), a
// sixth of the arithmetic, a third of the shared memory: 5,000 locations, n =
// 50, 1.3 -> 0.55 ms.
template <int NM, int T>
__global__ void __launch_bounds__(T, (NM == 3 ? 512 : 1024) / T)
mle_fx_kernel(GpArgs a, FxLaunch f, double *dv, double dmin, double dmax, int max_iter, MleOut o,
              unsigned long long *work) {
    const int nmax = f.cls_hi, p = a.p;
    double *xd = reinterpret_cast<double *>(fx_smem);  // before the matrices are filled
    const int y_at = (int)max(NM * f.words * 16, (nmax * p * 8 + 15) & ~15);
    double *y = reinterpret_cast<double *>(fx_smem + y_at);
    double *dist = f.dist + (size_t)blockIdx.x * (nmax * (nmax + 1) / 2);
    __shared__ int s_loc, s_flag, red[T / 32];
    __shared__ double s_lgam;
    const Blk b{(int)threadIdx.x, (int)threadIdx.x & 31, (int)threadIdx.x >> 5};
    unsigned long long n_llik = 0, n_derivs = 0;  // evaluations x n^3 (thread 0's count)
    for (;;) {
        if (b.tid == 0) s_loc = atomicAdd(f.counter, 1);
        __syncthreads();
        const int64_t loc = s_loc;
        __syncthreads();
        if (loc >= a.M) break;
        const int nm = a.n ? a.n[loc] : a.nmax;
        if (!fx_mine(f, nm, a.nmax)) continue;
        int st = load_design<T>(a, loc, nm, dv, xd, y, &s_flag, b);
        const unsigned long long n3 = (unsigned long long)nm * nm * nm;
        FxEval r{CUDART_NAN, CUDART_NAN, CUDART_NAN, 0};
        int it = 0, kept = 0;  // iterations; those that FP64 takes over
        double d = dv[loc];
        if (st == LAGP_OK) {
            const double g = a.g;
            d = fmin(fmax(d, dmin), dmax);
            const int ey = fx_exponent<T>(y, nm, red, b);
            bool odd = ey == INT32_MAX;
            for (int e = b.tid; e < nm * (nm + 1) / 2 && !odd; e += T) {
                int i, k;
                fx_tri(e, i, k);
                const double D = sqd(xd + (size_t)i * p, xd + (size_t)k * p, p);
                odd |= !(D < CUDART_INF);
                dist[e] = D;  // read back by this thread only
            }
            if (b.tid == 0) {
                const double hn = 0.5 * nm;
                s_lgam = lgamma(hn) - hn * log(2.0 * CUDART_PI);
            }
            odd = __syncthreads_or(odd);
            const double lgam = s_lgam;
            const FxFactor F{f.words, nm, nm + 1, y_at, nmax};
            int zs = ey + FX_Z0;
            // one evaluation; out of range: once more with a wider z
            auto eval = [&](double at) {
                FxEval q = fx_llik<NM, T>(F, dist, at, g, zs, lgam, b);
                if (q.flag == 1 && zs < ey + FX_Z1) {
                    zs = ey + FX_Z1;
                    q = fx_llik<NM, T>(F, dist, at, g, zs, lgam, b);
                }
                return q;
            };
            unsigned long long ll = 0, de = 0;
            if (odd) {
                st = FX_REDO;
            } else {
                r = eval(d);
                ll += n3;
                if (r.flag) {
                    st = FX_REDO;
                } else {
                    if (NM == 3) de += n3;
                    while (NM == 3 && it < max_iter) {
                        it++;
                        double delta;
                        if (r.d2l < 0.0) delta = -r.dl / r.d2l;
                        else delta = (r.dl > 0.0) ? d : -0.5 * d;
                        bool accepted = false;
                        double dn = d;
                        FxEval t = r;
                        // a short Newton step near the maximiser raises l below the
                        // FP64 resolution of l: taken without comparing l values
                        const bool short_newton = r.d2l < 0.0 && fabs(delta) <= 1e-3 * d;
                        for (int h = 0; h <= 20; h++) {
                            dn = fmin(fmax(d + delta, dmin), dmax);
                            t = eval(dn);
                            ll += n3;
                            if (t.flag == 1) break;
                            if (short_newton || t.l >= r.l) {
                                accepted = true;
                                break;
                            }
                            delta *= 0.5;
                        }
                        // (flag 2: only a point that is taken needs its derivatives;
                        // FP64 goes on from the point before it, whose own hold)
                        if (t.flag == 1 || (accepted && t.flag)) {
                            st = FX_REDO;
                            if (t.flag == 2) kept = it - 1;
                            break;
                        }
                        if (!accepted) break;
                        const double step = fabs(dn - d);
                        d = dn;
                        r = t;
                        de += n3;
                        if (step < 1e-10 * d) break;
                    }
                }
            }
            if (st != FX_REDO || kept) {
                n_llik += ll;
                n_derivs += de;
            }
        }
        if (b.tid == 0) {
            const bool ok = st == LAGP_OK;
            if (st == FX_REDO) atomicAdd(f.redo, 1);
            if (ok || kept) dv[loc] = d;
            if (o.llik) o.llik[loc] = ok ? r.l : CUDART_NAN;
            if (o.dllik) o.dllik[loc] = ok ? r.dl : CUDART_NAN;
            if (o.d2llik) o.d2llik[loc] = ok ? r.d2l : CUDART_NAN;
            if (o.iters) o.iters[loc] = it;
            o.status[loc] = st - kept;
        }
        __syncthreads();
    }
    if (b.tid == 0 && work) {
        atomicAdd(work, n_llik);
        atomicAdd(work + 1, n_derivs);
    }
}

size_t fx_predict_smem(int n, int p) {
    return (size_t)fx_words(n, n + 2) * 16 + ((size_t)n * p + p + 4 * (size_t)n) * 8;
}
size_t fx_mle_smem(int n, int p, int nm) {
    const size_t area = std::max((size_t)nm * fx_words(n, n + 1) * 16, (size_t)n * p * 8);
    return area + (size_t)n * 20 + 64;
}

// Upper ends of the size classes: one launch a class, so that a location's
// shared memory (n^2, 48 KB at n = 60 for the MLE) follows its own design size
// and not the largest one's.  They lie where one CTA less fits an SM for the
// MLE: four up to 64 rows, three to 76, two to 94 (against 40, 64, 80, 104, 128:
// 20,000 locations of 30 to 100 rows, whole method, 307 -> 285 ms).
constexpr int FX_CLASSES[] = {40, 64, 76, 94, 128};

// Calls fn(lo, hi, first) for every class of sizes up to nmax, the largest
// first.  One class when all locations have the same size, and for up to
// sixteen locations a CTA that is resident with the largest one's shared memory
// (smem bytes): the launches run one after the other, each as long as its
// longest location's chain, about 6 ms for the MLE of 33 to 99 rows and 0.7 ms
// for the prediction; beyond, smaller designs gain more from their occupancy
// (MLE 5.8 us a location in one class, 3.4 in five; prediction 0.165, 0.13).
// 26 locations of 33 to 99 rows, prediction: 0.53 -> 0.20 ms, MLE 4.7 -> 1.3 ms;
// 900 locations: 0.79 -> 0.33, 10.6 -> 5.2 ms.
template <typename Fn>
lagp_status fx_each_class(lagp_ctx *ctx, const GpArgs &a, size_t smem, Fn fn) {
    const int64_t fit = std::min<int64_t>(8, (int64_t)(ctx->smem_optin / (smem + 2048)));
    if (!a.n || a.M <= 16 * ctx->num_sms * std::max<int64_t>(fit, 1)) return fn(0, a.nmax, true);
    int hi = a.nmax;
    bool first = true;
    for (int c = (int)(sizeof FX_CLASSES / sizeof *FX_CLASSES) - 1; c >= 0; c--) {
        const int lo = c ? FX_CLASSES[c - 1] : 0;
        if (hi <= lo) continue;
        LAGP_TRY(fn(lo, hi, first));
        first = false;
        hi = lo;
    }
    return LAGP_OK;
}

template <typename Kern>
int fx_grid(lagp_ctx *ctx, Kern kern, int threads, size_t smem, int64_t M) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)ctx->num_sms * std::max(occ, 1), M));
}

}  // namespace

bool gp_fixed_supported(lagp_ctx *ctx, const GpArgs &a, bool mle) {
    if (a.nmax > FX_NMAX || !(a.g < 1.0)) return false;
    return (mle ? fx_mle_smem(a.nmax, a.p, 3) : fx_predict_smem(a.nmax, a.p)) + 2048 <= ctx->smem_optin;
}

size_t gp_fixed_workspace(lagp_ctx *ctx, const GpArgs &a) {
    const size_t ctas = (size_t)std::min<int64_t>((int64_t)ctx->num_sms * 16, a.M);
    return ctas * ((size_t)a.nmax * (a.nmax + 1) / 2) * 8;
}

lagp_status launch_predict_fixed(lagp_ctx *ctx, const GpArgs &a, const double *d, double *mean, double *s2,
                                 double *df, int32_t *status, int *counters, int *redo) {
    return fx_each_class(ctx, a, fx_predict_smem(a.nmax, a.p), [&](int lo, int hi, bool first) -> lagp_status {
        const size_t smem = fx_predict_smem(hi, a.p);
        const int grid = fx_grid(ctx, predict_fx_kernel, FXT, smem, a.M);
        const FxLaunch f{lo, hi, first, fx_words(hi, hi + 2), counters++, redo, nullptr};
        predict_fx_kernel<<<grid, FXT, smem, ctx->stream>>>(a, f, d, mean, s2, df, status);
        ctx->launches++;
        return lagp_cuda_check(ctx, cudaGetLastError(), "predict_fx_kernel");
    });
}

lagp_status launch_mle_fixed(lagp_ctx *ctx, const GpArgs &a, double *d, double dmin, double dmax, int32_t max_iter,
                             const MleOut &o, unsigned long long *work, double *ws, int *counters, int *redo) {
    const int nm = max_iter == 0 && !o.dllik && !o.d2llik ? 1 : 3;
    return fx_each_class(ctx, a, fx_mle_smem(a.nmax, a.p, nm), [&](int lo, int hi, bool first) -> lagp_status {
        const size_t smem = fx_mle_smem(hi, a.p, nm);
        auto go = [&](auto kern, int threads) {
            const int grid = std::min(fx_grid(ctx, kern, threads, smem, a.M), ctx->num_sms * 16);
            const FxLaunch f{lo, hi, first, fx_words(hi, hi + 1), counters++, redo, ws};
            kern<<<grid, threads, smem, ctx->stream>>>(a, f, d, dmin, dmax, max_iter, o, work);
        };
        // where shared memory leaves room for two CTAs an SM, or one, a CTA has
        // twice or three times the warps: 2,000 locations, n = 100, 13.7 -> 11.1 ms
        // (256 threads 11.4, 512 11.6; 256 threads where three CTAs fit: no gain)
        const int fit = (int)(ctx->smem_optin / (smem + 2048));
        if (nm == 1) go(mle_fx_kernel<1, FXT>, FXT);
        else if (fit < 2) go(mle_fx_kernel<3, 3 * FXT>, 3 * FXT);
        else if (fit < 3) go(mle_fx_kernel<3, 2 * FXT>, 2 * FXT);
        else go(mle_fx_kernel<3, FXT>, FXT);
        ctx->launches++;
        return lagp_cuda_check(ctx, cudaGetLastError(), "mle_fx_kernel");
    });
}
