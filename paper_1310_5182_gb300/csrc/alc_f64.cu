// a2..a6, plain FP64 form: greedy ALC local design search (Fig. 1 step 2 of
// the paper) with every candidate's criterion evaluated by Eq. (dxy) in FP64.
//
// Layout: one persistent CTA works on one location at a time (locations are
// taken from an atomic counter).  Shared memory holds K_j^{-1} (FP64, leading
// dimension n_max) and the design's k_j(x); a per-CTA global panel holds
// K(x_c, x_i) for every candidate c and design row i, one column appended per
// step (the paper rebuilds these covariances every step; appending gives the
// same values for N' exponentials per step instead of N' j).
//
// Per step j, one warp per candidate (lane t owns design index t, t+32, ...):
//   b   = K_j^{-1} k_j(x_c)                 (the O(j^2) contraction, paper step 3)
//   m^-1 = 1 + g - k_j(x_c)^T b,  k_j(x)^T g_j = -m k_j(x)^T b   (steps 4-5, 7)
//   Delta = (k^T g)^2 m^-1 + 2 (k^T g) K(x_c,x) + K(x_c,x)^2 m      (Eq. dxy, step 8)
// then a block argmax (ties to the lower design row) and the partitioned
// inverse update of Sec. 2.2.  GB300 runs FP64 at 1/62 of the FP32 rate, so
// this form is bound by the FP64 pipe; it is the plain reference form.
//
// Few locations (at least two resident CTAs a location, as on the
// 100-location 2-d toy): one location per thread-block cluster of CS CTAs
// instead (CS up to 4, not necessarily a power of two).  CTA r of the
// cluster scores, and appends panel columns for, the candidates c with
// c mod CS = r; each step the CTAs exchange their best through distributed
// shared memory (one cluster barrier a step, the records double-buffered by
// the step's parity) and every CTA applies the same partitioned-inverse
// update to its own copy of K^{-1}, reading the winner's panel row from its
// owner's global panel after the barrier: the copies stay identical bit for
// bit, and so do the results whatever CS is.
//
// For nuggets below 1 the contraction runs in 59-bit fixed point on the
// integer pipe (alc_f64fx_kernel below): same criterion, same K^{-1} grown in
// FP64, every candidate's quadratic form evaluated in full each step.
#include <algorithm>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "device_util.cuh"
#include "exp64.cuh"
#include "fx_chol.cuh"
#include "lagp_internal.h"

namespace {

constexpr int F64_THREADS = 256;
constexpr int F64_WARPS = F64_THREADS / 32;
constexpr int NMAX_SMEM = 128;

struct F64Shared {
    double *Kinv;    // nmax x nmax
    double *kx;      // nmax: k_j(x)
    double *yd;      // nmax: responses of the design (fused prediction)
    double *alpha;   // nmax: K^{-1} Y_j (fused prediction)
    double *bstar;   // nmax: K^{-1} k*
    double *part;    // 4 x ld: partial sums of K^{-1} k*
    double *xd;      // nmax x p: design coordinates
    double *xq;      // p: reference location
    unsigned char *chosen;  // Npmax
};

// Contraction for one candidate (paper steps 3-4 and the k_j(x) dot product
// of step 7): lane t accumulates b_t = sum_k K^{-1}[k][t] kc[k] for its
// columns t = lane + 32 r, r < JQ; returns warp-uniform kc^T b and kx^T b.
// K^{-1} rows have leading dimension ld (a multiple of 32), so every read is
// inside the row; columns >= j are masked out of the sums.
template <int JQ>
__device__ __forceinline__ void contract_cand(const double *__restrict__ prow, const double *Kinv,
                                              int ld, const double *kx, int j, int lane,
                                              double &quad, double &kxb) {
    double kc[JQ], b[JQ];
#pragma unroll
    for (int r = 0; r < JQ; r++) {
        kc[r] = (lane + 32 * r < j) ? prow[lane + 32 * r] : 0.0;
        b[r] = 0.0;
    }
#pragma unroll
    for (int r = 0; r < JQ; r++) {
        const int kend = min(32, j - 32 * r);
        for (int kk = 0; kk < kend; kk++) {
            const double v = __shfl_sync(LAGP_FULL_MASK, kc[r], kk);
            const double *row = Kinv + (size_t)(32 * r + kk) * ld + lane;
#pragma unroll
            for (int r2 = 0; r2 < JQ; r2++) b[r2] = fma(row[32 * r2], v, b[r2]);
        }
    }
    double q = 0.0, x = 0.0;
#pragma unroll
    for (int r = 0; r < JQ; r++)
        if (lane + 32 * r < j) {
            q = fma(kc[r], b[r], q);
            x = fma(kx[lane + 32 * r], b[r], x);
        }
    quad = warp_sum(q);
    kxb = warp_sum(x);
}

__device__ __forceinline__ double kern64(const double *a, const void *X, int64_t r, int p,
                                         lagp_dtype dt, double d) {
    double s = 0.0;
    for (int i = 0; i < p; i++) {
        double diff = a[i] - load_coord64(X, r, p, i, dt);
        s += diff * diff;
    }
    return exp(-s / d);
}

namespace cg = cooperative_groups;

// CL: one location per cluster (candidates split over its CTAs)
template <bool CL>
__global__ void __launch_bounds__(F64_THREADS)
alc_f64_kernel(AlcArgs a, int *__restrict__ counter, double *__restrict__ panel_ws,
               double *__restrict__ kappa_ws) {
    // after the fixed-point kernel: the locations it left (status FX_REDO)
    if (a.retry_count && *a.retry_count == 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nmax = a.nmax, p = a.p, Npmax = a.Npmax;
    const int ld = (nmax + 31) & ~31;  // K^{-1} leading dimension
    F64Shared S;
    S.Kinv = reinterpret_cast<double *>(smem_raw);
    S.kx = S.Kinv + (size_t)(nmax + 1) * ld;
    S.yd = S.kx + ld;
    S.alpha = S.yd + ld;
    S.bstar = S.alpha + ld;
    S.part = S.bstar + nmax;
    S.xd = S.part + 4 * (size_t)ld;
    S.xq = S.xd + (size_t)nmax * p;
    S.chosen = reinterpret_cast<unsigned char *>(S.xq + p);
    __shared__ int s_loc, s_bad, s_cstar;
    __shared__ double w_v[F64_WARPS];
    __shared__ int w_row[F64_WARPS], w_slot[F64_WARPS];
    __shared__ double s_delta, s_mu, s_ry, s_cx, s_psi, s_qx, s_ystar;
    // the cluster's exchange of the step's best (by the step's parity)
    __shared__ double x_v[2];
    __shared__ int x_row[2], x_slot[2], x_bad[2];
    const bool fused = a.mean != nullptr;

    double *panel = panel_ws + (size_t)blockIdx.x * Npmax * nmax;  // [c][i], ld nmax
    double *kappa = kappa_ws + (size_t)blockIdx.x * Npmax;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // cluster rank and size (1 and 0 without clusters); candidates c with
    // c mod CS = rank are this CTA's
    const int CS = CL ? (int)cg::this_cluster().num_blocks() : 1;
    const int rank = CL ? (int)cg::this_cluster().block_rank() : 0;
    int64_t next_loc = CL ? blockIdx.x / CS : 0;

    for (;;) {
        int64_t loc;
        if constexpr (CL) {
            loc = next_loc;  // a static share of the locations per cluster
            next_loc += gridDim.x / CS;
        } else {
            if (tid == 0) s_loc = atomicAdd(counter, 1);
            __syncthreads();
            loc = s_loc;
            __syncthreads();
        }
        if (loc >= a.M) break;
        if (a.retry_count && a.status[loc] != FX_REDO) continue;

        const int k = a.Np ? a.Np[loc] : Npmax;
        const int nm = a.n ? a.n[loc] : nmax;
        const double d = a.d[loc], g = a.g;
        const int32_t *cands = a.idx + loc * Npmax;
        int32_t *sel = a.sel + loc * nmax;
        double *alc = a.alc ? a.alc + loc * nmax : nullptr;

        // per-location validation
        if (tid == 0) s_bad = (k < 1 || k > Npmax || nm < a.n0 || nm > nmax || nm > k || !(d > 0.0) ||
                               !isfinite(d)) ? LAGP_EINVAL : LAGP_OK;
        __syncthreads();
        if (s_bad == LAGP_OK)
            for (int c = tid; c < k; c += F64_THREADS) {
                int32_t r = cands[c];
                if (r < 0 || r >= a.N) s_bad = LAGP_EINVAL;
            }
        __syncthreads();
        // (outputs: the cluster's rank 0 alone writes them)
        if (rank == 0)
            for (int t = tid; t < nmax; t += F64_THREADS) {
                sel[t] = -1;
                if (alc) alc[t] = CUDART_NAN;
            }
        if (s_bad != LAGP_OK) {
            if (tid == 0 && rank == 0) {
                a.status[loc] = s_bad;
                if (fused) a.mean[loc] = a.s2[loc] = a.df[loc] = CUDART_NAN;
            }
            __syncthreads();
            continue;  // next location
        }

        // reference location, chosen flags, K(x_c, x) for every candidate
        for (int i = tid; i < p; i += F64_THREADS) S.xq[i] = load_coord64(a.Xref, loc, p, i, a.dtype);
        for (int c = tid; c < k; c += F64_THREADS) S.chosen[c] = 0;
        __syncthreads();
        for (int c = tid; c < k; c += F64_THREADS) kappa[c] = kern64(S.xq, a.X, cands[c], p, a.dtype, d);
        __syncthreads();

        int status = LAGP_OK;
        if (tid == 0) s_psi = s_qx = 0.0;
        for (int j = 0; j < nm; j++) {
            int cstar;
            double delta = CUDART_NAN;
            if (j < a.n0) {
                cstar = j;  // Fig. 1 step 2(a): the nearest neighbours, in order
                // (the owner's panel row of the seed is read after the barrier)
                if constexpr (CL) cg::this_cluster().sync();
            } else {
                // ---- score every unchosen candidate (this CTA's share), one
                // warp per candidate
                ArgBest best{0.0, -1, -1};
                for (int c = rank + CS * warp; c < k; c += CS * F64_WARPS) {
                    if (S.chosen[c]) continue;
                    const double *prow = panel + (size_t)c * nmax;
                    double quad, kxb;
                    switch ((j + 31) >> 5) {
                        case 1: contract_cand<1>(prow, S.Kinv, ld, S.kx, j, lane, quad, kxb); break;
                        case 2: contract_cand<2>(prow, S.Kinv, ld, S.kx, j, lane, quad, kxb); break;
                        case 3: contract_cand<3>(prow, S.Kinv, ld, S.kx, j, lane, quad, kxb); break;
                        default: contract_cand<4>(prow, S.Kinv, ld, S.kx, j, lane, quad, kxb); break;
                    }
                    const double minv = (1.0 + g) - quad;  // m_j^{-1}(x_c), Eq. (piedef)
                    const double m = 1.0 / minv;
                    const double kxg = -m * kxb;           // k_j(x)^T g_j(x_c)
                    const double kap = kappa[c];
                    double dl = kxg * kxg * minv + 2.0 * kxg * kap + kap * kap * m;
                    if (!(minv > 0.0)) dl = -CUDART_INF;  // breakdown, flagged below
                    if (!(minv > 0.0) && lane == 0) s_bad = LAGP_ENOTPD;
                    if (better(dl, cands[c], best.v, best.row)) best = ArgBest{dl, cands[c], c};
                }
                if (lane == 0) {
                    w_v[warp] = best.v;
                    w_row[warp] = best.row;
                    w_slot[warp] = best.slot;
                }
                __syncthreads();
                if (tid == 0) {
                    ArgBest b0{w_v[0], w_row[0], w_slot[0]};
                    for (int w = 1; w < F64_WARPS; w++)
                        if (better(w_v[w], w_row[w], b0.v, b0.row)) b0 = ArgBest{w_v[w], w_row[w], w_slot[w]};
                    s_cstar = b0.slot;
                    s_delta = b0.v;
                    if constexpr (CL) {
                        x_v[j & 1] = b0.v;
                        x_row[j & 1] = b0.row;
                        x_slot[j & 1] = b0.slot;
                        x_bad[j & 1] = s_bad;
                    } else if (b0.slot < 0) {
                        s_bad = LAGP_ENOTPD;
                    }
                }
                if constexpr (CL) {
                    // the cluster's best (ties to the lower row), the same in every CTA
                    cg::cluster_group cl = cg::this_cluster();
                    cl.sync();
                    if (tid == 0) {
                        ArgBest b0{-CUDART_INF, INT32_MAX, -1};
                        int bad = LAGP_OK;
                        for (int r = 0; r < CS; r++) {
                            const double v = *cl.map_shared_rank(&x_v[j & 1], r);
                            const int row = *cl.map_shared_rank(&x_row[j & 1], r);
                            const int slot = *cl.map_shared_rank(&x_slot[j & 1], r);
                            const int rb = *cl.map_shared_rank(&x_bad[j & 1], r);
                            if (rb != LAGP_OK) bad = rb;
                            if (slot >= 0 && (b0.slot < 0 || better(v, row, b0.v, b0.row))) b0 = ArgBest{v, row, slot};
                        }
                        s_cstar = b0.slot;
                        s_delta = b0.v;
                        s_bad = bad != LAGP_OK ? bad : (b0.slot < 0 ? LAGP_ENOTPD : LAGP_OK);
                    }
                }
                __syncthreads();
                if (s_bad != LAGP_OK) {
                    status = s_bad;
                    break;
                }
                cstar = s_cstar;
                delta = s_delta;
            }
            // ---- partitioned inverse update with x* = candidate cstar (Sec. 2.2);
            // its panel row from the CTA that owns it
            const double *kst =
                (CL ? panel_ws + (size_t)(blockIdx.x - rank + cstar % CS) * Npmax * nmax : panel) +
                (size_t)cstar * nmax;
            // b* = K^{-1} k*: each output summed by QS threads over a share of
            // the rows, two chains each (short dependent FP64 chains)
            {
                const int QS = j * 4 <= F64_THREADS ? 4 : (j * 2 <= F64_THREADS ? 2 : 1);
                for (int e = tid; e < j * QS; e += F64_THREADS) {
                    const int t = e % j, q = e / j, k0 = q * j / QS, k1 = (q + 1) * j / QS;
                    double s0 = 0.0, s1 = 0.0;
                    int kk = k0;
                    for (; kk + 1 < k1; kk += 2) {
                        s0 = fma(S.Kinv[(size_t)kk * ld + t], kst[kk], s0);
                        s1 = fma(S.Kinv[(size_t)(kk + 1) * ld + t], kst[kk + 1], s1);
                    }
                    if (kk < k1) s0 = fma(S.Kinv[(size_t)kk * ld + t], kst[kk], s0);
                    S.part[(size_t)q * ld + t] = s0 + s1;
                }
                __syncthreads();
                for (int t = tid; t < j; t += F64_THREADS) {
                    double s = S.part[t];
                    for (int q = 1; q < QS; q++) s += S.part[(size_t)q * ld + t];
                    S.bstar[t] = s;
                }
            }
            __syncthreads();
            if (tid < 32) {
                double q = 0.0, xb = 0.0, yb = 0.0;
                for (int t = lane; t < j; t += 32) {
                    q = fma(kst[t], S.bstar[t], q);
                    if (fused) {
                        xb = fma(S.kx[t], S.bstar[t], xb);
                        yb = fma(S.yd[t], S.bstar[t], yb);
                    }
                }
                q = warp_sum(q);
                if (fused) {
                    xb = warp_sum(xb);
                    yb = warp_sum(yb);
                }
                if (lane == 0) {
                    double minv = (1.0 + g) - q;
                    s_mu = 1.0 / minv;
                    if (!(minv > 0.0)) s_bad = LAGP_ENOTPD;
                    if (fused) {
                        const int32_t row = cands[cstar];
                        s_ystar = a.dtype == LAGP_F64 ? static_cast<const double *>(a.Y)[row]
                                                      : (double)static_cast<const float *>(a.Y)[row];
                        s_ry = s_ystar - yb;          // y* - Y_j^T K^{-1} k*
                        s_cx = kappa[cstar] - xb;     // K(x*,x) - k_j(x)^T K^{-1} k*
                    }
                }
            }
            __syncthreads();
            if (s_bad != LAGP_OK) {
                status = s_bad;
                break;
            }
            const double mu = s_mu;
            // K^{-1} + g g^T / m with g = -mu b*:  += mu b* b*^T (lower triangle
            // and its mirror) ; border = -mu b*
            for (int e = tid; e < j * (j + 1) / 2; e += F64_THREADS) {
                int r = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
                while ((r + 1) * (r + 2) / 2 <= e) r++;
                while (r * (r + 1) / 2 > e) r--;
                const int c = e - r * (r + 1) / 2;
                const double val = fma(mu * S.bstar[r], S.bstar[c], S.Kinv[(size_t)r * ld + c]);
                S.Kinv[(size_t)r * ld + c] = val;
                S.Kinv[(size_t)c * ld + r] = val;
            }
            const double ry = fused ? s_ry : 0.0;
            for (int t = tid; t < j; t += F64_THREADS) {
                double gt = -mu * S.bstar[t];
                S.Kinv[(size_t)t * ld + j] = gt;
                S.Kinv[(size_t)j * ld + t] = gt;
                if (fused) S.alpha[t] = fma(-mu * ry, S.bstar[t], S.alpha[t]);
            }
            if (tid == 0) {
                if (fused) {
                    // Eqs. (predgp), (preds2) carried by the partitioned inverse
                    S.alpha[j] = mu * ry;
                    S.yd[j] = s_ystar;
                    s_psi = fma(mu * ry, ry, s_psi);
                    s_qx = fma(mu * s_cx, s_cx, s_qx);
                }
                S.Kinv[(size_t)j * ld + j] = mu;
                S.kx[j] = kappa[cstar];
                S.chosen[cstar] = 1;
                if (rank == 0) {
                    sel[j] = cands[cstar];
                    if (alc) alc[j] = delta;
                }
            }
            for (int i = tid; i < p; i += F64_THREADS)
                S.xd[(size_t)j * p + i] = load_coord64(a.X, cands[cstar], p, i, a.dtype);
            __syncthreads();
            // ---- append panel column j: K(x_c, x*) for every candidate (no nugget)
            if (j + 1 < nm) {
                const double *xs = S.xd + (size_t)j * p;
                for (int c = rank + CS * tid; c < k; c += CS * F64_THREADS)
                    panel[(size_t)c * nmax + j] = kern64(xs, a.X, cands[c], p, a.dtype, d);
            }
            __syncthreads();
        }
        if (status != LAGP_OK && rank == 0) {
            for (int t = tid; t < nmax; t += F64_THREADS) {
                sel[t] = -1;
                if (alc) alc[t] = CUDART_NAN;
            }
        }
        if (fused) {
            __syncthreads();
            if (warp == 0 && rank == 0) {
                double m = 0.0;
                for (int t = lane; t < nm; t += 32) m = fma(S.kx[t], S.alpha[t], m);
                m = warp_sum(m);
                if (lane == 0) {
                    const bool ok = status == LAGP_OK;
                    a.mean[loc] = ok ? m : CUDART_NAN;
                    a.s2[loc] = ok ? s_psi * ((1.0 + g) - s_qx) / nm : CUDART_NAN;
                    a.df[loc] = ok ? (double)nm : CUDART_NAN;
                }
            }
        }
        if (tid == 0 && rank == 0) a.status[loc] = status;
        __syncthreads();
    }
    // no CTA leaves while another may still read its exchange records
    if constexpr (CL) cg::this_cluster().sync();
}

// ------------------------------------------------ the contraction in fixed point
//
// One thread per candidate.  k_j(x_c)^T K_j^{-1} k_j(x_c) = 2 sum_t k_t c_t with
// c_t = sum_{i<t} (K^{-1})_{ti} k_i + (K^{-1})_{tt} k_t / 2 (the matrix is
// symmetric: half the products of K^{-1} k), and k_j(x)^T K^{-1} k_j(x_c) =
// a^T k_j(x_c) with a = K_j^{-1} k_j(x) carried along by the partitioned inverse.
// K^{-1} and a enter as limbs scaled by 2^-es, es four above the exponent of
// K^{-1}'s largest diagonal entry (no entry is larger; the partial sums c_t
// then stay in range), so that the quadratic form carries an error of about
// 2^(es - 59) sqrt(j), below the 2^-53 |k|^T |K^{-1}| |k| of an FP64 evaluation.
// The covariances are absolute (2^-59), so that this holds where the winner's
// are not small.  R = K(x*, x) - k_j(x)^T K^{-1} k* carries up to 2^(es - 58) (1 +
// |k*|_1) here, and 2^(es - 57) |k_j(x)|_1 |k*|_1 in FP64 (the K^{-1} basis): a step
// is trusted when the second is at least a quarter of the first, or |R| is 2^30
// times the first.  The winner's criterion is evaluated again in FP64, from the
// products that the update of K^{-1} needs.  A location with a step that is not
// trusted is left to the FP64 kernel, and so is one whose nearest candidate
// has K(x_c, x) < 2^-6 or whose values leave the range.  (With candidates many
// lengthscales apart the criterion of all but the nearest would be noise.)
//
// Bound: the integer multiply pipe; a product costs three multiply-adds, 12
// cycles a warp against 64 on the FP64 unit, and half as many are made; the
// exponentials and the criterion's scalars stay in FP64 and overlap.  B rows
// t at a time share a candidate's k_i (8 bytes from the panel) and read the
// limbs of K^{-1} as broadcasts (no result depends on B).  Measured: 100
// locations of the 2-d toy, n = 50, N' = 1000, 20.7 -> 2.9 ms (one CTA an SM, B
// = 8; two with B = 4: 3.2; 2.84 now); 1,000 locations in 5 dimensions 186 -> 16.4 ms
// (two CTAs, B = 4; one with B = 8: 19.5; 256 threads: 20.7).
constexpr int PF_THREADS = 512;
constexpr int PF_BMAX = 8;
constexpr int PF_HEAD = 4;
// Products between folds of a middle sum: covariances are at most 1 and K^{-1}'s
// limbs at most 2^-4, so that 28 products stay below 2^63; c_t and a are below 2,
// so that the up to 8 rows of a block do (3 2^58 each).  Without folds a sum
// of 56 equal products wrapped (equidistant rows), and at n = 112 of dense rows
// the largest of 10^6 came to 0.65 2^63.
constexpr int PF_FOLD = 24;

__host__ __device__ inline int pf_ld(int nmax) { return nmax | 1; }
__host__ __device__ inline int pf_ldk(int nmax) { return (nmax + PF_BMAX - 1) / PF_BMAX * PF_BMAX; }
__host__ __device__ inline size_t pf_smem(int nmax, int p) {
    const size_t ldk = pf_ldk(nmax);
    return ((size_t)nmax * pf_ld(nmax) + (size_t)nmax * ldk + ldk + 6 * (size_t)nmax + (size_t)nmax * p + p) * 8 + 64;
}

template <int B>
__global__ void __launch_bounds__(PF_THREADS, B == PF_BMAX ? 1 : 2)
alc_f64fx_kernel(AlcArgs a, int *__restrict__ counter, int *__restrict__ redo, int2 *__restrict__ panel_ws,
                 double *__restrict__ kappa_ws, double *__restrict__ coord_ws, unsigned char *__restrict__ chosen_ws) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nmax = a.nmax, p = a.p, Npmax = a.Npmax, ld = pf_ld(nmax), ldk = pf_ldk(nmax);
    int2 *KL = reinterpret_cast<int2 *>(smem_raw);                 // nmax x ldk: limbs of K^{-1}[i][t], t >= i
    int2 *aL = KL + (size_t)nmax * ldk;                            // ldk: limbs of a
    double *Kinv = reinterpret_cast<double *>(aL + ldk);           // nmax x ld
    double *kx = Kinv + (size_t)nmax * ld, *yd = kx + nmax, *alpha = yd + nmax, *bstar = alpha + nmax,
           *av = bstar + nmax, *kst = av + nmax;                   // nmax each
    double *xd = kst + nmax, *xq = xd + (size_t)nmax * p;
    constexpr int W = PF_THREADS / 32;
    __shared__ int s_loc, s_bad, s_cstar, s_top;
    __shared__ double w_v[W], s_delta, s_mu, s_ry, s_cx, s_psi, s_qx, s_ystar;
    __shared__ int w_row[W], w_slot[W];
    const bool fused = a.mean != nullptr;
    int2 *panel = panel_ws + (size_t)blockIdx.x * nmax * Npmax;    // [i][c]
    double *kappa = kappa_ws + (size_t)blockIdx.x * Npmax;
    double *cx = coord_ws + (size_t)blockIdx.x * p * Npmax;         // [i][c]: candidate coordinates
    unsigned char *chosen = chosen_ws + (size_t)blockIdx.x * Npmax;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    for (;;) {
        if (tid == 0) s_loc = atomicAdd(counter, 1);
        __syncthreads();
        const int64_t loc = s_loc;
        __syncthreads();
        if (loc >= a.M) break;
        const int k = a.Np ? a.Np[loc] : Npmax;
        const int nm = a.n ? a.n[loc] : nmax;
        const double d = a.d[loc], g = a.g, ninv_d = -1.0 / d;
        const int32_t *cands = a.idx + loc * Npmax;
        int32_t *sel = a.sel + loc * nmax;
        double *alc = a.alc ? a.alc + loc * nmax : nullptr;
        if (tid == 0) {
            s_bad = (k < 1 || k > Npmax || nm < a.n0 || nm > nmax || nm > k || !(d > 0.0) || !isfinite(d))
                        ? LAGP_EINVAL : LAGP_OK;
            s_top = 0;
            s_psi = s_qx = 0.0;
        }
        __syncthreads();
        if (s_bad == LAGP_OK)
            for (int c = tid; c < k; c += PF_THREADS) {
                const int32_t r = cands[c];
                if (r < 0 || r >= a.N) s_bad = LAGP_EINVAL;
            }
        __syncthreads();
        for (int t = tid; t < nmax; t += PF_THREADS) {
            sel[t] = -1;
            if (alc) alc[t] = CUDART_NAN;
        }
        if (s_bad != LAGP_OK) {
            if (tid == 0) {
                a.status[loc] = s_bad;
                if (fused) a.mean[loc] = a.s2[loc] = a.df[loc] = CUDART_NAN;
            }
            __syncthreads();
            continue;
        }
        for (int i = tid; i < p; i += PF_THREADS) xq[i] = load_coord64(a.Xref, loc, p, i, a.dtype);
        for (int e = tid; e < nmax * ldk; e += PF_THREADS) KL[e] = make_int2(0, 0);
        for (int e = tid; e < ldk; e += PF_THREADS) aL[e] = make_int2(0, 0);
        __syncthreads();
        // squared distance of candidate c to a point
        auto dist = [&](const double *at, int c) {
            double s = 0.0;
            for (int i = 0; i < p; i++) {
                const double df = at[i] - cx[(size_t)i * Npmax + c];
                s = fma(df, df, s);
            }
            return s;
        };
        bool odd = false;
        for (int c = tid; c < k; c += PF_THREADS) {
            for (int i = 0; i < p; i++) cx[(size_t)i * Npmax + c] = load_coord64(a.X, cands[c], p, i, a.dtype);
            const double s = dist(xq, c);
            odd |= !(s < CUDART_INF);
            const double v = exp64_tang(s * ninv_d, exp64_table_g);
            kappa[c] = v;
            chosen[c] = 0;
            if (v >= 0x1p-6) s_top = 1;
        }
        odd = __syncthreads_or(odd);
        int status = odd || s_top == 0 ? FX_REDO : LAGP_OK;
        __syncthreads();
        if (tid == 0) s_top = 0;  // from here: exponent field of the largest diagonal entry
        for (int j = 0; j < nm && status == LAGP_OK; j++) {
            int cstar;
            if (j < a.n0) {
                cstar = j;  // Fig. 1 step 2(a): the nearest neighbours, in order
            } else {
                const int es = s_top - 1022 + PF_HEAD;
                ArgBest best{0.0, -1, -1};
                unsigned bad = 0;
                for (int c = tid; c < k; c += PF_THREADS) {
                    if (chosen[c]) continue;
                    const int2 *pc = panel + c;
                    long long qh = 0, qm = FX_HALF, xh = 0, xm = FX_HALF;
                    for (int t0 = 0; t0 < j; t0 += B) {
                        long long hi[B], mid[B];
#pragma unroll
                        for (int r = 0; r < B; r++) hi[r] = 0, mid[r] = FX_HALF;
                        for (int i0 = 0; i0 < t0; i0 += PF_FOLD) {
                            const int i1 = min(i0 + PF_FOLD, t0);
#pragma unroll 2
                            for (int i = i0; i < i1; i++) {
                                const int2 u = pc[(size_t)i * Npmax];
                                const int4 *row = reinterpret_cast<const int4 *>(KL + (size_t)i * ldk + t0);
#pragma unroll
                                for (int r = 0; r < B; r += 2) {
                                    const int4 l = row[r / 2];
                                    hi[r] = fx_mad(u.x, l.x, hi[r]);
                                    mid[r] = fx_mad(u.y, l.x, fx_mad(u.x, l.y, mid[r]));
                                    hi[r + 1] = fx_mad(u.x, l.z, hi[r + 1]);
                                    mid[r + 1] = fx_mad(u.y, l.z, fx_mad(u.x, l.w, mid[r + 1]));
                                }
                            }
#pragma unroll
                            for (int r = 0; r < B; r++) fx_fold_half(hi[r], mid[r]);
                        }
#pragma unroll
                        for (int r = 0; r < B; r++) {  // the diagonal block (its diagonal halved)
                            if (t0 + r >= j) break;
                            const int2 u = pc[(size_t)(t0 + r) * Npmax], al = aL[t0 + r];
#pragma unroll
                            for (int q = r; q < B; q++) {
                                const int2 l = KL[(size_t)(t0 + r) * ldk + t0 + q];
                                hi[q] = fx_mad(u.x, l.x, hi[q]);
                                mid[q] = fx_mad(u.y, l.x, fx_mad(u.x, l.y, mid[q]));
                            }
                            const Fx ct = fx_split((hi[r] << 1) + (mid[r] >> 29)), uf{u.x, u.y};
                            bad |= (unsigned)(ct.h + (1 << 30)) >> 31;
                            qh = fx_hi(qh, ct, uf);
                            qm = fx_mid(qm, ct, uf);
                            xh = fx_hi(xh, Fx{al.x, al.y}, uf);
                            xm = fx_mid(xm, Fx{al.x, al.y}, uf);
                        }
                        fx_fold(qh, qm);
                        fx_fold(xh, xm);
                    }
                    const double quad = fx_double(fx_sum(qh, qm), es + 1), kxb = fx_double(fx_sum(xh, xm), es);
                    const double minv = (1.0 + g) - quad;  // m_j^{-1}(x_c), Eq. (piedef)
                    const double m = 1.0 / minv;
                    const double kxg = -m * kxb;           // k_j(x)^T g_j(x_c)
                    const double kap = kappa[c];
                    const double dl = kxg * kxg * minv + 2.0 * kxg * kap + kap * kap * m;
                    bad |= !(minv > 0.0);  // for FP64 to decide
                    if (better(dl, cands[c], best.v, best.row)) best = ArgBest{dl, cands[c], c};
                }
                best = warp_argmax(best);
                if (lane == 0) {
                    w_v[warp] = best.v;
                    w_row[warp] = best.row;
                    w_slot[warp] = best.slot;
                }
                if (__syncthreads_or(bad)) {
                    status = FX_REDO;
                    break;
                }
                if (warp == 0) {
                    ArgBest b0{lane < W ? w_v[lane] : 0.0, lane < W ? w_row[lane] : -1, lane < W ? w_slot[lane] : -1};
                    b0 = warp_argmax(b0);
                    if (lane == 0) s_cstar = b0.slot;
                }
                __syncthreads();
                cstar = s_cstar;
                if (cstar < 0) {  // (no candidate compares: left to FP64 as well)
                    status = FX_REDO;
                    break;
                }
            }
            // ---- partitioned inverse update with x* = candidate cstar (Sec. 2.2)
            const int32_t rstar = cands[cstar];
            for (int i = tid; i < p; i += PF_THREADS) xd[(size_t)j * p + i] = cx[(size_t)i * Npmax + cstar];
            for (int t = tid; t < j; t += PF_THREADS)
                kst[t] = exp64_tang(dist(xd + (size_t)t * p, cstar) * ninv_d, exp64_table_g);
            __syncthreads();
            // b* = K^{-1} k*: a quarter warp an output, two chains a lane
            for (int t = tid >> 3; t < j; t += PF_THREADS / 8) {
                double s0 = 0.0, s1 = 0.0;
                const double *row = Kinv + (size_t)t * ld;
                for (int i = tid & 7; i < j; i += 16) {
                    s0 = fma(row[i], kst[i], s0);
                    if (i + 8 < j) s1 = fma(row[i + 8], kst[i + 8], s1);
                }
                s0 += s1;
                const unsigned m8 = 0xffu << (lane & 24);
                for (int o = 4; o > 0; o >>= 1) s0 += __shfl_xor_sync(m8, s0, o);
                if ((tid & 7) == 0) bstar[t] = s0;
            }
            __syncthreads();
            if (warp == 0) {
                double q = 0.0, xb = 0.0, yb = 0.0;
                float ks = 0.f, xs = 0.f;
                for (int t = lane; t < j; t += 32) {
                    q = fma(kst[t], bstar[t], q);
                    xb = fma(kx[t], bstar[t], xb);
                    ks += (float)kst[t];
                    xs += (float)kx[t];
                    if (fused) yb = fma(yd[t], bstar[t], yb);
                }
                q = warp_sum(q);
                xb = warp_sum(xb);
                if (fused) yb = warp_sum(yb);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    ks += __shfl_xor_sync(LAGP_FULL_MASK, ks, o);
                    xs += __shfl_xor_sync(LAGP_FULL_MASK, xs, o);
                }
                if (lane == 0) {
                    const double minv = (1.0 + g) - q, kap = kappa[cstar], m = 1.0 / minv;
                    s_mu = m;
                    if (!(minv > 0.0)) s_bad = FX_REDO;
                    s_cx = kap - xb;  // K(x*,x) - k_j(x)^T K^{-1} k*
                    if (j >= a.n0) {
                        const double kxg = -m * xb;
                        s_delta = kxg * kxg * minv + 2.0 * kxg * kap + kap * kap * m;
                        const float err = ldexpf(1.f + ks, s_top - 1022 + PF_HEAD - 58);
                        if (!(8.f * xs * ks >= 1.f + ks) && !(fabs(s_cx) >= 0x1p30 * err)) s_bad = FX_REDO;
                    }
                    if (fused) {
                        s_ystar = a.dtype == LAGP_F64 ? static_cast<const double *>(a.Y)[rstar]
                                                      : (double)static_cast<const float *>(a.Y)[rstar];
                        s_ry = s_ystar - yb;  // y* - Y_j^T K^{-1} k*
                    }
                }
            }
            __syncthreads();
            if (s_bad != LAGP_OK) {
                status = s_bad;
                break;
            }
            const double mu = s_mu, ex = mu * s_cx, ry = fused ? s_ry : 0.0;
            // K^{-1} += mu b* b*^T (lower triangle and its mirror), border -mu b*
            for (int e = tid; e < j * (j + 1) / 2; e += PF_THREADS) {
                int r = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
                if ((r + 1) * (r + 2) / 2 <= e) r++;
                if (r * (r + 1) / 2 > e) r--;
                const int c = e - r * (r + 1) / 2;
                const double val = fma(mu * bstar[r], bstar[c], Kinv[(size_t)r * ld + c]);
                Kinv[(size_t)r * ld + c] = val;
                Kinv[(size_t)c * ld + r] = val;
                if (r == c) atomicMax(&s_top, (__double2hiint(val) >> 20) & 0x7ff);
            }
            for (int t = tid; t < j; t += PF_THREADS) {
                const double gt = -mu * bstar[t];
                Kinv[(size_t)t * ld + j] = gt;
                Kinv[(size_t)j * ld + t] = gt;
                av[t] = fma(-ex, bstar[t], av[t]);  // a = K^{-1} k(x)
                if (fused) alpha[t] = fma(-mu * ry, bstar[t], alpha[t]);
            }
            if (tid == 0) {
                if (fused) {
                    // Eqs. (predgp), (preds2) carried by the partitioned inverse
                    alpha[j] = mu * ry;
                    yd[j] = s_ystar;
                    s_psi = fma(mu * ry, ry, s_psi);
                    s_qx = fma(mu * s_cx, s_cx, s_qx);
                }
                Kinv[(size_t)j * ld + j] = mu;
                atomicMax(&s_top, (__double2hiint(mu) >> 20) & 0x7ff);
                av[j] = ex;
                kx[j] = kappa[cstar];
                chosen[cstar] = 1;
                sel[j] = rstar;
                if (alc && j >= a.n0) alc[j] = s_delta;
            }
            __syncthreads();
            if (j + 1 < nm) {
                // the limbs of K^{-1} (lower triangle, diagonal halved) and a
                const int es = s_top - 1022 + PF_HEAD;
                if (j + 1 >= a.n0)
                    for (int e = tid; e < (j + 1) * (j + 2) / 2 + j + 1; e += PF_THREADS) {
                        int r = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
                        if ((r + 1) * (r + 2) / 2 <= e) r++;
                        if (r * (r + 1) / 2 > e) r--;
                        const int c = e - r * (r + 1) / 2;
                        const double v = r > j ? av[c] : Kinv[(size_t)r * ld + c];
                        // (|a| <= (j + 1) max |K^{-1}|: four bits of headroom and the range of 4 hold it;
                        // a value that large is left out of range for the check below)
                        const double w = fx_shift(v, -(r == c ? es + 1 : es));
                        if (!(fabs(w) < 2.0)) s_bad = FX_REDO;
                        const Fx f = fx_split(fx_from(fabs(w) < 2.0 ? w : 0.0));
                        (r > j ? aL[c] : KL[(size_t)c * ldk + r]) = make_int2(f.h, f.l);
                    }
                // ---- panel row j: K(x_c, x*) for every candidate (no nugget)
                const double *xs = xd + (size_t)j * p;
                for (int c = tid; c < k; c += PF_THREADS) {
                    const Fx f = fx_split(fx_from(exp64_tang(dist(xs, c) * ninv_d, exp64_table_g)));
                    panel[(size_t)j * Npmax + c] = make_int2(f.h, f.l);
                }
            }
            __syncthreads();
            if (s_bad != LAGP_OK) {
                status = s_bad;
                break;
            }
        }
        __syncthreads();
        if (status != LAGP_OK)
            for (int t = tid; t < nmax; t += PF_THREADS) {
                sel[t] = -1;
                if (alc) alc[t] = CUDART_NAN;
            }
        if (fused && warp == 0) {
            double m = 0.0;
            for (int t = lane; t < nm; t += 32) m = fma(kx[t], alpha[t], m);
            m = warp_sum(m);
            if (lane == 0) {
                const bool ok = status == LAGP_OK;
                a.mean[loc] = ok ? m : CUDART_NAN;
                a.s2[loc] = ok ? s_psi * ((1.0 + g) - s_qx) / nm : CUDART_NAN;
                a.df[loc] = ok ? (double)nm : CUDART_NAN;
            }
        }
        if (tid == 0) {
            a.status[loc] = status;
            if (status == FX_REDO) atomicAdd(redo, 1);
        }
        __syncthreads();
    }
}

}  // namespace

lagp_status launch_alc_f64(lagp_ctx *ctx, const AlcArgs &args) {
    AlcArgs a = args;
    if (a.nmax > NMAX_SMEM)
        return lagp_fail(ctx, LAGP_EINVAL, "lagp_alc_select: n_max above 128 is not supported");
    cudaStream_t st = ctx->stream;
    const size_t ld = (size_t)((a.nmax + 31) & ~31);
    // K^{-1} (n_max x ld, plus one spare row so masked reads stay inside), kx, b*,
    // design coordinates, reference location, chosen flags
    size_t smem = ((size_t)a.nmax + 1) * ld * 8 + ld * 8 * 4 + 4 * ld * 8 + (size_t)a.nmax * a.p * 8 +
                  (size_t)a.p * 8 + (size_t)a.Npmax + 16;
    if (smem > ctx->smem_optin) return lagp_fail(ctx, LAGP_EINVAL, "lagp_alc_select: shared memory");
    // cluster size: with few locations, the CTAs of a cluster share one
    // location's candidates, as many as keep every cluster resident at once
    // (at most 4; 1 = no clusters, and whenever the user fixes the CTAs per SM)
    int cs = 1;
    if (ctx->tuning.ctas_per_sm == 0 && ctx->tune_override == 0) {
        cudaFuncSetAttribute(alc_f64_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int occ = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, alc_f64_kernel<true>, F64_THREADS, smem);
        const int64_t fit = (int64_t)ctx->num_sms * std::max(occ, 1) / std::max<int64_t>(a.M, 1);
        cs = (int)std::min<int64_t>(4, fit);  // (4 measured faster than 6 on the 2-d toy)
        if (cs < 2) cs = 1;
    }
    int64_t grid;
    if (cs > 1) {
        ctx->last_alc_key = alc_shape_key("alc_f64", 0, a.nmax, a.p, a.mean != nullptr);
        grid = a.M * cs;
    } else {
        cudaFuncSetAttribute(alc_f64_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int occ = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, alc_f64_kernel<false>, F64_THREADS, smem);
        int per_sm = alc_ctas_per_sm(ctx, alc_shape_key("alc_f64", 0, a.nmax, a.p, a.mean != nullptr), 2);
        if (occ > 0 && per_sm > occ) per_sm = occ;
        grid = (int64_t)ctx->num_sms * per_sm;
        if (grid > a.M) grid = a.M;
        if (grid < 1) grid = 1;
    }
    // in fixed point where that holds (nugget below 1, K^{-1} twice in shared
    // memory: n_max up to about 115), then in FP64 what it leaves
    const size_t smem_fx = pf_smem(a.nmax, a.p);
    int64_t grid_fx = 0;
    // one CTA an SM with all its registers for up to a location an SM, else two
    const auto kern_fx = a.M <= ctx->num_sms ? alc_f64fx_kernel<PF_BMAX> : alc_f64fx_kernel<4>;
    const bool fixed = a.g < 1.0 && smem_fx <= lagp_smem_room(ctx, kern_fx);
    if (fixed) {
        cudaFuncSetAttribute(kern_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_fx);
        int occ = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern_fx, PF_THREADS, smem_fx);
        int per_sm = alc_ctas_per_sm(ctx, alc_shape_key(kern_fx == alc_f64fx_kernel<4> ? "alc_f64fx" : "alc_f64fxwide", 0,
                                                        a.nmax, a.p, a.mean != nullptr), 2);
        if (occ > 0 && per_sm > occ) per_sm = occ;
        grid_fx = std::max<int64_t>(1, std::min<int64_t>((int64_t)ctx->num_sms * per_sm, a.M));
    }
    const size_t per_fx = (size_t)a.Npmax * (((size_t)a.nmax + 1 + a.p) * 8 + 1) + 8;
    char *ws = static_cast<char *>(lagp_ws(
        ctx, WS_ALC_PANEL, std::max((size_t)grid * a.Npmax * ((size_t)a.nmax + 1) * 8, (size_t)grid_fx * per_fx) + 256));
    int *counter = static_cast<int *>(lagp_ws(ctx, WS_ALC_COUNTER, 256));
    if (!ws || !counter) return LAGP_ENOMEM;
    double *panel = reinterpret_cast<double *>(ws);
    double *kappa = panel + (size_t)grid * a.Npmax * a.nmax;
    LAGP_CUDA(ctx, cudaMemsetAsync(counter, 0, 11 * sizeof(int), st));
    if (fixed) {
        int2 *fp = reinterpret_cast<int2 *>(ws);
        double *fk = reinterpret_cast<double *>(fp + (size_t)grid_fx * a.nmax * a.Npmax);
        double *fc = fk + (size_t)grid_fx * a.Npmax;
        unsigned char *fs = reinterpret_cast<unsigned char *>(fc + (size_t)grid_fx * a.p * a.Npmax);
        kern_fx<<<(unsigned)grid_fx, PF_THREADS, smem_fx, st>>>(a, counter + 2, counter + 10, fp, fk, fc, fs);
        ctx->launches++;
        LAGP_CUDA(ctx, cudaGetLastError());
        a.retry_count = counter + 10;
    }
    if (cs > 1) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(F64_THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        LAGP_CUDA(ctx, cudaLaunchKernelEx(&cfg, alc_f64_kernel<true>, a, counter, panel, kappa));
    } else {
        alc_f64_kernel<false><<<(unsigned)grid, F64_THREADS, smem, st>>>(a, counter, panel, kappa);
    }
    ctx->launches++;
    LAGP_CUDA(ctx, cudaGetLastError());
    return LAGP_OK;
}
