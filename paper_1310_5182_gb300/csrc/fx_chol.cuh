// Cholesky factorisation of a local correlation matrix in 59-bit fixed point
// (fx59.cuh), with further rows and, optionally, its first and second
// derivatives in forward mode; one CTA of T threads (FXT unless stated), all in shared memory.
#pragma once
#include <cuda_runtime.h>

#include "device_util.cuh"
#include "fx59.cuh"
#include "gp_common.cuh"

namespace {

constexpr int FXT = 128, FXW = FXT / 32;
constexpr int FX_NMAX = 128;

// Matrices are stored by pairs of columns: entry (i, k) in the 16-byte word
// i + q (m - 1) - q^2, q = k / 2, half k mod 2 (rows i >= 2q of m; a pair's
// rows are adjacent, so that the lanes of a warp read without conflicts).
__host__ __device__ inline int fx_words(int n, int m) {
    const int Q = (n + 1) / 2;
    return Q * (m - 1) - (Q - 1) * (Q - 1) + 1;
}
__device__ __forceinline__ int fx_slot(int i, int k, int m) {
    const int q = k >> 1;
    return 2 * (i + q * (m - 1) - q * q) + (k & 1);
}

// What a step's threads need of its 2 x 2 diagonal block (negated where it
// is subtracted).
struct __align__(16) FxDiag {
    Fx y[2];             // 1 / l = y 2^t
    int t[2];
    Fx nl1[2], nl2[2];   // -l1, -l2
    Fx na, nb, ne;       // -L, -L1, -L2 of the lower left entry
    int pad[2];
};

// The dynamic shared memory: `words` 16-byte words a matrix from the start,
// then (at byte y_at) n responses, n reciprocals of the pivots (1 / l = ry
// 2^(rt - 59)) and their exponents.  Its parts are addressed from the symbol,
// so that the compiler sees shared memory also behind a call.
extern __shared__ __align__(16) unsigned char fx_smem[];

struct FxFactor {
    int words, n, m;  // matrix words, order, rows with the further ones
    int y_at, nmax;
};

__device__ __forceinline__ int4 *fx_mat(const FxFactor &F, int mat) {
    return reinterpret_cast<int4 *>(fx_smem) + mat * F.words;
}
__device__ __forceinline__ double *fx_y(const FxFactor &F) { return reinterpret_cast<double *>(fx_smem + F.y_at); }
__device__ __forceinline__ long long *fx_ry(const FxFactor &F) {
    return reinterpret_cast<long long *>(fx_smem + F.y_at) + F.nmax;
}
__device__ __forceinline__ int *fx_rt(const FxFactor &F) {
    return reinterpret_cast<int *>(fx_smem + F.y_at) + 4 * F.nmax;
}
__device__ __forceinline__ long long *fx_raw(const FxFactor &F, int mat, int slot) {
    return reinterpret_cast<long long *>(fx_mat(F, mat)) + slot;
}
__device__ __forceinline__ void fx_store(const FxFactor &F, int mat, int slot, Fx f) {
    reinterpret_cast<int2 *>(fx_mat(F, mat))[slot] = make_int2(f.h, f.l);
}
__device__ __forceinline__ long long fx_load(const FxFactor &F, int mat, int slot) {
    const int2 v = reinterpret_cast<const int2 *>(fx_mat(F, mat))[slot];
    return fx_join(Fx{v.x, v.y});
}

// v 2^t y, |v 2^t| < 2 (so that the result stays below 2.84)
__device__ __forceinline__ long long fx_scaled(long long v, int t, Fx y, unsigned &bad) {
    bad |= fx_beyond(v, 28 - t);
    return fx_mul(fx_split(v << t), y);
}

// Nonzero unless |x| < 2 (the high limb may be doubled).
__device__ __forceinline__ unsigned fx_beyond_h(Fx x) { return (unsigned)(x.h + (1 << 30)) >> 31; }

// One column of a row: L = S0 / l, L1 = (S1 - L l1) / l, L2 = (S2 - 2 L1 l1 - L l2) / l.
template <int NM>
struct FxRow {
    Fx v[NM];
};
template <int NM>
__device__ __forceinline__ void fx_column(const long long (&S)[NM], Fx y, int t, Fx nl1, Fx nl2, FxRow<NM> &r,
                                          unsigned &bad) {
    r.v[0] = fx_split(fx_scaled(S[0], t, y, bad));
    bad |= fx_beyond_h(r.v[0]);
    if constexpr (NM == 3) {
        const Fx a = r.v[0];
        const Fx p = r.v[1] =
            fx_split(fx_scaled(fx_hi(fx_sum(S[1], fx_mid(FX_HALF, a, nl1)), a, nl1), t, y, bad));
        bad |= fx_beyond_h(p);
        long long v = fx_sum(S[2], fx_mid(fx_mid(FX_HALF, a, nl2), p, fx_twice(nl1)));
        v = fx_hi(fx_hi(fx_hi(v, a, nl2), p, nl1), p, nl1);
        r.v[2] = fx_split(fx_scaled(v, t, y, bad));
        bad |= fx_beyond_h(r.v[2]);
    }
}

// The next column's S of a row, less the products with this column: (na, nb,
// ne) are -L, -L1, -L2 of the next column's own row in this column.
template <int NM>
__device__ __forceinline__ void fx_update(long long (&S)[NM], const FxRow<NM> &r, Fx na, Fx nb, Fx ne) {
    const Fx a = r.v[0];
    S[0] = fx_hi(fx_sum(S[0], fx_mid(FX_HALF, a, na)), a, na);
    if constexpr (NM == 3) {
        const Fx p = r.v[1], q = r.v[2];
        S[1] = fx_sum(S[1], fx_mid(fx_mid(FX_HALF, p, na), a, nb));
        S[1] = fx_hi(fx_hi(S[1], p, na), a, nb);
        S[2] = fx_sum(S[2], fx_mid(fx_mid(fx_mid(FX_HALF, q, na), a, ne), p, fx_twice(nb)));
        S[2] = fx_hi(fx_hi(fx_hi(fx_hi(S[2], q, na), a, ne), p, nb), p, nb);
    }
}

// hi += x_h y_h, mid += x_h y_l + x_l y_h
__device__ __forceinline__ void fx_acc(long long &hi, long long &mid, int xh, int xl, int yh, int yl) {
    hi = fx_mad(xh, yh, hi);
    mid = fx_mad(xl, yh, fx_mad(xh, yl, mid));
}

// The sums of columns c, c + 1 over k < c, subtracted from the rows below the
// diagonal block, by the warps 1 and up.  2^KL lanes share a row's sum.
template <int NM, int KL, int T>
__device__ __forceinline__ void fx_sums(const FxFactor &F, int c, int lane, int warp) {
    constexpr int RP = 32 >> KL, KS = 1 << KL;  // row pairs and shares of a warp
    const int m = F.m, n = F.n;
    const int rp = lane & (RP - 1), ks = lane / RP;
    for (int base = min(c + 2, n) + (warp - 1) * 2 * RP; base < m; base += (T / 32 - 1) * 2 * RP) {
        const int iA = base + rp, iB = iA + RP;
        const int ia = min(iA, m - 1), ib = min(iB, m - 1), j1 = min(c + 1, m - 1);
        long long hi[NM][2][2], mid[NM][2][2];
#pragma unroll
        for (int g = 0; g < NM; g++)
#pragma unroll
            for (int x = 0; x < 4; x++) hi[g][x >> 1][x & 1] = mid[g][x >> 1][x & 1] = 0;
        int off = ks * (m - 1) - ks * ks;
        int inc = KS * (m - 1) - 2 * ks * KS - KS * KS;
        for (int q = ks; q < (c >> 1); q += KS) {
            int4 r[NM][2], s[NM][2];
#pragma unroll
            for (int g = 0; g < NM; g++) {
                const int4 *P = fx_mat(F, g) + off;
                r[g][0] = P[ia];
                r[g][1] = P[ib];
                s[g][0] = P[c];
                s[g][1] = P[j1];
            }
            off += inc;
            inc -= 2 * KS * KS;
#pragma unroll
            for (int x = 0; x < 2; x++)
#pragma unroll
                for (int y = 0; y < 2; y++)
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        const int x0h = k ? r[0][x].z : r[0][x].x, x0l = k ? r[0][x].w : r[0][x].y;
                        const int y0h = k ? s[0][y].z : s[0][y].x, y0l = k ? s[0][y].w : s[0][y].y;
                        fx_acc(hi[0][x][y], mid[0][x][y], x0h, x0l, y0h, y0l);
                        if constexpr (NM == 3) {
                            const int x1h = k ? r[1][x].z : r[1][x].x, x1l = k ? r[1][x].w : r[1][x].y;
                            const int y1h = k ? s[1][y].z : s[1][y].x, y1l = k ? s[1][y].w : s[1][y].y;
                            const int x2h = k ? r[2][x].z : r[2][x].x, x2l = k ? r[2][x].w : r[2][x].y;
                            const int y2h = k ? s[2][y].z : s[2][y].x, y2l = k ? s[2][y].w : s[2][y].y;
                            fx_acc(hi[1][x][y], mid[1][x][y], x1h, x1l, y0h, y0l);
                            fx_acc(hi[1][x][y], mid[1][x][y], x0h, x0l, y1h, y1l);
                            fx_acc(hi[2][x][y], mid[2][x][y], x2h, x2l, y0h, y0l);
                            fx_acc(hi[2][x][y], mid[2][x][y], x0h, x0l, y2h, y2l);
                            fx_acc(hi[2][x][y], mid[2][x][y], x1h, x1l, 2 * y1h, 2 * y1l);
                        }
                    }
        }
        // the shares added up: first the columns, then the rows of the tile
        // are split between lanes (half of the values change hands), then
        // whole values
        long long v[NM];
#pragma unroll
        for (int g = 0; g < NM; g++) {
            long long w[2];
#pragma unroll
            for (int x = 0; x < 2; x++) {
                const long long v0 = (hi[g][x][0] << 1) + (mid[g][x][0] >> 29);
                const long long v1 = (hi[g][x][1] << 1) + (mid[g][x][1] >> 29);
                w[x] = (ks & 1 ? v1 : v0) + __shfl_xor_sync(LAGP_FULL_MASK, ks & 1 ? v0 : v1, RP);
            }
            v[g] = (ks & 2 ? w[1] : w[0]) + __shfl_xor_sync(LAGP_FULL_MASK, ks & 2 ? w[0] : w[1], 2 * RP);
#pragma unroll
            for (int o = 4 * RP; o < 32; o <<= 1) v[g] += __shfl_xor_sync(LAGP_FULL_MASK, v[g], o);
        }
        const int i = ks & 2 ? iB : iA, j = c + (ks & 1);
        if (ks < 4 && i < m && j < n) {
            const int slot = fx_slot(i, j, m);
#pragma unroll
            // (each share that is not empty was rounded down, by a half on average)
            for (int g = 0; g < NM; g++) *fx_raw(F, g, slot) -= v[g] + min(KS, c >> 1) / 2;
        }
    }
}

// The diagonal block of columns c, c + 1, one warp: the sums of its three
// entries (eight lanes an entry), then the block's factor, every lane the same.
// Returns nonzero when a value left the range.
template <int NM>
__device__ __forceinline__ unsigned fx_diagonal(const FxFactor &F, FxDiag *diag, int c, int lane) {
    const int n = F.n, m = F.m;
    const bool two = c + 1 < n;
    const int slot[3] = {fx_slot(c, c, m), fx_slot(c + 1, c, m), fx_slot(c + 1, c + 1, m)};
    long long S[3][NM];  // entries (c, c), (c + 1, c), (c + 1, c + 1)
#pragma unroll
    for (int g = 0; g < NM; g++)
#pragma unroll
        for (int e = 0; e < 3; e++) S[e][g] = e && !two ? 0 : *fx_raw(F, g, slot[e]);
    if (c > 0) {
        const int e = lane >> 3, ks = lane & 7;
        const int row = min(e == 0 ? c : c + 1, m - 1), col = min(e == 2 ? c + 1 : c, m - 1);
        long long hi[NM], mid[NM];
#pragma unroll
        for (int g = 0; g < NM; g++) hi[g] = mid[g] = 0;
        for (int q = ks; q < (c >> 1); q += 8) {
            const int off = q * (m - 1) - q * q;
            int4 r[NM], s[NM];
#pragma unroll
            for (int g = 0; g < NM; g++) {
                const int4 *P = fx_mat(F, g) + off;
                r[g] = P[row];
                s[g] = P[col];
            }
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int x0h = k ? r[0].z : r[0].x, x0l = k ? r[0].w : r[0].y;
                const int y0h = k ? s[0].z : s[0].x, y0l = k ? s[0].w : s[0].y;
                fx_acc(hi[0], mid[0], x0h, x0l, y0h, y0l);
                if constexpr (NM == 3) {
                    const int x1h = k ? r[1].z : r[1].x, x1l = k ? r[1].w : r[1].y;
                    const int y1h = k ? s[1].z : s[1].x, y1l = k ? s[1].w : s[1].y;
                    const int x2h = k ? r[2].z : r[2].x, x2l = k ? r[2].w : r[2].y;
                    const int y2h = k ? s[2].z : s[2].x, y2l = k ? s[2].w : s[2].y;
                    fx_acc(hi[1], mid[1], x1h, x1l, y0h, y0l);
                    fx_acc(hi[1], mid[1], x0h, x0l, y1h, y1l);
                    fx_acc(hi[2], mid[2], x2h, x2l, y0h, y0l);
                    fx_acc(hi[2], mid[2], x0h, x0l, y2h, y2l);
                    fx_acc(hi[2], mid[2], x1h, x1l, 2 * y1h, 2 * y1l);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < NM; g++) {
            long long v = (hi[g] << 1) + (mid[g] >> 29);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(LAGP_FULL_MASK, v, o);
            v += min(8, c >> 1) / 2;  // (shares rounded down)
#pragma unroll
            for (int x = 0; x < 3; x++) S[x][g] -= __shfl_sync(LAGP_FULL_MASK, v, 8 * x);
        }
    }
    unsigned bad = 0;
    FxDiag D;
    auto pivot = [&](int j, const long long (&s)[NM]) {
        long long s0 = s[0], l;
        // (a pivot below 2^-47, or not positive, is for FP64 to decide)
        const bool odd = s0 < (1ll << 12) || s0 >= (1ll << 60);
        bad |= odd;
        if (odd) s0 = FX_ONE;
        D.y[j] = fx_rsqrt(s0, &D.t[j], &l);
        const int at = slot[2 * j];
        if (lane == 0) {
            fx_store(F, 0, at, fx_split(l));
            fx_ry(F)[c + j] = fx_join(D.y[j]);
            fx_rt(F)[c + j] = D.t[j];
        }
        if constexpr (NM == 3) {
            const Fx l1 = fx_split(fx_scaled(s[1], D.t[j], D.y[j], bad) >> 1);  // (below 1.42)
            D.nl1[j] = fx_neg(l1);
            const long long v = fx_hi(fx_sum(s[2] >> 1, fx_mid(FX_HALF, l1, D.nl1[j])), l1, D.nl1[j]);
            const Fx l2 = fx_split(fx_scaled(v, D.t[j], D.y[j], bad));
            bad |= fx_beyond_h(l2);
            D.nl2[j] = fx_neg(l2);
            if (lane == 0) {
                fx_store(F, 1, at, l1);
                fx_store(F, 2, at, l2);
            }
        }
    };
    __syncwarp();  // every lane has read the entries that are written now
    pivot(0, S[0]);
    if (two) {
        FxRow<NM> r;
        fx_column<NM>(S[1], D.y[0], D.t[0], D.nl1[0], D.nl2[0], r, bad);
        D.na = fx_neg(r.v[0]);
        if constexpr (NM == 3) {
            D.nb = fx_neg(r.v[1]);
            D.ne = fx_neg(r.v[2]);
        }
        fx_update<NM>(S[2], r, D.na, D.nb, D.ne);
#pragma unroll
        for (int g = 0; g < NM; g++)
            if (lane == 0) fx_store(F, g, slot[1], r.v[g]);
        pivot(1, S[2]);
    }
    if (lane == 0) *diag = D;
    return bad;
}

// The factorisation (and its derivatives for NM = 3), in place; shared memory holds
// the raw values on entry and the limbs of L (L1, L2) after.  Two phases a
// pair of columns: one thread a row finishes the two columns, then one warp
// makes the next diagonal block (a serial chain) while
// the others form the sums of the next two columns.  Returns true when a value
// left the range, as soon as the pair of columns is done.  The verdict travels
// with the barriers and not through a word of shared memory, so that every
// thread has the same one and a caller may factorise again at once.
template <int NM, int T = FXT>
__device__ bool fx_factorise(const FxFactor &F, const Blk &b) {
    const int n = F.n, m = F.m;
    __shared__ FxDiag s_diag;
    unsigned bad = 0;  // this thread's share of the verdict
    __syncthreads();
    if (b.warp == 0) bad = fx_diagonal<NM>(F, &s_diag, 0, b.lane);
    __syncthreads();
    for (int c = 0; c < n; c += 2) {
        const bool two = c + 1 < n;
        const FxDiag D = s_diag;
        // (rows from warp 1 on: warp 0 has the serial chains)
        for (int i = c + (two ? 2 : 1) + (b.warp + T / 32 - 1) % (T / 32) * 32 + b.lane; i < m; i += T) {
            const int at = fx_slot(i, c, m);  // columns c, c + 1 of a row are adjacent
            long long S[NM], S2[NM];
#pragma unroll
            for (int g = 0; g < NM; g++) {
                const longlong2 v = *reinterpret_cast<const longlong2 *>(fx_raw(F, g, at));
                S[g] = v.x;
                S2[g] = v.y;
            }
            FxRow<NM> r, q;
            fx_column<NM>(S, D.y[0], D.t[0], D.nl1[0], D.nl2[0], r, bad);
            if (two) {
                fx_update<NM>(S2, r, D.na, D.nb, D.ne);
                fx_column<NM>(S2, D.y[1], D.t[1], D.nl1[1], D.nl2[1], q, bad);
            }
            // |x| < 1 in the further rows, whose norm nothing bounds
            if (i >= n)
#pragma unroll
                for (int g = 0; g < NM; g++) {
                    bad |= (unsigned)(r.v[g].h + (1 << 29)) >> 30;
                    if (two) bad |= (unsigned)(q.v[g].h + (1 << 29)) >> 30;
                }
#pragma unroll
            for (int g = 0; g < NM; g++) {
                if (two)
                    *reinterpret_cast<int4 *>(fx_raw(F, g, at)) = make_int4(r.v[g].h, r.v[g].l, q.v[g].h, q.v[g].l);
                else
                    fx_store(F, g, at, r.v[g]);
            }
        }
        if (__syncthreads_or(bad)) return true;
        if (c + 2 < n) {
            const int R = m - (c + 4);
            if (b.warp == 0) bad |= fx_diagonal<NM>(F, &s_diag, c + 2, b.lane);
            else if (R > 24) fx_sums<NM, 2, T>(F, c + 2, b.lane, b.warp);
            else if (R > 12) fx_sums<NM, 3, T>(F, c + 2, b.lane, b.warp);
            else fx_sums<NM, 4, T>(F, c + 2, b.lane, b.warp);
            __syncthreads();
        }
    }
    return false;
}

// Exponent e with max_i |v_i| < 2^e over the block's n values (INT_MAX when
// one is not finite or all are zero); red: T / 32 ints.
template <int T = FXT>
__device__ int fx_exponent(const double *v, int n, int *red, const Blk &b) {
    int top = 0;
    __syncthreads();
    for (int i = b.tid; i < n; i += T) top = max(top, (__double2hiint(v[i]) >> 20) & 0x7ff);
    top = __reduce_max_sync(LAGP_FULL_MASK, top);
    if (b.lane == 0) red[b.warp] = top;
    __syncthreads();
    for (int w = 0; w < T / 32; w++) top = max(top, red[w]);
    __syncthreads();
    // (subnormal responses and those near the largest double: FP64 kernels)
    return top < 64 || top > 1983 ? INT32_MAX : top - 1022;
}

// x 2^e by the exponent field (x = 0 or a result out of range: 0)
__device__ __forceinline__ double fx_shift(double x, int e) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
    return ex == 0 || ex + e <= 0 ? 0.0 : __hiloint2double(hi + (e << 20), __double2loint(x));
}

__device__ __forceinline__ void fx_tri(int e, int &i, int &k) {  // e-th entry of a lower triangle by rows
    int r = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
    if ((r + 1) * (r + 2) / 2 <= e) r++;
    if (r * (r + 1) / 2 > e) r--;
    i = r;
    k = e - r * (r + 1) / 2;
}

}  // namespace
