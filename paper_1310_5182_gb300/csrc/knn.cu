// a1: exact N'-nearest-neighbour candidate sets (Sec. 3.1 of the paper: the
// ALC search runs over the N' nearest neighbours of x; Fig. 1 step 2(a)).
//
// Design (GB300): distances are screened in FP32 (74 TFLOP/s) and only the
// few candidates near the N'-th distance are re-ranked in FP64 (1.2 TFLOP/s).
//   knn_bounds  per-coordinate minimum and maximum of the design and the
//               reference locations (the centre c and half-width B).
//   knn_prep    centred FP32 copy of the design, y = fl32(x - c), with the
//               FP32 squared norm |y|^2 as an extra column.
//   knn_sample  with the tensor-core collection: the sampled thresholds alone
//               (its passes A and B by a bound from part of the sample).
//   knn_screen  persistent; 16 queries per CTA, two per warp, sharing every
//               design tile in shared memory.  The main launch evaluates
//               |y_x|^2 + |y_q|^2 - 2 y_x . y_q (one add and p FMAs a pair);
//               the exact retry the direct sum of squared differences.
//               (A, B) 2-level histogram (FP32 distance bits [30:21], then
//               [20:11] inside the boundary bin) over a strided sample of the
//               design, giving a threshold tau0 expected to bound about 1.3 N'
//               rows (with stride 1, exactly the N'-th smallest distance);
//               (C) one pass over the whole design collecting every row below
//               tau0 widened by a rigorous FP32-vs-FP64 error margin (see
//               expansion_margin, screen_margin) and counting the rows below
//               tau0.  A query whose count is short of N', or whose buffer
//               overflowed, is redone by a second launch with stride 1 (the
//               exact method), where a block with at most four such queries
//               gives each a team of warps that share its sweep.
//   knn_rank    one CTA per query: buckets the collected rows by direct-form
//               FP32 distance and orders each bucket; exact FP64 distances
//               (separately rounded subtract/multiply/add in coordinate order,
//               on the original coordinates) inside runs of near ties; first N'
//               rows written out.
//   knn_sort    the same by a radix selection and a bitonic sort, for what
//               knn_rank leaves and after the exact retry.
// Large problems (ORD_MIN_PAIRS) first sort rows and locations by cell
// (knn_cells, knn_cell_starts, knn_cell_scatter), so that blocks of them have
// small bounding boxes (knn_boxes) and the tensor-core collection skips the
// block pairs that are too far apart; candidates are then positions in that
// order, mapped back to design rows by the sort.
// The collected set provably contains the exact FP64 top-N', so the result
// equals an FP64 sort of all N rows bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

#include "device_util.cuh"
#include "knn_common.cuh"
#include "lagp_internal.h"

namespace {

constexpr int QPW = 2;                // queries per warp
constexpr int SCREEN_THREADS = 256;
constexpr int QB = QPW * SCREEN_THREADS / 32;  // 16 queries per CTA
constexpr int HB = 1024;              // histogram bins per level (10 bits)
constexpr int L1_SHIFT = 21;          // level 1: FP32 distance bits [30:21]
constexpr int L2_SHIFT = 11;          // level 2: bits [20:11] inside the boundary bin
constexpr uint32_t L2_LOW = (1u << L2_SHIFT) - 1;
constexpr int SAMPLE_DEPTH = 16;       // sampled distances that a thread lists below the first sweep's bound
constexpr int SAMPLE_TILE_FLOATS = 5120;
constexpr int TILE_FLOATS = 4096;     // floats of one design tile (tile length x row stride)

// Floats per centred row: p coordinates and the squared norm, padded to an
// odd count so that lanes reading consecutive rows of a shared-memory tile
// hit distinct banks.
__host__ __device__ inline int row_stride(int p) { return (p + 1) | 1; }

// Design rows per tile: a multiple of 32 with tile length x row stride <=
// TILE_FLOATS, at most 512.
__host__ __device__ inline int tile_len(int ps) {
    int t = (TILE_FLOATS / ps) & ~31;
    return t > 512 ? 512 : (t < 32 ? 32 : t);
}


// Rows of a tile of the sampling sweep: a multiple of 64, at most 1,024.
__host__ __device__ inline int sample_tile(int ps) {
    int t = (SAMPLE_TILE_FLOATS / ps) & ~63;
    return t > 1024 ? 1024 : (t < 64 ? 64 : t);
}

// 16-byte asynchronous global-to-shared copy (bypassing L1), and its fences
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
constexpr int CAND_CAP = 8192;        // candidate capacity cap (sort in shared memory)
// kNN meta area: the tensor-core screen's failure word (offset 0), two block
// counters (64), the coordinate bounds (256 and 768, 64 keys each), the
// launch constants (KnnConst, 1280), then per-query candidate counts and
// retry flags
constexpr size_t META_HEAD = 2048;
constexpr size_t META_CONST = 1280;

// Constants of one kNN launch, written once by knn_prep: the centre c and
// half-width B of the coordinates, e2 = 2uB sqrt(p) and the power bounds
// g_half >= (1 + u)^((p+4)/2), (1 - u)^(-(p+4)/2) and g_full >= (1 + u)^(p+4).
struct KnnConst {
    double c[64];
    double B, e2, g_half, g_full;
};
constexpr int SORT_THREADS = 256;

// Per-coordinate bounds of the design and the reference locations:
// kmax[i] = key of max_i, kmin[i] = ~key of min_i (both maximised).  Eight
// coordinates per sweep: each thread keeps their bounds in registers over its
// rows, then warp and block reductions, one atomic per block and coordinate.
__global__ void knn_bounds(const void *__restrict__ X, int64_t N, const void *__restrict__ Xr,
                           int64_t M, int p, lagp_dtype dt, unsigned long long *kmax,
                           unsigned long long *kmin) {
    __shared__ unsigned long long smax[64], smin[64];
    for (int i = threadIdx.x; i < p; i += blockDim.x) smax[i] = smin[i] = 0ull;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int i0 = 0; i0 < p; i0 += 8) {
        double lo[8], hi[8];
#pragma unroll
        for (int c = 0; c < 8; c++) {
            lo[c] = CUDART_INF;
            hi[c] = -CUDART_INF;
        }
        for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < N + M; r += stride) {
            const bool des = r < N;
            const void *A = des ? X : Xr;
            const int64_t rr = des ? r : r - N;
#pragma unroll
            for (int c = 0; c < 8; c++) {
                if (i0 + c >= p) break;
                const double v = load_coord64(A, rr, p, i0 + c, dt);
                if (isfinite(v)) {  // a non-finite row only spoils its own distances
                    lo[c] = fmin(lo[c], v);
                    hi[c] = fmax(hi[c], v);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 8; c++) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo[c] = fmin(lo[c], __shfl_xor_sync(LAGP_FULL_MASK, lo[c], o));
                hi[c] = fmax(hi[c], __shfl_xor_sync(LAGP_FULL_MASK, hi[c], o));
            }
            if ((threadIdx.x & 31) == 0 && i0 + c < p && hi[c] >= lo[c]) {
                atomicMax(&smax[i0 + c], dkey(hi[c]));
                atomicMax(&smin[i0 + c], ~dkey(lo[c]));
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < p; i += blockDim.x) {
        if (smax[i]) atomicMax(&kmax[i], smax[i]);
        if (smin[i]) atomicMax(&kmin[i], smin[i]);
    }
}

// Centred FP32 copy of the design row at position r, (y_0 .. y_{p-1}, |y|^2, 0 padding),
// with y_i = fl32(x_i - c_i) and |y|^2 an FP32 fused multiply-add chain in
// coordinate order; rows past N are zero.
__device__ __forceinline__ void centred_row(const void *X, int64_t N, int64_t r, const int32_t *perm, int p,
                                            int ps, lagp_dtype dt, const double *c, float *out) {
    float n2 = 0.f;
    const int64_t row = r < N && perm ? perm[r] : r;
    for (int i = 0; i < p; i++) {
        const float y = r < N ? (float)(load_coord64(X, row, p, i, dt) - c[i]) : 0.f;
        out[i] = y;
        n2 = fmaf(y, y, n2);
    }
    for (int i = p; i < ps; i++) out[i] = i == p ? n2 : 0.f;
}

// Rigorous upper bounds of the powers of (1 + u) and 1 / (1 - u) that the
// margins need (n u < 1): (1 + u)^m <= (1 - u)^-m <= 1 / (1 - m u) for
// m <= n, without a call to pow (whose latency on the FP64 unit would
// serialise the threads that wait for the margin).
__device__ __forceinline__ double pow_bound(double u, double n) { return 1.0 / (1.0 - ceil(n) * u); }

// In the order of perm (null: as given).  Y: all rows (Npad of them), Ys: the
// nsamp positions 0, s, 2s, ... (null when s = 1, where the sample is the whole
// design; padded with zero rows to nsamp_pad), stepping through them by `spread`
// positions (prime to nsamp, near the golden section), so that its first rows
// are themselves an even sample, Yv: the
// coordinates of Y with a row stride of p rounded up to 4; kc: the launch's
// constants (block 0).
__global__ void knn_prep(const void *__restrict__ X, int64_t N, int p, lagp_dtype dt,
                         const unsigned long long *kmax, const unsigned long long *kmin,
                         const int32_t *__restrict__ perm, float *__restrict__ Y, int64_t Npad,
                         float *__restrict__ Ys, int64_t nsamp, int64_t nsamp_pad, int64_t sstride, int64_t spread,
                         KnnConst *kc,
                         float *__restrict__ Yv) {
    __shared__ double c[64];
    __shared__ double sB;
    if (threadIdx.x == 0) {
        centre_and_bound(kmax, kmin, p, c, sB);
        if (blockIdx.x == 0) {
            const double u = 0x1p-24 * (1.0 + 0x1p-27);
            for (int i = 0; i < p; i++) kc->c[i] = c[i];
            kc->B = sB;
            kc->e2 = 2.0 * u * sB * sqrt((double)p);
            kc->g_half = pow_bound(u, 0.5 * (p + 4));
            kc->g_full = pow_bound(u, (double)(p + 4));
        }
    }
    __syncthreads();
    const int ps = row_stride(p);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < Npad; r += stride) {
        centred_row(X, N, r, perm, p, ps, dt, c, Y + r * ps);
        // the same coordinates with a row stride of p rounded up to 4 (vector gathers in the sort)
        const int pv = (p + 3) & ~3;
        for (int i = 0; i < pv; i++) Yv[r * pv + i] = i < p ? Y[r * ps + i] : 0.f;
    }
    if (Ys)
        for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < nsamp_pad; r += stride)
            centred_row(X, N, r < nsamp ? r * spread % nsamp * sstride : N, perm, p, ps, dt, c, Ys + r * ps);
}

// ------------------------------------------------------------ spatial order
// The design rows and the locations sorted by the cell they lie in, so that
// 128 rows (or 64 locations) in a row have a small bounding box: a counting
// sort on a 16-bit cell number, the coordinates' leading bits (up to 16 cuts
// in halves, taken round the coordinates) read as a Gray code, so that
// neighbouring cells in the order differ in one cut.  The order within a cell
// is whatever the atomics make it: no result depends on it.
constexpr int ORD_BITS = 16, ORD_CELLS = 1 << ORD_BITS;
// From here on: the order costs four launches and 60 to 500 us, the collection
// of 2^30 pairs 0.55 ms (100,000 x 10,000 in 8 dimensions: 10.55 ms a call
// without, 10.80 with it; 500,000 x 201,600 in 3: 49.1 without, 19.7 with).
constexpr int64_t ORD_MIN_ROWS = 1 << 15, ORD_MIN_PAIRS = 1ll << 30;

__global__ void knn_cells(const void *__restrict__ X, int64_t N, const void *__restrict__ Xr, int64_t M, int p,
                          lagp_dtype dt, const unsigned long long *kmax, const unsigned long long *kmin,
                          uint16_t *__restrict__ cell, uint32_t *__restrict__ hist) {
    __shared__ double lo[ORD_BITS], inv[ORD_BITS];
    const int dims = min(p, ORD_BITS);
    if (threadIdx.x < dims) {
        const int i = threadIdx.x;
        const double a = kmax[i] ? dkey_inv(~kmin[i]) : 0.0, b = kmax[i] ? dkey_inv(kmax[i]) : 0.0;
        lo[i] = a;
        inv[i] = b > a ? 1.0 / (b - a) : 0.0;
    }
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < N + M; r += stride) {
        const bool des = r < N;
        uint32_t code = 0;
        for (int i = 0; i < dims; i++) {
            const int bits = (ORD_BITS - i + dims - 1) / dims;  // cuts of this coordinate
            const float t = (float)((load_coord64(des ? X : Xr, des ? r : r - N, p, i, dt) - lo[i]) * inv[i]);
            const uint32_t v = min((uint32_t)(fmaxf(t, 0.f) * (float)(1 << bits)), (1u << bits) - 1u);  // (NaN: 0)
            for (int b = 0; b < bits; b++)
                code |= ((v >> (bits - 1 - b)) & 1u) << (ORD_BITS - 1 - (b * dims + i));
        }
        code ^= code >> 1;  // Gray code to its rank
        code ^= code >> 2;
        code ^= code >> 4;
        code ^= code >> 8;
        cell[r] = (uint16_t)code;
        atomicAdd(hist + (des ? 0 : ORD_CELLS) + code, 1u);
    }
}

// Exclusive prefix sums of the two histograms (block 0: rows, 1: locations).
__global__ void __launch_bounds__(1024) knn_cell_starts(uint32_t *hist) {
    constexpr int PER = ORD_CELLS / 1024;
    __shared__ uint32_t wsum[32];
    uint32_t *h = hist + (size_t)blockIdx.x * ORD_CELLS + threadIdx.x * PER;
    uint32_t s = 0;
    for (int i = 0; i < PER; i += 4) {
        const uint4 v = *reinterpret_cast<const uint4 *>(h + i);
        s += v.x + v.y + v.z + v.w;
    }
    uint32_t incl = s;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(LAGP_FULL_MASK, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    uint32_t at = incl - s;
    for (int i = 0; i < w; i++) at += wsum[i];
    for (int i = 0; i < PER; i += 4) {
        uint4 v = *reinterpret_cast<uint4 *>(h + i);
        const uint4 n = v;
        v.x = at, v.y = v.x + n.x, v.z = v.y + n.y, v.w = v.z + n.z;
        at = v.w + n.w;
        *reinterpret_cast<uint4 *>(h + i) = v;
    }
}

__global__ void knn_cell_scatter(const uint16_t *__restrict__ cell, int64_t N, int64_t M,
                                 uint32_t *__restrict__ starts, int32_t *__restrict__ row,
                                 int32_t *__restrict__ query) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < N + M; r += stride) {
        const bool des = r < N;
        const uint32_t at = atomicAdd(starts + (des ? 0 : ORD_CELLS) + cell[r], 1u);
        (des ? row : query)[at] = (int32_t)(des ? r : r - N);
    }
}

// Bounding boxes of the blocks of 128 positions, from the ordered centred
// copy: one warp a block.
__global__ void knn_boxes(const float *__restrict__ Y, int64_t N, int p, int nmb, float *__restrict__ box) {
    const int lane = threadIdx.x & 31, ps = row_stride(p);
    for (int mb = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); mb < nmb; mb += gridDim.x * (blockDim.x >> 5))
        for (int i = 0; i < p; i++) {
            float lo = CUDART_INF_F, hi = -CUDART_INF_F;  // (fminf and fmaxf leave NaN out)
            for (int64_t r = (int64_t)mb * 128 + lane; r < min(N, (int64_t)mb * 128 + 128); r += 32) {
                lo = fminf(lo, Y[r * ps + i]);
                hi = fmaxf(hi, Y[r * ps + i]);
            }
            for (int o = 16; o > 0; o >>= 1) {
                lo = fminf(lo, __shfl_xor_sync(LAGP_FULL_MASK, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(LAGP_FULL_MASK, hi, o));
            }
            if (lane == 0) {
                box[(int64_t)i * nmb + mb] = lo;
                box[(int64_t)(p + i) * nmb + mb] = hi;
            }
        }
}

// Widened thresholds for the collection pass.  With u = 2^-24 (widened by
// 2^-27 for the FP64 centring), centred coordinates rounded to FP32 with
// absolute error <= u B, the FP32 screen value s of a row relates to its
// exact distance r as follows.
//
// screen_margin (direct form: FP32 differences, squares and sums, each
// rounded once):
//     (1-u)^((p+4)/2) (r - 2uB sqrt(p)) <= sqrt(s) <= (1+u)^((p+4)/2) (r + 2uB sqrt(p)).
// Every row with s <= tau then has r <= r_hi = sqrt(tau) (1-u)^(-(p+4)/2) + 2uB sqrt(p),
// so the N'-th exact distance is <= r_hi, and every row of the exact top-N' has
// sqrt(s) <= (r_hi + 2uB sqrt(p)) (1+u)^((p+4)/2).
//
// expansion_margin (s = max(0, |y_x|^2 + |y_q|^2 - 2 y_x . y_q), every norm
// and the dot product FMA chains of at most 2p + 4 roundings in all):
//     |s - |y_q - y_x|^2| <= E = gamma_{2p+4} 4 p B^2,   gamma_k = k u / (1 - k u),
// and |y_q - y_x| lies within 2uB sqrt(p) of r.  A row with s <= tau then has
// r <= r_hi = sqrt(tau + E) + 2uB sqrt(p), and every row of the exact top-N'
// has s <= (r_hi + 2uB sqrt(p))^2 + E.
//
// The final factors cover the rounding of the FP64 reference distances (the
// order is that of the FP64 sums, within a relative 1e-15 of r^2) and of
// this computation.
// g >= (1 - u)^-(p+4)/2 and (1 + u)^(p+4)/2, e2 = 2uB sqrt(p)
__device__ __forceinline__ double screen_margin_c(float tau, double g, double e2) {
    const double r_hi = sqrt((double)tau) * g * (1.0 + 1e-13) + e2;
    const double r_col = (r_hi + e2) * g;
    return r_col * r_col * (1.0 + 1e-12);
}

__device__ double screen_margin(float tau, int p, double B) {
    const double u = 0x1p-24 * (1.0 + 0x1p-27);
    return screen_margin_c(tau, pow_bound(u, 0.5 * (p + 4)), 2.0 * u * B * sqrt((double)p));
}

__device__ double expansion_margin(float tau, int p, double B) {
    const double u = 0x1p-24 * (1.0 + 0x1p-27);
    const double Bt = B * (1.0 + u);
    const double e2 = 2.0 * u * B * sqrt((double)p);
    const double k = 2.0 * p + 4.0;
    const double E = (k * u / (1.0 - k * u)) * 4.0 * p * Bt * Bt;
    const double r_hi = sqrt((double)tau + E) * (1.0 + 1e-13) + e2;
    const double r_col = r_hi + e2;
    return (r_col * r_col + E) * (1.0 + 1e-12);
}

// Smallest bin b of the warp's histogram h with cum(h[0..b]) >= target,
// and the count strictly before it.  Requires sum(h) >= target >= 1.
__device__ void find_bin(const uint32_t *h, uint32_t target, int lane, uint32_t &bin,
                         uint32_t &before) {
    constexpr int PER = HB / 32;
    uint32_t s = 0;
    for (int b = 0; b < PER; b++) s += h[lane * PER + b];
    uint32_t incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t v = __shfl_up_sync(LAGP_FULL_MASK, incl, o);
        if (lane >= o) incl += v;
    }
    unsigned ball = __ballot_sync(LAGP_FULL_MASK, incl >= target);
    int L = ball ? __ffs(ball) - 1 : 31;
    uint32_t base = __shfl_sync(LAGP_FULL_MASK, incl - s, L);
    // resolve inside lane L's PER bins, 32 at a time
    bin = (uint32_t)(L * PER + PER - 1);
    before = base;
    for (int half = 0; half < PER; half += 32) {
        uint32_t v = h[L * PER + half + lane];
        uint32_t c = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(LAGP_FULL_MASK, c, o);
            if (lane >= o) c += t;
        }
        unsigned bb = __ballot_sync(LAGP_FULL_MASK, base + c >= target);
        if (bb) {
            int l2 = __ffs(bb) - 1;
            bin = (uint32_t)(L * PER + half + l2);
            before = base + __shfl_sync(LAGP_FULL_MASK, c - v, l2);
            return;
        }
        base += __shfl_sync(LAGP_FULL_MASK, c, 31);
    }
}

// Rank, in a sample of every stride-th row (nsamp of them), of the threshold
// for k rows: 1.3 k / stride + 16, exactly k when the sample is the design.
__host__ __device__ inline int sample_rank(int k, int64_t stride, int64_t nsamp) {
    if (stride == 1) return k;
    const int64_t rt = (13 * (int64_t)k + 10 * stride - 1) / (10 * stride) + 16;
    return (int)(rt < nsamp ? rt : nsamp);
}

// One design tile against a warp's QPW queries, rows r0, r0 + rstep, ... of
// the tile.  PASS 0: level-1 histogram; PASS 1: level-2 histogram inside the
// boundary bin; PASS 2: collection.
// Tile row pt holds (y_0 .. y_{p-1}, |y|^2) of a centred design row, with
// row stride PS.  EXP: s = max(0, |y_x|^2 + |y_q|^2 - 2 y_x . y_q) with
// qr = -2 y_q and qn = |y_q|^2 (negative values, from rounding, clamped to 0);
// otherwise s = sum (y_x - y_q)^2 with qr = y_q.
template <int P, int PASS, bool EXP>
__device__ __forceinline__ void screen_tile(const float *t, int ps_rt, int cnt, int r0, int rstep, int p,
                                            const float (&qr)[QPW][P > 0 ? P : 1],
                                            const float (&qn)[QPW], const float *qsw,
                                            const bool (&ok)[QPW], uint32_t *histw,
                                            const uint32_t (&b1)[QPW], const float (&tau0)[QPW],
                                            const float (&tau2f)[QPW], int32_t *cntw, int32_t *cnt0w,
                                            int32_t *__restrict__ cand, const int64_t (&q)[QPW],
                                            int32_t Cmax, int64_t base) {
    const int np = P > 0 ? P : p;
    const int PS = P > 0 ? ((P + 1) | 1) : ps_rt;
    for (int pt = r0; pt < cnt; pt += rstep) {
        const float *row = t + pt * PS;
        float sd[QPW];
        if constexpr (EXP) {
            const float xn = row[np];
#pragma unroll
            for (int h = 0; h < QPW; h++) sd[h] = xn + qn[h];
        } else {
#pragma unroll
            for (int h = 0; h < QPW; h++) sd[h] = 0.f;
        }
        if constexpr (P > 0) {
#pragma unroll
            for (int i = 0; i < P; i++) {
                const float x = row[i];
#pragma unroll
                for (int h = 0; h < QPW; h++) {
                    if constexpr (EXP) {
                        sd[h] = fmaf(x, qr[h][i], sd[h]);
                    } else {
                        const float df = x - qr[h][i];
                        sd[h] = fmaf(df, df, sd[h]);
                    }
                }
            }
        } else {
            for (int i = 0; i < p; i++) {
                const float x = row[i];
#pragma unroll
                for (int h = 0; h < QPW; h++) {
                    const float qv = qsw[h * PS + i];
                    if constexpr (EXP) {
                        sd[h] = fmaf(x, -2.f * qv, sd[h]);
                    } else {
                        const float df = x - qv;
                        sd[h] = fmaf(df, df, sd[h]);
                    }
                }
            }
        }
#pragma unroll
        for (int h = 0; h < QPW; h++) {
            if constexpr (EXP) sd[h] = sd[h] < 0.f ? 0.f : sd[h];  // keeps NaN
            if constexpr (PASS == 0) {
                if (ok[h]) atomicAdd(&histw[h * HB + ((__float_as_uint(sd[h]) >> L1_SHIFT) & (HB - 1))], 1u);
            } else if constexpr (PASS == 1) {
                const uint32_t bits = __float_as_uint(sd[h]);
                if (ok[h] && ((bits >> L1_SHIFT) & (HB - 1)) == b1[h])
                    atomicAdd(&histw[h * HB + ((bits >> L2_SHIFT) & (HB - 1))], 1u);
            } else {
                if (ok[h] && sd[h] <= tau2f[h]) {
                    if (sd[h] <= tau0[h]) atomicAdd(&cnt0w[h], 1);
                    const int pos = atomicAdd(&cntw[h], 1);
                    if (pos < Cmax) cand[q[h] * Cmax + pos] = (int32_t)(base + pt);
                }
            }
        }
    }
}

// Screen of one block of QB queries (two per warp) against the design.
//   Passes A, B: 2-level histogram of the FP32 distances to the sampled rows
//   r = 0, s, 2s, ...; the rtarget-th smallest sampled distance gives tau0
//   (upper edge of its level-2 bin).  With s = 1 (small designs, and the exact
//   retry) rtarget = N' and tau0 bounds the N'-th smallest FP32 distance.
//   Pass C: every row whose FP32 distance is <= the widened threshold is
//   collected, and the rows <= tau0 are counted; when that count reaches N'
//   the collected set provably holds the exact FP64 top N' (see the margin
//   functions).  Otherwise (a sample that underestimated the threshold) or
//   when the buffer overflows, the query is flagged for the exact retry.
template <int P, bool EXP>
__global__ void __launch_bounds__(SCREEN_THREADS, 2)
knn_screen(const float *__restrict__ Y32, const float *__restrict__ Ys, int64_t N, int p,
           const void *__restrict__ Xref,
           lagp_dtype dt, int64_t M, const int32_t *__restrict__ Np, int32_t Npmax,
           const unsigned long long *__restrict__ kmax, const unsigned long long *__restrict__ kmin,
           int32_t *__restrict__ cand, int32_t Cmax, int32_t *__restrict__ cand_count,
           int32_t *__restrict__ status, int64_t stride, int32_t *__restrict__ retry, int retry_pass,
           int *__restrict__ counter) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int pp = row_stride(p);              // floats per centred row (coordinates, norm, pad)
    const int TT = tile_len(pp);               // rows per tile
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw);   // QB x HB
    float *tiles = reinterpret_cast<float *>(hist + QB * HB);  // 2 x TT x pp, 16-byte aligned
    float *qs = tiles + 2 * (size_t)TT * pp;                     // (QB + 1) x pp: centred queries
    __shared__ int32_t s_count[QB], s_count0[QB], s_flag[QB], s_rt[QB];
    __shared__ int64_t s_blk;
    __shared__ double s_c[64], s_B;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) centre_and_bound(kmax, kmin, p, s_c, s_B);
    // a spare zero slot past the QB queries (read, never used, by the second
    // query slot of a warp that screens the last query of a block together
    // with other warps)
    for (int i = threadIdx.x; i < pp; i += SCREEN_THREADS) qs[QB * pp + i] = 0.f;
    __syncthreads();
    const double B = s_B;
    const int64_t nsamp = (N + stride - 1) / stride;

    for (;;) {
        if (threadIdx.x == 0) s_blk = atomicAdd(counter, 1);
        __syncthreads();
        const int64_t blk = s_blk;
        __syncthreads();
        if (blk * QB >= M) break;

        int64_t q[QPW];
        int k[QPW], rtarget[QPW];
        bool ok[QPW], active[QPW];
        bool mine_any = false;
#pragma unroll
        for (int h = 0; h < QPW; h++) {
            const int ql = w * QPW + h;
            q[h] = blk * QB + ql;
            active[h] = q[h] < M;
            k[h] = active[h] ? (Np ? Np[q[h]] : Npmax) : 0;
            ok[h] = active[h] && k[h] >= 1 && k[h] <= Npmax;
            if (retry_pass) ok[h] = ok[h] && retry[q[h]] != 0;  // exact retry: flagged queries only
            mine_any |= ok[h];
            rtarget[h] = stride == 1 ? k[h]
                                     : sample_rank(k[h], stride, nsamp);
            if (lane == 0) {
                float n2 = 0.f;
                for (int i = 0; i < p; i++) {
                    const float y = active[h] ? (float)(load_coord64(Xref, q[h], p, i, dt) - s_c[i]) : 0.f;
                    qs[ql * pp + i] = y;
                    n2 = fmaf(y, y, n2);
                }
                qs[ql * pp + p] = n2;
                for (int i = p + 1; i < pp; i++) qs[ql * pp + i] = 0.f;
            }
            for (int b = lane; b < HB; b += 32) hist[ql * HB + b] = 0;
            if (lane == 0) {
                s_count[ql] = s_count0[ql] = 0;
                s_flag[ql] = ok[h] ? 1 : 0;
                s_rt[ql] = rtarget[h];
            }
        }
        // a block without a query to screen skips the passes (not the results)
        const bool any_ok = __syncthreads_or(mine_any);
        // The queries a warp screens: its own QPW (slots sbase, sbase + 1) or,
        // in the exact retry of a block with at most four flagged queries,
        // one flagged query shared by a team of W = 8 / nf warps (nf rounded
        // up to a power of two; a team of four idle when nf = 3).  A team
        // splits every tile's rows (warp `sub` of the team takes the 32-row
        // groups sub, sub + W, ...) and adds into the query's one histogram
        // and counters, so that one query's sweep over all N rows runs on
        // the whole CTA instead of one warp.  The results are the same
        // either way: the counts do not depend on which warp adds them, and
        // the sort orders the collected rows.
        int nf = 0;
        if (retry_pass)
            for (int c = 0; c < QB; c++) nf += s_flag[c];
        const bool coop = nf >= 1 && nf <= 4;
        int sbase = w * QPW, r0 = lane, rstep = 32;
        bool leader = true;  // the warp that clears the team's histogram
        bool sok[QPW];
        int srt[QPW];
        int64_t sq[QPW];
#pragma unroll
        for (int h = 0; h < QPW; h++) {
            sok[h] = ok[h];
            srt[h] = rtarget[h];
            sq[h] = q[h];
        }
        if (coop) {
            const int W = nf == 1 ? 8 : (nf == 2 ? 4 : 2);
            const int team = w / W, sub = w - team * W;
            int slot = -1;  // the team-th flagged slot
            for (int c = 0, f = 0; c < QB; c++)
                if (s_flag[c]) {
                    if (f == team) slot = c;
                    f++;
                }
            sbase = slot >= 0 ? slot : 0;
#pragma unroll
            for (int h = 0; h < QPW; h++) {
                sok[h] = h == 0 && slot >= 0;
                srt[h] = s_rt[sbase];
                sq[h] = blk * QB + sbase;
            }
            r0 = lane + 32 * sub;
            rstep = 32 * W;
            leader = sub == 0;
        }
        float qr[QPW][P > 0 ? P : 1] = {};
        float qn[QPW] = {};
#pragma unroll
        for (int h = 0; h < QPW; h++) {
            qn[h] = qs[(sbase + h) * pp + p];
            if constexpr (P > 0) {
#pragma unroll
                for (int i = 0; i < P; i++) {
                    const float y = qs[(sbase + h) * pp + i];
                    qr[h][i] = EXP ? -2.f * y : y;
                }
            }
        }

        uint32_t b1[QPW] = {}, before[QPW] = {};
        // thresholds as floats: for a float distance s, s <= t (t real) holds
        // exactly when s <= t rounded down to a float, so the hot loop compares
        // in FP32 (an FP64 compare per point would occupy the slow FP64 unit)
        float tau0[QPW] = {}, tau2f[QPW] = {};
        const int npass = any_ok ? 3 : 0;
        for (int pass = 0; pass < npass; pass++) {
            // passes A, B: the sampled rows (contiguous in Ys); C: all rows
            const float *src = pass < 2 ? Ys : Y32;
            const int64_t nrows = pass < 2 ? nsamp : N;
            const int64_t ntiles = (nrows + TT - 1) / TT;
            // tile `tile` into buffer `buf`: its rows rounded up to a multiple of
            // 4 (zero rows past the end of the padded copies), 16 bytes a copy
            auto issue = [&](int64_t tile, int buf) {
                const int64_t base = tile * TT;
                const int cnt4 = (int)round_up(min((int64_t)TT, nrows - base), 4);
                const int nchunk = cnt4 * pp / 4;
                const float *g = src + base * pp;
                float *t = tiles + (size_t)buf * TT * pp;
                for (int e = threadIdx.x; e < nchunk; e += SCREEN_THREADS) cp_async16(t + 4 * e, g + 4 * e);
                cp_async_commit();
            };
            issue(0, 0);
            cp_async_wait_all();
            __syncthreads();
            for (int64_t tile = 0; tile < ntiles; tile++) {
                const int buf = (int)(tile & 1);
                if (tile + 1 < ntiles) issue(tile + 1, buf ^ 1);  // in flight during the screen
                const int64_t base = tile * TT;
                const int cnt = (int)min((int64_t)TT, nrows - base);
                const float *t = tiles + (size_t)buf * TT * pp;
                const float *qsw = qs + sbase * pp;
                uint32_t *histw = hist + sbase * HB;
                if (pass == 0)
                    screen_tile<P, 0, EXP>(t, pp, cnt, r0, rstep, p, qr, qn, qsw, sok, histw, b1, tau0, tau2f,
                                           s_count + sbase, s_count0 + sbase, cand, sq, Cmax, base);
                else if (pass == 1)
                    screen_tile<P, 1, EXP>(t, pp, cnt, r0, rstep, p, qr, qn, qsw, sok, histw, b1, tau0, tau2f,
                                           s_count + sbase, s_count0 + sbase, cand, sq, Cmax, base);
                else
                    screen_tile<P, 2, EXP>(t, pp, cnt, r0, rstep, p, qr, qn, qsw, sok, histw, b1, tau0, tau2f,
                                           s_count + sbase, s_count0 + sbase, cand, sq, Cmax, base);
                // the next tile has landed and every warp is done with this one
                cp_async_wait_all();
                __syncthreads();
            }
#pragma unroll
            for (int h = 0; h < QPW; h++) {
                if (!sok[h]) continue;
                const uint32_t *hh = hist + (sbase + h) * HB;
                if (pass == 0) {
                    find_bin(hh, (uint32_t)srt[h], lane, b1[h], before[h]);
                } else if (pass == 1) {
                    uint32_t b2, before2;
                    find_bin(hh, (uint32_t)srt[h] - before[h], lane, b2, before2);
                    tau0[h] = __uint_as_float((b1[h] << L1_SHIFT) | (b2 << L2_SHIFT) | L2_LOW);
                    tau2f[h] = __double2float_rd(EXP ? expansion_margin(tau0[h], p, B)
                                                     : screen_margin(tau0[h], p, B));
                }
            }
            if (pass == 0) {
                // every warp of a team has read the level-1 histogram before
                // its leader clears it for level 2
                __syncthreads();
                if (leader)
#pragma unroll
                    for (int h = 0; h < QPW; h++)
                        if (sok[h])
                            for (int b = lane; b < HB; b += 32) hist[(sbase + h) * HB + b] = 0;
            }
            __syncthreads();
        }
#pragma unroll
        for (int h = 0; h < QPW; h++) {
            if (!active[h] || lane != 0) continue;
            const int ql = w * QPW + h;
            const int c = s_count[ql], c0 = s_count0[ql];
            const bool kvalid = k[h] >= 1 && k[h] <= Npmax;
            if (!retry_pass) {
                const bool done = ok[h] && c0 >= k[h] && c <= Cmax;
                retry[q[h]] = (ok[h] && !done) ? 1 : 0;
                cand_count[q[h]] = done ? c : 0;
                if (status) status[q[h]] = kvalid ? LAGP_OK : LAGP_EINVAL;
            } else if (ok[h]) {
                // exact retry: fewer rows than N' under the threshold only happens
                // with non-finite distances (NaN or overflowing coordinates)
                cand_count[q[h]] = (c0 >= k[h] && c <= Cmax) ? c : 0;
                if (status) status[q[h]] = c0 < k[h] ? LAGP_EINVAL : (c > Cmax ? LAGP_ENOMEM : LAGP_OK);
            }
        }
        __syncthreads();
    }
}

// Sampled thresholds of the tensor-core collection: per query the rank-th
// smallest distance (norm expansion) to the sampled rows, rounded up to the
// end of its 2^-12-wide bin (bits [30:11]); NaN for a query that is not
// screened.  Eight warps share nq = 8 QW / W queries: groups of W warps, QW
// queries a warp, the group's warps splitting every tile's rows.
//   First sweep (nsub > 0): the first nsub rows of Ys (an even subset: the
//   order spreads them), histogram of bits [30:19].  The bin's end U at the
//   wanted rank bounds the threshold of all rows from above, whatever the
//   subset.
//   Second sweep: all rows; the values up to U (a few hundred) are listed, and the wanted rank selected from the list.
//   Without a first sweep (a rank too large for the list: small designs), or
//   when a list overflows, two histogram sweeps over all rows instead, bits
//   [30:21], then [20:11] inside the boundary bin.
// What bounds it: the second sweep's instructions, about half of the issue
// slots, the rest latency and the barrier a tile (four smaller tiles in flight:
// 15% slower; lists shared through an atomic or a ballot: 10 to 50% slower).
// Two histogram sweeps with two queries a warp (an atomic a pair, most of a
// warp's lanes in the same few bins) took 4.1 -> 2.2 ms (62,500 sampled rows,
// p = 8, 25,000 queries), 4.9 -> 3.1 ms (12,196 rows, p = 3, 201,600 queries) and
// 93 -> 25 us (10,000 rows, p = 2, 100 queries: sixteen a CTA met 7 SMs).
template <int P, int QW, int W>
__global__ void __launch_bounds__(SCREEN_THREADS, 2)
knn_sample(const float *__restrict__ Ys, int64_t nsamp, int64_t nsub, int p, const void *__restrict__ Xref,
           lagp_dtype dt, int64_t M, const int32_t *__restrict__ Np, int32_t Npmax, int64_t stride,
           const unsigned long long *__restrict__ kmax, const unsigned long long *__restrict__ kmin,
           int *__restrict__ counter, float *__restrict__ tau_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int pp = row_stride(p), TT = sample_tile(pp), np = P > 0 ? P : p, PS = P > 0 ? ((P + 1) | 1) : pp;
    constexpr int nq = 8 * QW / W;
    constexpr int COLS = 32 * W, SLOT = SAMPLE_DEPTH * COLS;  // a query's list: SAMPLE_DEPTH values a thread of its group
    static_assert(SLOT >= HB, "a query's histogram fits its list's place");
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw);   // nq x SLOT: histograms (HB words), or lists
    float *tiles = reinterpret_cast<float *>(hist + nq * SLOT);  // 2 x TT x pp, 16-byte aligned
    float *qs = tiles + 2 * (size_t)TT * pp;                   // nq x pp: centred queries
    __shared__ int32_t s_rt[nq];
    __shared__ float s_U[nq], s_tau[nq];
    __shared__ uint8_t s_n[nq * COLS];  // list lengths
    __shared__ int64_t s_blk;
    __shared__ double s_c[64], s_B;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q0 = w / W * QW, sub = w % W;  // the warp's first query slot, its share of the rows
    if (threadIdx.x == 0) centre_and_bound(kmax, kmin, p, s_c, s_B);
    __syncthreads();
    // first sweep's bins: 16 an octave, 64 octaves down from above the largest distance
    const int cbase = (int)(__float_as_uint((float)(4.0 * p * s_B * s_B * 1.01)) >> 19) - (HB - 1);

    for (;;) {
        if (threadIdx.x == 0) s_blk = atomicAdd(counter, 1);
        __syncthreads();
        const int64_t blk = s_blk;
        if (blk * nq >= M) break;
        for (int ql = threadIdx.x; ql < nq; ql += SCREEN_THREADS) {
            const int64_t q = blk * nq + ql;
            const int k = q < M ? (Np ? Np[q] : Npmax) : 0;
            s_rt[ql] = k >= 1 && k <= Npmax ? sample_rank(k, stride, nsamp) : 0;  // 0: not screened
            s_tau[ql] = CUDART_NAN_F;
            float n2 = 0.f;
            for (int i = 0; i < p; i++) {
                const float y = q < M ? (float)(load_coord64(Xref, q, p, i, dt) - s_c[i]) : 0.f;
                qs[ql * pp + i] = y;
                n2 = fmaf(y, y, n2);
            }
            qs[ql * pp + p] = n2;
        }
        auto clear = [&]() {
            for (int b = threadIdx.x; b < nq * HB; b += SCREEN_THREADS) hist[b / HB * SLOT + b % HB] = 0;
            __syncthreads();
        };
        clear();
        int rt[QW];
        float qr[QW][P > 0 ? P : 1] = {}, qn[QW];
        bool any = false;
#pragma unroll
        for (int h = 0; h < QW; h++) {
            rt[h] = s_rt[q0 + h];
            any |= rt[h] > 0;
            qn[h] = qs[(q0 + h) * pp + p];
            if constexpr (P > 0) {
#pragma unroll
                for (int i = 0; i < P; i++) qr[h][i] = -2.f * qs[(q0 + h) * pp + i];
            }
        }
        // body(h, value, whether the lane holds a row) for the first nrows rows
        auto clamp = [](float v) { return v < 0.f ? 0.f : v; };  // keeps NaN
        auto sweep = [&](int64_t nrows, auto body) {
            const int64_t ntiles = (nrows + TT - 1) / TT;
            // a tile's rows, rounded up to a multiple of 4 (within the padded copy), 16 bytes a copy
            auto issue = [&](int64_t tile) {
                const int64_t base = tile * TT;
                const int nchunk = (int)round_up(min((int64_t)TT, nrows - base), 4) * pp / 4;
                const float *g = Ys + base * pp;
                float *t = tiles + (size_t)(tile & 1) * TT * pp;
                for (int e = threadIdx.x; e < nchunk; e += SCREEN_THREADS) cp_async16(t + 4 * e, g + 4 * e);
                cp_async_commit();
            };
            issue(0);
            cp_async_wait_all();
            __syncthreads();
            for (int64_t tile = 0; tile < ntiles; tile++) {
                if (tile + 1 < ntiles) issue(tile + 1);  // in flight during the sweep
                const int cnt = (int)min((int64_t)TT, nrows - tile * TT);
                const float *t = tiles + (size_t)(tile & 1) * TT * pp;
                for (int pt = 32 * sub; pt < cnt; pt += 32 * W) {
                    // (lanes past the last row read the buffer, and are masked)
                    const bool live = pt + lane < cnt;
                    const float *row = t + (pt + lane) * PS;
                    float sd[QW];
                    const float xn = row[np];
#pragma unroll
                    for (int h = 0; h < QW; h++) sd[h] = xn + qn[h];
                    if constexpr (P > 0) {
#pragma unroll
                        for (int i = 0; i < P; i++) {
                            const float x = row[i];
#pragma unroll
                            for (int h = 0; h < QW; h++) sd[h] = fmaf(x, qr[h][i], sd[h]);
                        }
                    } else {
                        for (int i = 0; i < p; i++) {
                            const float x = row[i];
#pragma unroll
                            for (int h = 0; h < QW; h++) sd[h] = fmaf(x, -2.f * qs[(q0 + h) * pp + i], sd[h]);
                        }
                    }
#pragma unroll
                    for (int h = 0; h < QW; h++) body(h, sd[h], live);
                }
                // the next tile has landed and every warp is done with this one
                cp_async_wait_all();
                __syncthreads();
            }
        };
        bool two = true;  // two histogram sweeps over all rows
        if (!__syncthreads_or(any)) {
            two = false;
        } else if (nsub > 0) {
            sweep(nsub, [&](int h, float v, bool live) {
                const int b = min(max((int)(__float_as_uint(clamp(v)) >> 19) - cbase, 0), HB - 1);
                if (rt[h] > 0 && live) atomicAdd(&hist[(q0 + h) * SLOT + b], 1u);
            });
            float U[QW];
#pragma unroll
            for (int h = 0; h < QW; h++) {
                U[h] = -1.f;
                if (rt[h] == 0) continue;
                uint32_t b, before;
                find_bin(hist + (q0 + h) * SLOT, (uint32_t)rt[h], lane, b, before);
                U[h] = b == HB - 1 ? CUDART_INF_F : __uint_as_float((uint32_t)((int)b + cbase) << 19 | 0x7FFFFu);
                if (lane == 0) s_U[q0 + h] = U[h];  // (the warps of a group write the same value)
            }
            __syncthreads();
            // each thread a column of its own in the lists: no atomic, no branch
            int n[QW] = {};
            uint32_t *col = hist + q0 * SLOT + sub * 32 + lane;
            sweep(nsamp, [&](int h, float v, bool live) {
                const bool hit = live && v <= U[h];
                if (hit && n[h] < SAMPLE_DEPTH) col[h * SLOT + n[h] * COLS] = __float_as_uint(v);
                n[h] += hit;
            });
#pragma unroll
            for (int h = 0; h < QW; h++) s_n[(q0 + h) * COLS + sub * 32 + lane] = (uint8_t)min(n[h], 255);
            __syncthreads();
            // A list holds the wanted rank unless a column overflowed, or the
            // subset's bound is no number.  Selection by a warp a query: histogram of the
            // distance below U in units of 2^17 (64ths of an octave), then of 2^11.
            bool bad = false;
            uint32_t *h2 = reinterpret_cast<uint32_t *>(tiles) + w * 256;
            for (int ql = w; ql < nq; ql += 8) {
                const int target = s_rt[ql];
                if (target == 0) continue;
                int len[W], n = 0, longest = 0;  // of the lane's columns
#pragma unroll
                for (int v = 0; v < W; v++) {
                    len[v] = s_n[ql * COLS + v * 32 + lane];
                    n += len[v];
                    longest = max(longest, len[v]);
                }
                n = (int)__reduce_add_sync(LAGP_FULL_MASK, (unsigned)n);
                if (__any_sync(LAGP_FULL_MASK, longest > SAMPLE_DEPTH) || n < target || !(s_U[ql] < CUDART_INF_F)) {
                    bad = true;
                    continue;
                }
                const uint32_t Ub = __float_as_uint(s_U[ql]), *list = hist + ql * SLOT + lane;
                // (descending distance below U: the smallest values lie in the last bins)
                uint32_t d17 = 0;
                int rank = n - target + 1;  // of the wanted value by distance below U, the smallest first
                for (int level = 0; level < 2; level++) {
                    const int nb = level == 0 ? 256 : 64;
                    for (int b = lane; b < nb; b += 32) h2[b] = 0;
                    __syncwarp();
#pragma unroll
                    for (int v = 0; v < W; v++)
                        for (int e = 0; e < len[v]; e++) {
                            const float f = __uint_as_float(list[e * COLS + v * 32]);
                            const uint32_t d = Ub - __float_as_uint(clamp(f));
                            if (level == 0) atomicAdd(&h2[min(d >> 17, 255u)], 1u);
                            else if (min(d >> 17, 255u) == d17) atomicAdd(&h2[d >> 11 & 63u], 1u);
                        }
                    __syncwarp();
                    // the bin that holds the rank, 8 (2) bins a lane
                    const int per = nb / 32;
                    int sum = 0;
                    for (int b = 0; b < per; b++) sum += (int)h2[lane * per + b];
                    int incl = sum;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int t = __shfl_up_sync(LAGP_FULL_MASK, incl, o);
                        if (lane >= o) incl += t;
                    }
                    const int L = __ffs(__ballot_sync(LAGP_FULL_MASK, incl >= rank)) - 1;
                    int c = __shfl_sync(LAGP_FULL_MASK, incl - sum, L);
                    int b = L * per;
                    for (; b < L * per + per - 1 && c + (int)h2[b] < rank; b++) c += (int)h2[b];
                    rank -= c;
                    __syncwarp();
                    if (level == 0) {
                        d17 = (uint32_t)b;
                        if (d17 == 255u) {  // four octaves below the bound or more
                            bad = true;
                            break;
                        }
                    } else if (lane == 0) {
                        s_tau[ql] = __uint_as_float(((Ub >> L2_SHIFT) - (d17 << 6 | (uint32_t)b)) << L2_SHIFT | L2_LOW);
                    }
                }
            }
            two = __syncthreads_or(bad);
            if (two) clear();
        }
        if (two) {
            uint32_t b1[QW] = {}, before[QW] = {};
            for (int pass = 0; pass < 2; pass++) {
                sweep(nsamp, [&](int h, float v, bool live) {
                    const uint32_t bits = __float_as_uint(clamp(v));
                    uint32_t *hh = hist + (q0 + h) * SLOT;
                    if (rt[h] == 0 || !live) return;
                    if (pass == 0) atomicAdd(&hh[bits >> L1_SHIFT & (HB - 1)], 1u);
                    else if ((bits >> L1_SHIFT & (HB - 1)) == b1[h]) atomicAdd(&hh[bits >> L2_SHIFT & (HB - 1)], 1u);
                });
#pragma unroll
                for (int h = 0; h < QW; h++) {
                    if (rt[h] == 0) continue;
                    uint32_t b, bf;
                    find_bin(hist + (q0 + h) * SLOT, (uint32_t)rt[h] - before[h], lane, b, bf);
                    if (pass == 0) b1[h] = b, before[h] = bf;
                    else if (lane == 0) s_tau[q0 + h] = __uint_as_float(b1[h] << L1_SHIFT | b << L2_SHIFT | L2_LOW);
                }
                __syncthreads();
                if (pass == 0) clear();
            }
        }
        __syncthreads();
        for (int ql = threadIdx.x; ql < nq && blk * nq + ql < M; ql += SCREEN_THREADS) tau_out[blk * nq + ql] = s_tau[ql];
        __syncthreads();
    }
}

// Block-wide exclusive prefix sum of one int per thread (NT threads); returns
// the thread's offset, *total the sum.
template <int NT>
__device__ int block_excl_scan(int v, int *wsum, int *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(LAGP_FULL_MASK, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    int off = 0, tot = 0;
    for (int i = 0; i < NT / 32; i++) {
        off += i < w ? wsum[i] : 0;
        tot += wsum[i];
    }
    __syncthreads();
    *total = tot;
    return off + incl - v;
}

// Bound Delta on |s - r^2| for the direct-form FP32 value s of a row whose
// FP32 value is at most tau (its exact distance r is then at most
// Rm = sqrt(tau) (1-u)^(-(p+4)/2) + e2, e2 = 2uB sqrt(p)):
//     |s - r^2| <= ((1+u)^(p+4) - 1) (Rm + e2)^2 + 2 Rm e2 + e2^2,
// widened by 1e-6 relative, plus 2e-15 Rm^2 for the rounding of the FP64
// sums that define the order.  Two rows whose FP32 values differ by more
// than 2 Delta are in the same order by their FP64 distances, strictly.
// g_half >= (1 - u)^-(p+4)/2, g_full >= (1 + u)^(p+4), e2 = 2uB sqrt(p)
__device__ __forceinline__ double tie_bound(float tau, double g_half, double g_full, double e2) {
    const double Rm = sqrt((double)tau) * g_half * (1.0 + 1e-13) + e2;
    const double d0 = (g_full - 1.0) * (Rm + e2) * (Rm + e2) + 2.0 * Rm * e2 + e2 * e2;
    return d0 * (1.0 + 1e-6) + 2e-15 * Rm * Rm;
}

__device__ __forceinline__ bool pair_less(double da, uint32_t ra, double db, uint32_t rb) {
    return da < db || (da == db && ra < rb);
}

// One CTA per query.
//  (1) direct-form FP32 value s = sum (y_x - y_q)^2 of every collected row;
//  (2) radix selection of the N'-th smallest, v_k;
//  (3) survivors: rows with s <= screen_margin(v_k), which hold the exact
//      FP64 top N' (at least N' collected rows have s <= v_k, so the N'-th
//      exact distance is bounded as in the screen);
//  (4) bitonic sort of the survivors on (s, row) as one 64-bit key;
//  (5) runs of neighbours closer than 2 tie_bound get their exact FP64
//      distances (separately rounded subtract/multiply/add in coordinate
//      order, on the original coordinates) and are re-ordered on (d2, row)
//      within the run; outside the runs the FP32 order is the FP64 order.
//      A run longer than 32 sends the query to a full FP64 sort instead;
//  (6) the first N' rows.
// Ascending bitonic sort of sk[0, S) (S <= 1,024; the keys past S act as
// +infinity) by 256 threads, four keys a thread in registers: element e =
// 128 warp + 4 lane + r.  Compare-exchanges at distance 1, 2 stay in the
// thread, 4..64 go through warp shuffles, 128..512 through shared memory
// (two alternating buffers of 1,024 keys, sk and alt: one barrier a step).
// The sorted keys end in sk[0, 1024).
__device__ void sort1024_registers(unsigned long long *sk, int S, unsigned long long *alt) {
    static_assert(SORT_THREADS == 256, "four keys a thread for 1,024");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int base = warp * 128 + lane * 4;
    unsigned long long x[4];
#pragma unroll
    for (int r = 0; r < 4; r++) x[r] = base + r < S ? sk[base + r] : ~0ull;
    __syncthreads();  // every key is read before sk serves as an exchange buffer
    int buf = 0;
    for (int size = 2; size <= 1024; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 128) {
                unsigned long long *b = buf ? alt : sk;
                buf ^= 1;
#pragma unroll
                for (int r = 0; r < 4; r++) b[base + r] = x[r];
                __syncthreads();
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    const int e = base + r;
                    const unsigned long long y = b[e ^ stride];
                    // take y when it belongs here: smaller for the low end of an
                    // ascending pair (or the high end of a descending one)
                    if ((y < x[r]) == (((e & stride) == 0) == ((e & size) == 0))) x[r] = y;
                }
            } else if (stride >= 4) {
                const int lm = stride >> 2;
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    const int e = base + r;
                    const unsigned long long y = __shfl_xor_sync(LAGP_FULL_MASK, x[r], lm);
                    if ((y < x[r]) == (((lane & lm) == 0) == ((e & size) == 0))) x[r] = y;
                }
            } else {
                // within the thread: pairs (0, 2), (1, 3) at distance 2, (0, 1),
                // (2, 3) at distance 1 (constant register indices)
                auto cx = [&](unsigned long long &a, unsigned long long &c, int e) {
                    const bool asc = (e & size) == 0;
                    if (asc ? c < a : a < c) {
                        const unsigned long long t = a;
                        a = c;
                        c = t;
                    }
                };
                if (stride == 2) {
                    cx(x[0], x[2], base);
                    cx(x[1], x[3], base + 1);
                } else {
                    cx(x[0], x[1], base);
                    cx(x[2], x[3], base + 2);
                }
            }
        }
    }
    __syncthreads();  // the last exchange buffer is read before sk is written
#pragma unroll
    for (int r = 0; r < 4; r++) sk[base + r] = x[r];
    __syncthreads();
}

// The general sort, for the queries that knn_rank leaves (bigf) and, after the
// exact retry, the flagged ones: any number of survivors, any run of ties, in
// shared memory.  One CTA a query, the grid striding over the queries.
__device__ void knn_sort_query(const void *__restrict__ X, const float *__restrict__ Yv,
                               const int32_t *__restrict__ perm, int p, lagp_dtype dt,
                               const void *__restrict__ Xref, int64_t q, const int32_t *__restrict__ Np,
                               int32_t Npmax, const int32_t *__restrict__ cand,
                               const int32_t *__restrict__ cand_count, int32_t Cmax, int32_t *__restrict__ idx,
                               const KnnConst *__restrict__ kc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int C = cand_count[q];
    const int k = Np ? Np[q] : Npmax;
    int32_t *out = idx + q * Npmax;
    if (C < k || C > Cmax || k < 1 || k > Npmax) {  // invalid or overflowed: empty row
        for (int t = threadIdx.x; t < Npmax; t += SORT_THREADS) out[t] = -1;
        return;
    }
    int Cp = 1;
    while (Cp < Cmax) Cp <<= 1;
    // region 1 (R1 doubles): FP32 keys and positions for steps 1-3, then FP64
    // keys; region 2 (R1 words of 64 bits): the survivors' (s, row) keys
    const int R1 = Cp;
    uint32_t *key32 = reinterpret_cast<uint32_t *>(smem_raw);           // Cmax
    int32_t *rowA = reinterpret_cast<int32_t *>(key32 + R1);            // Cmax
    double *dk = reinterpret_cast<double *>(smem_raw);                  // R1
    unsigned long long *sk = reinterpret_cast<unsigned long long *>(smem_raw + (size_t)R1 * 8);  // R1
    __shared__ double xq[64];
    __shared__ float yq[64];
    __shared__ float s_d2f;
    __shared__ uint32_t hist[256];
    __shared__ int wsum[SORT_THREADS / 32];
    __shared__ uint32_t s_prefix;
    __shared__ int s_kk, s_big;
    __shared__ float s_tauf;
    __shared__ uint32_t tied[CAND_CAP / 32];
    if (threadIdx.x < p) {
        xq[threadIdx.x] = load_coord64(Xref, q, p, threadIdx.x, dt);
        yq[threadIdx.x] = (float)(xq[threadIdx.x] - kc->c[threadIdx.x]);
    }
    if (threadIdx.x == 0) {
        s_prefix = 0u;
        s_kk = k;
        s_big = 0;
    }
    __syncthreads();
    // (1) direct-form FP32 values (non-negative floats order like their
    // bits); four rows a thread in flight
    const int pv = (p + 3) & ~3;  // row stride of Yv
#pragma unroll 4
    for (int e = threadIdx.x; e < C; e += SORT_THREADS) {
        const int32_t r = cand[q * Cmax + e];
        const float4 *yr = reinterpret_cast<const float4 *>(Yv + (int64_t)r * pv);
        float sv = 0.f;
        for (int i4 = 0; i4 < pv; i4 += 4) {
            const float4 v = yr[i4 >> 2];
            const float t[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (i4 + j < p) {  // coordinate order, as the direct form defines
                    const float df = t[j] - yq[i4 + j];
                    sv = fmaf(df, df, sv);
                }
        }
        key32[e] = __float_as_uint(sv);  // NaN keeps the largest keys
        rowA[e] = r;
    }
    // (2) radix selection of the k-th smallest key, 8 bits at a time
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int b = threadIdx.x; b < 256; b += SORT_THREADS) hist[b] = 0u;
        __syncthreads();
        const uint32_t prefix = s_prefix;
        const uint32_t hmask = shift == 24 ? 0u : (0xffffffffu << (shift + 8));
        // one atomic per distinct bin of a warp (most keys share their top bits)
        const int lane = threadIdx.x & 31;
        for (int e0 = threadIdx.x - lane; e0 < C; e0 += SORT_THREADS) {
            uint32_t bin = 0xFFFFFFFFu;
            if (e0 + lane < C) {
                const uint32_t kv = key32[e0 + lane];
                if ((kv & hmask) == prefix) bin = (kv >> shift) & 255u;
            }
            const unsigned peers = __match_any_sync(LAGP_FULL_MASK, bin);
            if (bin != 0xFFFFFFFFu && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            const int kk = s_kk;
            uint32_t sub = 0;
            for (int b = 0; b < 8; b++) sub += hist[lane * 8 + b];
            uint32_t incl = sub;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(LAGP_FULL_MASK, incl, o);
                if (lane >= o) incl += t;
            }
            const unsigned ball = __ballot_sync(LAGP_FULL_MASK, incl >= (uint32_t)kk);
            const int L = __ffs(ball) - 1;  // the k-th key is in lane L's bins
            if (lane == L) {
                uint32_t cum = incl - sub;
                int b = 0;
                for (; b < 7; b++) {
                    if (cum + hist[lane * 8 + b] >= (uint32_t)kk) break;
                    cum += hist[lane * 8 + b];
                }
                s_prefix = prefix | ((uint32_t)(lane * 8 + b) << shift);
                s_kk = kk - (int)cum;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        // the margins with the launch's constants
        const double g = kc->g_half, e2 = kc->e2;
        const float vk = __uint_as_float(s_prefix);
        const float tauf = __double2float_rd(screen_margin_c(vk, g, e2));
        s_tauf = tauf;
        s_d2f = __double2float_ru(2.0 * tie_bound(tauf, g, kc->g_full, e2));
    }
    __syncthreads();
    const float tauf = s_tauf;
    // (3) survivors, in candidate order, as (s, row) keys
    int mine = 0;
    for (int e = threadIdx.x; e < C; e += SORT_THREADS) mine += __uint_as_float(key32[e]) <= tauf;
    int S = 0;
    int pos = block_excl_scan<SORT_THREADS>(mine, wsum, &S);  // S is block-uniform
    int Sp = 1;
    while (Sp < S) Sp <<= 1;
    for (int e = threadIdx.x; e < C; e += SORT_THREADS)
        if (__uint_as_float(key32[e]) <= tauf)
            sk[pos++] = ((unsigned long long)key32[e] << 32) | (uint32_t)(perm ? perm[rowA[e]] : rowA[e]);
    for (int e = S + threadIdx.x; e < Sp; e += SORT_THREADS) sk[e] = ~0ull;
    __syncthreads();
    // (4) bitonic sort on (s, row): up to 1,024 keys in registers (four a
    // thread), else in shared memory
    if (Sp <= 4 * SORT_THREADS) {
        sort1024_registers(sk, S, reinterpret_cast<unsigned long long *>(smem_raw));
    } else {
        for (int size = 2; size <= Sp; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int e = threadIdx.x; e < (Sp >> 1); e += SORT_THREADS) {
                    const int lo = 2 * e - (e & (stride - 1)), hi = lo + stride;
                    const bool up = ((lo & size) == 0);
                    const unsigned long long ka = sk[lo], kb = sk[hi];
                    if (up ? kb < ka : ka < kb) {
                        sk[lo] = kb;
                        sk[hi] = ka;
                    }
                }
                __syncthreads();
            }
        }
    }
    // (5) runs of near-equal FP32 values: FP64 keys, ordered within the run
    const float d2f = s_d2f;  // twice the tie bound, rounded up
    auto gap_ok = [&](int i) {  // rows i and i + 1 are in a certain FP64 order
        // the FP32 difference rounded down never exceeds the true one
        const float a = __uint_as_float((uint32_t)(sk[i] >> 32));
        const float b = __uint_as_float((uint32_t)(sk[i + 1] >> 32));
        return __fsub_rd(b, a) > d2f;
    };
    auto fp64_key = [&](int i) {
        const int32_t r = (int32_t)(uint32_t)sk[i];
        double sd = 0.0;
        for (int t = 0; t < p; t++) {
            const double diff = __dsub_rn(xq[t], load_coord64(X, r, p, t, dt));
            sd = __dadd_rn(sd, __dmul_rn(diff, diff));
        }
        return sd;
    };
    // tie flags first (bit i: rows i and i + 1 need their FP64 order), so that
    // no run is re-ordered while another thread still reads its FP32 keys
    for (int w = threadIdx.x; w < (Sp + 31) / 32; w += SORT_THREADS) tied[w] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i + 1 < S; i += SORT_THREADS)
        if (!gap_ok(i)) atomicOr(&tied[i >> 5], 1u << (i & 31));
    __syncthreads();
    auto is_tied = [&](int i) { return (tied[i >> 5] >> (i & 31)) & 1u; };
    for (int i = threadIdx.x; i < S; i += SORT_THREADS) {
        if (!is_tied(i) || (i > 0 && is_tied(i - 1))) continue;  // not the start of a run
        int end = i + 1;  // the run is [i, end]
        while (is_tied(end) && end - i < 32) end++;
        if (end - i >= 32) {
            s_big = 1;
            continue;
        }
        for (int t = i; t <= end; t++) dk[t] = fp64_key(t);
        for (int t = i + 1; t <= end; t++) {  // insertion sort on (d2, row)
            const double dv = dk[t];
            const unsigned long long kv = sk[t];
            int u = t - 1;
            while (u >= i && pair_less(dv, (uint32_t)kv, dk[u], (uint32_t)sk[u])) {
                dk[u + 1] = dk[u];
                sk[u + 1] = sk[u];
                u--;
            }
            dk[u + 1] = dv;
            sk[u + 1] = kv;
        }
    }
    __syncthreads();
    if (s_big) {
        // a long run: exact FP64 keys for every survivor and a full sort on (d2, row)
        for (int i = threadIdx.x; i < Sp; i += SORT_THREADS) dk[i] = i < S ? fp64_key(i) : CUDART_INF;
        __syncthreads();
        for (int size = 2; size <= Sp; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int e = threadIdx.x; e < (Sp >> 1); e += SORT_THREADS) {
                    const int lo = 2 * e - (e & (stride - 1)), hi = lo + stride;
                    const bool up = ((lo & size) == 0);
                    const double da = dk[lo], db = dk[hi];
                    const unsigned long long ka = sk[lo], kb = sk[hi];
                    const bool swap = up ? pair_less(db, (uint32_t)kb, da, (uint32_t)ka)
                                         : pair_less(da, (uint32_t)ka, db, (uint32_t)kb);
                    if (swap) {
                        dk[lo] = db;
                        dk[hi] = da;
                        sk[lo] = kb;
                        sk[hi] = ka;
                    }
                }
                __syncthreads();
            }
        }
    }
    // (6)
    for (int t = threadIdx.x; t < Npmax; t += SORT_THREADS) out[t] = t < k ? (int32_t)(uint32_t)sk[t] : -1;
}

__global__ void __launch_bounds__(SORT_THREADS)
knn_sort(const void *__restrict__ X, const float *__restrict__ Yv, const int32_t *__restrict__ perm, int p,
         lagp_dtype dt, const void *__restrict__ Xref, int64_t M, const int32_t *__restrict__ Np, int32_t Npmax,
         const int32_t *__restrict__ cand, const int32_t *__restrict__ cand_count, int32_t Cmax,
         int32_t *__restrict__ idx, const KnnConst *__restrict__ kc, const int32_t *__restrict__ retry,
         const int32_t *__restrict__ bigf) {
    for (int64_t q = blockIdx.x; q < M; q += gridDim.x) {
        if (!(retry && retry[q] != 0) && bigf[q] == 0) continue;
        knn_sort_query(X, Yv, perm, p, dt, Xref, q, Np, Npmax, cand, cand_count, Cmax, idx, kc);
        __syncthreads();  // shared memory is free for the next query
    }
}

// Rank of the collected rows without a comparison sort, one CTA a query: the
// rows' direct-form FP32 values (kept in registers, IT a thread) go into `nb`
// buckets of equal width between the smallest and the largest (a monotone
// map, so that the buckets are in order), about one row a bucket; a prefix sum
// of the counts places the rows of the buckets up to the one after the N'-th
// row's, and each bucket is ordered on (s, row) by one thread.  Then the
// margins, the collection check and the runs of near ties as in the steps
// above (3, 5, 6).  Linear in the number of rows, eight barriers, against the
// bitonic sort's (log^2) with a radix selection before it: N' = 1500 of 2,600
// rows, 201,600 queries, 32.8 -> 8.7 ms; N' = 2000 of 3,600, 25,000 queries,
// 14.7 -> 3.9 ms.  With the FP64 distances of all tied rows computed side by side
// (a run a thread kept the FP64 unit busy for 41% of the time): 7.3 and 2.4 ms.
// Bound: instruction issue and the latency of the gathers between barriers
// (128 or 512 threads a query in place of 256: 30% slower).  Left to knn_sort (bigf): distances that are not
// finite, a bucket of more than RANK_BUCKET rows, runs longer than 32 (many
// equal distances), survivors past the placed buckets.  knn_sort does not
// check the collection: a query is left to it only when the N'-th value, or the
// largest of its bucket, lies within the radius collected in full; otherwise,
// and with distances that are not finite, it goes to the exact retry.
constexpr int RANK_BUCKET = 24;

// Buckets for up to `cap` placed rows (cap FP64 keys reuse their space).
__host__ __device__ inline int rank_buckets(int cap) { return (2 * cap + 1023) / 1024 * 1024; }

template <int IT, int NT>
__global__ void __launch_bounds__(NT)
knn_rank(const void *__restrict__ X, const float *__restrict__ Yv, const int32_t *__restrict__ perm, int p,
         lagp_dtype dt, const void *__restrict__ Xref, const int32_t *__restrict__ Np, int32_t Npmax,
         const int32_t *__restrict__ cand, const int32_t *__restrict__ cand_count, int32_t Cmax, int cap,
         int32_t *__restrict__ idx, const KnnConst *__restrict__ kc, const float *__restrict__ rcol,
         int32_t *__restrict__ retry, int32_t *__restrict__ bigf) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t q = blockIdx.x;
    if (rcol && retry[q] != 0) return;  // (overflowed or not screened: the exact retry)
    const int C = cand_count[q], k = Np ? Np[q] : Npmax, tid = threadIdx.x, lane = tid & 31;
    int32_t *out = idx + q * Npmax;
    if (C < k || C > Cmax || k < 1 || k > Npmax) {  // invalid or overflowed: empty row
        for (int t = tid; t < Npmax; t += NT) out[t] = -1;
        return;
    }
    const int nb = rank_buckets(cap);
    uint32_t *start = reinterpret_cast<uint32_t *>(smem_raw);                           // nb: counts, then starts
    double *dk = reinterpret_cast<double *>(smem_raw);                                  // cap, after the buckets
    unsigned long long *sk = reinterpret_cast<unsigned long long *>(smem_raw + (size_t)nb * 4);  // cap (s, row) keys
    uint32_t *tied = reinterpret_cast<uint32_t *>(sk + cap);                            // cap / 32 + 1
    uint16_t *list = reinterpret_cast<uint16_t *>(tied + cap / 32 + 1);                 // cap: rows in runs of ties
    __shared__ double xq[64];
    __shared__ float yq[64];
    __shared__ int wsum[NT / 32];
    __shared__ uint32_t s_lo, s_hi, s_vk;
    __shared__ int s_kb, s_left, s_fail, s_S, s_ties;
    __shared__ float s_tauf, s_d2f;
    if (tid < p) {
        xq[tid] = load_coord64(Xref, q, p, tid, dt);
        yq[tid] = (float)(xq[tid] - kc->c[tid]);
    }
    if (tid == 0) s_lo = 0xFFFFFFFFu, s_hi = s_vk = 0u, s_left = s_ties = 0;
    for (int b = tid; b < nb; b += NT) start[b] = 0u;
    __syncthreads();
    // direct-form FP32 values (non-negative floats order like their bits)
    uint32_t key[IT];
    int32_t pos[IT];
    const int pv = (p + 3) & ~3;
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
    for (int i = 0; i < IT; i++) {
        const int e = tid + i * NT;
        pos[i] = e < C ? cand[q * Cmax + e] : -1;
    }
#pragma unroll
    for (int i = 0; i < IT; i++) {
        if (pos[i] < 0) continue;
        const float4 *yr = reinterpret_cast<const float4 *>(Yv + (int64_t)pos[i] * pv);
        float sv = 0.f;
        for (int i4 = 0; i4 < pv; i4 += 4) {
            const float4 v = yr[i4 >> 2];
            const float t[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (i4 + j < p) {  // coordinate order, as the direct form defines
                    const float df = t[j] - yq[i4 + j];
                    sv = fmaf(df, df, sv);
                }
        }
        key[i] = __float_as_uint(sv);
        lo = min(lo, key[i]);
        hi = max(hi, key[i]);
    }
    lo = __reduce_min_sync(LAGP_FULL_MASK, lo);
    hi = __reduce_max_sync(LAGP_FULL_MASK, hi);
    if (lane == 0) {
        atomicMin(&s_lo, lo);
        atomicMax(&s_hi, hi);
    }
    __syncthreads();
    const float base = __uint_as_float(s_lo), scale = (float)nb / (__uint_as_float(s_hi) - base);
    // at least the exact distance of a row whose direct-form value is v
    auto reach = [&](uint32_t v) { return sqrt((double)__uint_as_float(v)) * kc->g_half * (1.0 + 1e-13) + kc->e2; };
    if (s_hi >= 0x7f800000u) {  // infinite or NaN
        if (tid == 0) (rcol ? retry : bigf)[q] = 1;
        if (rcol)
            for (int t = tid; t < Npmax; t += NT) out[t] = -1;
        return;
    }
    // (equal values: 0 * infinity, bucket 0)
    auto bucket = [&](uint32_t b) { return min(nb - 1, (int)((__uint_as_float(b) - base) * scale)); };
    uint16_t rank[IT];
#pragma unroll
    for (int i = 0; i < IT; i++)
        if (pos[i] >= 0) rank[i] = (uint16_t)atomicAdd(&start[bucket(key[i])], 1u);
    __syncthreads();
    // starts of the buckets (a warp takes consecutive rows of 32); the N'-th
    // row's bucket
    {
        const int rows = nb / NT;  // rows of 32 buckets a warp
        uint32_t *mine = start + (tid >> 5) * rows * 32 + lane;
        int sum = 0, most = 0;
        for (int j = 0; j < rows; j++) {
            const int n = mine[32 * j];
            sum += n;
            most = max(most, n);
        }
        if (most > RANK_BUCKET) s_left = 1;
        int total;
        const int before = block_excl_scan<NT>(sum, wsum, &total);
        int at = __shfl_sync(LAGP_FULL_MASK, before, 0);  // rows before this warp's buckets
        for (int j = 0; j < rows; j++) {
            const int n = mine[32 * j];
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(LAGP_FULL_MASK, incl, o);
                if (lane >= o) incl += t;
            }
            const int from = at + incl - n;
            mine[32 * j] = from;
            if (from < k && from + n >= k) s_kb = ((tid >> 5) * rows + j) * 32 + lane;
            at += __shfl_sync(LAGP_FULL_MASK, incl, 31);
        }
    }
    __syncthreads();
    const int last = min(s_kb + 1, nb - 1);  // the buckets placed: 0 .. last
    const int cut = last + 1 < nb ? (int)start[last + 1] : C;
    if (s_left || cut > cap) {
        // the N'-th value is at most the largest of its bucket
        uint32_t top = 0u;
#pragma unroll
        for (int i = 0; i < IT; i++)
            if (pos[i] >= 0 && bucket(key[i]) == s_kb) top = max(top, key[i]);
        top = __reduce_max_sync(LAGP_FULL_MASK, top);
        if (lane == 0) atomicMax(&s_vk, top);
        __syncthreads();
        const bool fail = rcol && !(reach(s_vk) <= (double)rcol[q]);
        if (tid == 0) (fail ? retry : bigf)[q] = 1;
        if (fail)
            for (int t = tid; t < Npmax; t += NT) out[t] = -1;
        return;
    }
#pragma unroll
    for (int i = 0; i < IT; i++)
        if (pos[i] >= 0) {
            const int b = bucket(key[i]);
            if (b <= last)
                sk[start[b] + rank[i]] = ((unsigned long long)key[i] << 32) | (uint32_t)(perm ? perm[pos[i]] : pos[i]);
        }
    __syncthreads();
    for (int b = tid; b <= last; b += NT) {
        const int i0 = start[b], i1 = b + 1 < nb ? (int)start[b + 1] : C;
        for (int t = i0 + 1; t < i1; t++) {  // insertion sort on (s, row)
            const unsigned long long kv = sk[t];
            int u = t - 1;
            while (u >= i0 && kv < sk[u]) {
                sk[u + 1] = sk[u];
                u--;
            }
            sk[u + 1] = kv;
        }
    }
    __syncthreads();
    if (tid == 0) {
        // the margins with the launch's constants
        const double g = kc->g_half, e2 = kc->e2;
        const uint32_t vkb = (uint32_t)(sk[k - 1] >> 32);
        const float vk = __uint_as_float(vkb);
        const float tauf = __double2float_rd(screen_margin_c(vk, g, e2));
        s_tauf = tauf;
        s_d2f = __double2float_ru(2.0 * tie_bound(tauf, g, kc->g_full, e2));
        // rows collected on the tensor cores: the N'-th of them must lie
        // within the radius collected in full, else the query goes to the
        // exact retry
        s_fail = rcol ? !(reach(vkb) <= (double)rcol[q]) : 0;
        // the survivors (s <= tauf) must all be placed
        if (cut < C && bucket(__float_as_uint(tauf)) > last) s_left = 1;
        s_S = k;
    }
    __syncthreads();
    if (s_fail || s_left) {
        if (tid == 0) (s_fail ? retry : bigf)[q] = 1;
        if (s_fail)
            for (int t = tid; t < Npmax; t += NT) out[t] = -1;
        return;
    }
    const float tauf = s_tauf, d2f = s_d2f;
    for (int e = k + tid; e < cut; e += NT)
        if (__uint_as_float((uint32_t)(sk[e] >> 32)) <= tauf) atomicAdd(&s_S, 1);
    __syncthreads();
    const int S = s_S;
    // tie flags (bit i: rows i and i + 1 need their FP64 order) before any run is re-ordered
    for (int i0 = tid - lane; i0 < S; i0 += NT) {
        const int i = i0 + lane;
        bool t = false;
        if (i + 1 < S) {
            // the FP32 difference rounded down never exceeds the true one
            const float x = __uint_as_float((uint32_t)(sk[i] >> 32)), y = __uint_as_float((uint32_t)(sk[i + 1] >> 32));
            t = !(__fsub_rd(y, x) > d2f);
        }
        const uint32_t m = __ballot_sync(LAGP_FULL_MASK, t);
        if (lane == 0) tied[i0 >> 5] = m;
    }
    __syncthreads();
    auto is_tied = [&](int i) { return (tied[i >> 5] >> (i & 31)) & 1u; };
    // FP64 distances of the rows in runs, gathered so that they share the FP64
    // unit's instructions (it takes as long for one lane as for 32)
    for (int i = tid; i < S; i += NT)
        if (is_tied(i) || (i > 0 && is_tied(i - 1))) list[atomicAdd(&s_ties, 1)] = (uint16_t)i;
    __syncthreads();
    for (int e = tid; e < s_ties; e += NT) {
        const int t = list[e];
        const int32_t r = (int32_t)(uint32_t)sk[t];
        double sd = 0.0;
        for (int c = 0; c < p; c++) {
            const double diff = __dsub_rn(xq[c], load_coord64(X, r, p, c, dt));
            sd = __dadd_rn(sd, __dmul_rn(diff, diff));
        }
        dk[t] = sd;
    }
    __syncthreads();
    for (int i = tid; i < S; i += NT) {
        if (!is_tied(i) || (i > 0 && is_tied(i - 1))) continue;  // not the start of a run
        int end = i + 1;  // the run is [i, end]
        while (is_tied(end) && end - i < 32) end++;
        if (end - i >= 32) {
            s_left = 1;
            continue;
        }
        for (int t = i + 1; t <= end; t++) {  // insertion sort on (d2, row)
            const double dv = dk[t];
            const unsigned long long kv = sk[t];
            int u = t - 1;
            while (u >= i && pair_less(dv, (uint32_t)kv, dk[u], (uint32_t)sk[u])) {
                dk[u + 1] = dk[u];
                sk[u + 1] = sk[u];
                u--;
            }
            dk[u + 1] = dv;
            sk[u + 1] = kv;
        }
    }
    __syncthreads();
    if (s_left) {
        if (tid == 0) bigf[q] = 1;
        return;
    }
    for (int t = tid; t < Npmax; t += NT) out[t] = t < k ? (int32_t)(uint32_t)sk[t] : -1;
}

// The screen on CUDA cores (norm expansion), and the exact retry of the
// flagged queries (direct form).
template <int P>
void launch_screen(lagp_ctx *ctx, bool retry_pass, dim3 grid, size_t smem, const float *Y32, const float *Ys,
                   int64_t N, int p, const void *Xref, lagp_dtype dt, int64_t M, const int32_t *Np, int32_t Npmax,
                   const unsigned long long *kmax, const unsigned long long *kmin, int32_t *cand, int32_t Cmax,
                   int32_t *cc, int32_t *status, int64_t stride, int32_t *retry, int *counters) {
    cudaStream_t st = ctx->stream;
    if (!retry_pass) {
        cudaFuncSetAttribute(knn_screen<P, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        knn_screen<P, true><<<grid, SCREEN_THREADS, smem, st>>>(Y32, Ys, N, p, Xref, dt, M, Np, Npmax, kmax, kmin,
                                                                cand, Cmax, cc, status, stride, retry, 0, counters);
    } else {
        cudaFuncSetAttribute(knn_screen<P, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        knn_screen<P, false><<<grid, SCREEN_THREADS, smem, st>>>(Y32, Y32, N, p, Xref, dt, M, Np, Npmax, kmax,
                                                                 kmin, cand, Cmax, cc, status, 1, retry, 1,
                                                                 counters + 1);
    }
    ctx->launches++;
}

// The sampled thresholds.  Queries a warp, warps a query group and rows of the
// first sweep follow the problem: four queries a warp keep the sweep off the
// shared-memory loads (9 loads for 36 multiply-adds at p = 8); with few
// queries all eight warps share a group, and then one query, so that M = 100
// still meets 100 SMs.
template <int P>
void launch_sample(lagp_ctx *ctx, const float *Ys, int64_t nsamp, int p, const void *Xref, lagp_dtype dt, int64_t M,
                   const int32_t *Np, int32_t Npmax, int64_t stride, const unsigned long long *kmax,
                   const unsigned long long *kmin, int *counter, float *tau0) {
    const int64_t rt = sample_rank(Npmax, stride, nsamp);
    const int pp = row_stride(p);
    auto go = [&](auto kern, int qw, int W) {
        // first sweep: one row in `first`, so that a thread lists about a
        // quarter of its column's depth (a few in 10^4 columns overflow)
        const int64_t first = std::min<int64_t>(8, SAMPLE_DEPTH / 5 * 32 * W / rt);
        int64_t nsub = first >= 2 ? (nsamp + first - 1) / first : 0;
        if (nsub < rt) nsub = 0;
        const int nq = 8 * qw / W;
        const size_t smem = (size_t)nq * SAMPLE_DEPTH * 32 * W * 4 + 2 * (size_t)sample_tile(pp) * pp * 4 + (size_t)nq * pp * 4;
        const int64_t nblk = (M + nq - 1) / nq;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kern<<<(unsigned)std::min<int64_t>(nblk, (int64_t)ctx->num_sms * 2), SCREEN_THREADS, smem, ctx->stream>>>(
            Ys, nsamp, nsub, p, Xref, dt, M, Np, Npmax, stride, kmax, kmin, counter, tau0);
    };
    if (M >= 32 * (int64_t)ctx->num_sms) go(knn_sample<P, 4, 2>, 4, 2);
    else if (M >= 4 * (int64_t)ctx->num_sms) go(knn_sample<P, 4, 8>, 4, 8);
    else go(knn_sample<P, 1, 8>, 1, 8);
    ctx->launches++;
}

}  // namespace

lagp_status launch_knn(lagp_ctx *ctx, const void *X, int64_t N, int p, lagp_dtype dtype,
                       const void *Xref, int64_t M, const int32_t *Np, int32_t Npmax,
                       int32_t *idx, int32_t *status) {
    cudaStream_t st = ctx->stream;
    ctx->knn_last_M = M;
    // sample stride: about 8 N' sampled rows per candidate set, 1 (exact) for small designs
    const int64_t stride = std::max<int64_t>(1, std::min<int64_t>(64, N / (8 * (int64_t)Npmax)));
    const int64_t nsamp = (N + stride - 1) / stride;
    // candidate capacity: the sampled threshold (the rtarget-th smallest of
    // every stride-th row, rtarget ~ 1.3 N' / stride + 16) collects about
    // rtarget stride rows with a spread of about sqrt(rtarget) stride; six of
    // those spreads above (and 512 rows for the error margins) leave an
    // overflow, and so an exact retry over the whole design (one CTA's pass
    // over all N rows: at N = 4M it sets the pass's duration), to about one
    // query in 1e9.  At least 2 N' + 1024, and no more than the power of two
    // at or above that, or 4,096 where that is more: with few neighbours of many
    // rows the error margin widens the threshold most, and a capacity of 2,048
    // left a query in 30 to the exact retry (N = 1.4M, N' = 88, p = 2, 116
    // queries: 6.5 ms with three of them, 2.1 without).  Above 4,096 the rank takes 512 threads a
    // query, a third slower.
    int32_t Cmax = std::min(2 * Npmax + 1024, CAND_CAP);
    if (stride > 1) {
        int32_t pow2 = 1;
        while (pow2 < Cmax) pow2 <<= 1;
        const int64_t rt = sample_rank(Npmax, stride, nsamp);
        const double want = (double)rt * stride + 6.0 * std::sqrt((double)rt) * stride + 512.0;
        Cmax = (int32_t)std::min<double>(std::max<double>(Cmax, std::ceil(want)), std::min(std::max(pow2, 4096), CAND_CAP));
    }
    char *meta = static_cast<char *>(lagp_ws(ctx, WS_KNN_META, META_HEAD + (size_t)M * 12));
    int32_t *cand = static_cast<int32_t *>(lagp_ws(ctx, WS_KNN_CAND, (size_t)M * Cmax * 4));
    const int pp = row_stride(p);
    const int64_t Npad = round_up(N, 32);
    const int64_t nsamp_pad = stride > 1 ? round_up(nsamp, 32) : 0;
    const int pv = (p + 3) & ~3;
    float *Y32 = static_cast<float *>(lagp_ws(ctx, WS_KNN_X32, ((size_t)(Npad + nsamp_pad) * pp + (size_t)Npad * pv) * 4));
    if (!meta || !cand || !Y32) return LAGP_ENOMEM;
    float *Ys = stride > 1 ? Y32 + Npad * pp : Y32;
    float *Yv = Y32 + (Npad + nsamp_pad) * pp;  // 16-byte aligned: Npad is a multiple of 32
    int *counters = reinterpret_cast<int *>(meta + 64);
    unsigned long long *kmax = reinterpret_cast<unsigned long long *>(meta + 256);
    unsigned long long *kmin = reinterpret_cast<unsigned long long *>(meta + 768);
    int32_t *cc = reinterpret_cast<int32_t *>(meta + META_HEAD);
    int32_t *retry = cc + M;
    int32_t *bigf = retry + M;  // queries that the rank leaves to the general sort
    LAGP_CUDA(ctx, cudaMemsetAsync(meta, 0, META_HEAD, st));
    LAGP_CUDA(ctx, cudaMemsetAsync(bigf, 0, (size_t)M * 4, st));
    const int blocks = ctx->num_sms * 4;
    knn_bounds<<<blocks, 256, 0, st>>>(X, N, Xref, M, p, dtype, kmax, kmin);
    KnnConst *kc = reinterpret_cast<KnnConst *>(meta + META_CONST);
    // the spatial order, for the tensor-core collection of large problems
    const bool tc = ctx->tuning.knn_path == 0 && knn_tc_supported(p);
    KnnOrder order;
    if (tc && N >= ORD_MIN_ROWS && N * M >= ORD_MIN_PAIRS) {
        const int nmb = (int)((N + 127) / 128);
        const size_t oRow = (size_t)ORD_CELLS * 8, oQuery = oRow + (size_t)N * 4, oBox = oQuery + (size_t)M * 4,
                     oCell = oBox + (size_t)2 * p * nmb * 4;
        char *w = static_cast<char *>(lagp_ws(ctx, WS_KNN_ORDER, oCell + (size_t)(N + M) * 2 + 16));
        if (!w) return LAGP_ENOMEM;
        uint32_t *hist = reinterpret_cast<uint32_t *>(w);
        int32_t *row = reinterpret_cast<int32_t *>(w + oRow), *query = reinterpret_cast<int32_t *>(w + oQuery);
        uint16_t *cell = reinterpret_cast<uint16_t *>(w + oCell);
        LAGP_CUDA(ctx, cudaMemsetAsync(hist, 0, (size_t)ORD_CELLS * 8, st));
        knn_cells<<<blocks, 256, 0, st>>>(X, N, Xref, M, p, dtype, kmax, kmin, cell, hist);
        knn_cell_starts<<<2, 1024, 0, st>>>(hist);
        knn_cell_scatter<<<blocks, 256, 0, st>>>(cell, N, M, hist, row, query);
        ctx->launches += 3;
        order.row = row;
        order.query = query;
        order.box = reinterpret_cast<float *>(w + oBox);
    }
    int64_t spread = std::max<int64_t>(1, (int64_t)(0.6180339887 * (double)nsamp));
    while (std::gcd(spread, nsamp) != 1) spread++;
    knn_prep<<<blocks, 256, 0, st>>>(X, N, p, dtype, kmax, kmin, order.row, Y32, Npad, stride > 1 ? Ys : nullptr,
                                     nsamp, nsamp_pad, stride, spread, kc, Yv);
    ctx->launches += 2;
    if (order.box) {
        knn_boxes<<<blocks, 256, 0, st>>>(Y32, N, p, (int)((N + 127) / 128), order.box);
        ctx->launches++;
    }
    LAGP_CUDA(ctx, cudaGetLastError());
    // collection on the tensor cores unless the tuning asks for CUDA cores
    void *tc_ws = nullptr;
    float *tau0 = nullptr, *rcol = nullptr;
    if (tc) {
        tc_ws = lagp_ws(ctx, WS_KNN_TC, knn_tc_workspace(N, M, p));
        if (!tc_ws) return LAGP_ENOMEM;
        LAGP_TRY(launch_knn_tc_prep(ctx, tc_ws, X, N, p, dtype, Xref, M, kmax, kmin, order, &tau0, &rcol));
    }
    int *tc_err = reinterpret_cast<int *>(meta);

    size_t smem = (size_t)QB * HB * 4 + 2 * (size_t)tile_len(pp) * pp * 4 + (size_t)(QB + 1) * pp * 4;
    // persistent grid: two CTAs per SM, blocks of QB queries from a counter
    const int64_t nblk = (M + QB - 1) / QB;
    dim3 grid((unsigned)std::min<int64_t>(nblk, (int64_t)ctx->num_sms * 2));
    int Cp = 1;
    while (Cp < Cmax) Cp <<= 1;
    // shared memory of the rank (rows placed: N' and what shares the last
    // buckets) and of the general sort
    const int cap = std::min<int>((Npmax + Npmax / 8 + 128 + 31) & ~31, (Cmax + 31) & ~31);
    const size_t smem_rank = (size_t)rank_buckets(cap) * 4 + (size_t)cap * 10 + (size_t)(cap / 32 + 1) * 4;
    const size_t smem_big = (size_t)Cp * 16;
    if (std::max(smem_big, smem_rank) > ctx->smem_optin) return lagp_fail(ctx, LAGP_EINVAL, "lagp_knn: N' too large for the sort");
    cudaFuncSetAttribute(knn_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_big);
    auto screen = [&](bool retry_pass) {
        switch (p) {
            case 2: launch_screen<2>(ctx, retry_pass, grid, smem, Y32, Ys, N, p, Xref, dtype, M, Np, Npmax, kmax, kmin, cand, Cmax, cc, status, stride, retry, counters); break;
            case 3: launch_screen<3>(ctx, retry_pass, grid, smem, Y32, Ys, N, p, Xref, dtype, M, Np, Npmax, kmax, kmin, cand, Cmax, cc, status, stride, retry, counters); break;
            case 8: launch_screen<8>(ctx, retry_pass, grid, smem, Y32, Ys, N, p, Xref, dtype, M, Np, Npmax, kmax, kmin, cand, Cmax, cc, status, stride, retry, counters); break;
            default: launch_screen<0>(ctx, retry_pass, grid, smem, Y32, Ys, N, p, Xref, dtype, M, Np, Npmax, kmax, kmin, cand, Cmax, cc, status, stride, retry, counters); break;
        }
    };
    auto rank = [&]() {
        auto go = [&](auto kern, unsigned nt) {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_rank);
            kern<<<(unsigned)M, nt, smem_rank, st>>>(X, Yv, order.row, p, dtype, Xref, Np, Npmax, cand, cc, Cmax, cap,
                                                     idx, kc, rcol, retry, bigf);
        };
        if (Cmax <= 8 * 256) go(knn_rank<8, 256>, 256);
        else if (Cmax <= 16 * 256) go(knn_rank<16, 256>, 256);
        else go(knn_rank<16, 512>, 512);
        ctx->launches++;
    };
    auto sort = [&](int32_t *rflags) {
        const unsigned g = (unsigned)std::min<int64_t>(M, (int64_t)ctx->num_sms * 3);
        knn_sort<<<g, SORT_THREADS, smem_big, st>>>(X, Yv, order.row, p, dtype, Xref, M, Np, Npmax, cand, cc, Cmax,
                                                    idx, kc, rflags, bigf);
        ctx->launches++;
    };
    if (tc_ws) {
        switch (p) {
            case 2: launch_sample<2>(ctx, Ys, nsamp, p, Xref, dtype, M, Np, Npmax, stride, kmax, kmin, counters, tau0); break;
            case 3: launch_sample<3>(ctx, Ys, nsamp, p, Xref, dtype, M, Np, Npmax, stride, kmax, kmin, counters, tau0); break;
            case 8: launch_sample<8>(ctx, Ys, nsamp, p, Xref, dtype, M, Np, Npmax, stride, kmax, kmin, counters, tau0); break;
            default: launch_sample<0>(ctx, Ys, nsamp, p, Xref, dtype, M, Np, Npmax, stride, kmax, kmin, counters, tau0); break;
        }
    } else {
        screen(false);
    }
    LAGP_CUDA(ctx, cudaGetLastError());
    if (tc_ws) {
        // collection on the tensor cores, the rank (which checks each query's
        // collection), the exact retry of the flagged queries and their sort
        LAGP_TRY(launch_knn_tc_collect(ctx, tc_ws, N, p, Xref, dtype, M, Np, Npmax, kmax, kmin, order, cand, Cmax, cc,
                                       status, retry, tc_err, counters + 2, rcol, nullptr));
        rank();
        screen(true);
        sort(retry);
    } else {
        screen(true);
        rank();
        sort(nullptr);
    }
    LAGP_CUDA(ctx, cudaGetLastError());
    return LAGP_OK;
}

// Diagnostic: the tensor-core values s of every (query, design row) pair, as
// the collection pass computes them (out: M x N floats).
lagp_status launch_knn_tc_dist(lagp_ctx *ctx, const void *X, int64_t N, int p, lagp_dtype dtype,
                               const void *Xref, int64_t M, float *out) {
    if (!knn_tc_supported(p)) return lagp_fail(ctx, LAGP_EINVAL, "lagp_knn_tc_dist: p > 20");
    cudaStream_t st = ctx->stream;
    char *meta = static_cast<char *>(lagp_ws(ctx, WS_KNN_META, META_HEAD + (size_t)M * 12));
    void *tc_ws = lagp_ws(ctx, WS_KNN_TC, knn_tc_workspace(N, M, p));
    if (!meta || !tc_ws) return LAGP_ENOMEM;
    unsigned long long *kmax = reinterpret_cast<unsigned long long *>(meta + 256);
    unsigned long long *kmin = reinterpret_cast<unsigned long long *>(meta + 768);
    int32_t *cc = reinterpret_cast<int32_t *>(meta + META_HEAD);
    int32_t *retry = cc + M;
    LAGP_CUDA(ctx, cudaMemsetAsync(meta, 0, META_HEAD, st));
    knn_bounds<<<ctx->num_sms * 4, 256, 0, st>>>(X, N, Xref, M, p, dtype, kmax, kmin);
    ctx->launches++;
    LAGP_CUDA(ctx, cudaGetLastError());
    float *tau0 = nullptr, *rcol = nullptr;
    LAGP_TRY(launch_knn_tc_prep(ctx, tc_ws, X, N, p, dtype, Xref, M, kmax, kmin, KnnOrder{}, &tau0, &rcol));
    return launch_knn_tc_collect(ctx, tc_ws, N, p, Xref, dtype, M, nullptr, 1, kmax, kmin, KnnOrder{}, nullptr, 1, cc,
                                 nullptr, retry, reinterpret_cast<int *>(meta), reinterpret_cast<int *>(meta + 72), rcol,
                                 out);
}

// Diagnostic: of the last kNN call on the context, the queries that went to
// the exact retry and whether the tensor-core pass gave up on a wait.
lagp_status knn_last_stats(lagp_ctx *ctx, int64_t *n_retry, int32_t *tc_failed) {
    const int64_t M = ctx->knn_last_M;
    char *meta = static_cast<char *>(ctx->ws[WS_KNN_META]);
    if (!meta || M <= 0) {
        *n_retry = 0;
        *tc_failed = 0;
        return LAGP_OK;
    }
    std::vector<int32_t> r((size_t)M);
    int32_t f = 0;
    LAGP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    LAGP_CUDA(ctx, cudaMemcpy(r.data(), meta + META_HEAD + (size_t)M * 4, (size_t)M * 4, cudaMemcpyDeviceToHost));
    LAGP_CUDA(ctx, cudaMemcpy(&f, meta, 4, cudaMemcpyDeviceToHost));
    int64_t n = 0;
    for (int32_t v : r) n += v != 0;
    *n_retry = n;
    *tc_failed = f;
    return LAGP_OK;
}
