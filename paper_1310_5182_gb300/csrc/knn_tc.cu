// a1, collection pass of the exact N'-nearest-neighbour screen on the
// tensor cores (Sec. 3.1: the candidate set of a location is its N' nearest
// design points).
//
// The squared distances s = |y_q|^2 + |y_x|^2 - 2 y_q . y_x between centred
// FP32 coordinates form a dense (design x queries) contraction over the p
// coordinates, here one tcgen05.mma chain (kind::f16, FP32 accumulation) per
// 128 design rows.  The coordinates are scaled by the power of two 2^-e that
// brings them into [-1, 1] (exact), and every FP32 value v enters as a
// two-term FP16 split v = v_h + v_l, the dot product as the three products
//   y_qh . y_xh + y_ql . y_xh + y_qh . y_xl        (y_ql . y_xl dropped),
// each exact in FP32; the two squared norms enter split the same way against
// unit entries.  Operand rows (K FP16 values each, K = 3p + 4 rounded up to
// 16, one MMA instruction per 16):
//   design x: ( y_xh, y_xh, y_xl, 1, 1, n_xh, n_xl, 0 ... )
//   query q:  ( -2 y_qh, -2 y_ql, -2 y_qh, n_qh, n_ql, 1, 1, 0 ... )
// so that the accumulator holds s 2^-2e for every (design row, query) pair.
//
// Exactness: the rows with s <= tau2 are collected, tau2 a rigorous widening
// (tc_margin) of the sampled threshold tau0 (itself widened by 2 E_tc so that
// rows at the sample's boundary fall inside whatever the rounding of either
// pass).  The rank then checks that the N'-th collected row lies within the
// radius that tau2 guarantees collected (tc_collected_radius, stored per
// query), also before it leaves a query to the general sort; a query that
// fails, or whose buffer overflows, goes to the exact CUDA-core retry.  E_tc
// (knn_common.cuh) assumes that one tensor-core instruction adds its products
// and accumulator with an error of at most TC_ACC_ULPS = 64 units of 2^-24
// times the sum of their magnitudes, several times what a truncating
// alignment of its seventeen addends can lose.
//
// With a spatial order (KnnOrder) the operands' rows are sorted by cell, and a
// query block meets only the design blocks whose bounding box comes within the
// largest threshold of its own box: 500,000 rows in 3 dimensions, 201,600
// queries, 34.6 -> 5.7 ms.  In 8 dimensions few blocks fall away (a ball with
// 2,000 of 4M uniform rows reaches most of the cube): 40.1 -> 38.1 ms.
//
// Kernel layout (one CTA per SM, persistent over blocks of up to 64 queries):
// four groups, each of one warp that copies and multiplies and four epilogue
// warps (one per TMEM lane quarter), take the listed design blocks in turn.
// The one thread of a copy and MMA warp streams its design blocks into a ring
// of shared-memory stages with bulk asynchronous copies and issues their MMAs
// into the group's two accumulators of 64 columns; the epilogue warps read the
// distances back.  The thresholds are folded into the queries' norm terms
// (n_q - tau2), so that a row to collect is a negative accumulator: a lane
// gathers its design row's sign bits, one funnel shift a column, and visits
// the set bits (0.1 to 10% of the pairs) to append the row to the queries'
// candidate lists.
//
// What bounds it: the epilogue's funnel shifts, one a pair (the ALU pipe 62%
// busy, 55% of the issue slots taken; the tensor pipe 15%), and the design
// operand's reads from the L2 (5.5 TB/s).  With one thread for all copies, one for all MMAs (and
// 64-bit divisions in both), every design block waited for them in turn, 490 ns
// whatever its width; four such threads that also copy for themselves, 25.7 ->
// 23.8 ms (4M rows, 25,000 queries, p = 8, N' = 2,000); accumulators of 64
// columns, one TMEM load for all of them, and hits appended by the lane that
// found them, no queue, 23.8 -> 18.3 ms.  Before all of it 38.1 ms; 500,000 rows
// in 3 dimensions, 201,600 queries, N' = 1,500: 5.7 -> 3.6 ms.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>

#include "device_util.cuh"
#include "knn_common.cuh"
#include "lagp_internal.h"
#include "tc_sm100.cuh"

namespace {

constexpr int TC_EPI_GROUPS = 4;  // epilogue groups of four warps (one per TMEM lane quarter)
constexpr int TC_EPI_WARP = TC_EPI_GROUPS;  // a copy and MMA warp a group, then the epilogue
constexpr int TC_THREADS = 32 * (TC_EPI_WARP + 4 * TC_EPI_GROUPS);
constexpr int TC_MROWS = 128;    // design rows per MMA (M)
constexpr int TC_STAGES_MAX = 4; // design stages a group (3 for wide rows)
constexpr int TC_NACC = 2 * TC_EPI_GROUPS;  // TMEM accumulators: two a group
constexpr int TC_ACC_COLS = 64;
constexpr int TC_TMEM_COLS = TC_NACC * TC_ACC_COLS;  // 512: the whole tensor memory of the SM
constexpr int TC_QMAX = TC_ACC_COLS;  // queries per block (MMA N <= 64)
constexpr int TC_CHUNK = 8192;  // design blocks whose survivors are listed at a time

// Half offset of element k of operand row r in the no-swizzle K-major
// layout: 8-row groups of K / 8 core matrices (8 rows x 8 halves, 128 bytes),
// the core matrices of a group adjacent along K.
__device__ __forceinline__ int64_t tc_off(int64_t r, int k, int K) {
    return (r >> 3) * (8 * (int64_t)K) + (k >> 3) * 64 + (r & 7) * 8 + (k & 7);
}

// v = h + l with h, l FP16 (round to nearest): |v - h - l| <= max(2^-22 |v|, 2^-25)
// for |v| <= 2
__device__ __forceinline__ void f16_split(float v, __half &h, __half &l) {
    h = __float2half_rn(v);
    l = __float2half_rn(v - __half2float(h));
}

// The centred FP32 coordinates y and squared norm n of row r of A, exactly as
// the CUDA-core screen computes them (the norm an FMA chain in coordinate
// order).
__device__ __forceinline__ float centred_coords(const void *A, int64_t r, int p, lagp_dtype dt,
                                                const double *c, float *y) {
    float n2 = 0.f;
    for (int i = 0; i < p; i++) {
        y[i] = (float)(load_coord64(A, r, p, i, dt) - c[i]);
        n2 = fmaf(y[i], y[i], n2);
    }
    return n2;
}

// Design operand (Npad rows, blocked layout; rows past N are zero) and query
// operand rows (M x K, row-major), FP16, both in the launch's order.
__global__ void knn_tc_prep(const void *__restrict__ X, int64_t N, int64_t Npad, const void *__restrict__ Xr,
                            int64_t M, int p, lagp_dtype dt, const unsigned long long *kmax,
                            const unsigned long long *kmin, KnnOrder order, __half *__restrict__ A,
                            __half *__restrict__ Q) {
    __shared__ double c[64];
    __shared__ double sB;
    if (threadIdx.x == 0) centre_and_bound(kmax, kmin, p, c, sB);
    __syncthreads();
    const int K = tc_k(p);
    const float scale = ldexpf(1.f, -tc_scale_exp(sB));
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    float y[20];
    __half row[64];  // p <= 20, K <= 64 (knn_tc_supported)
    const __half one = __float2half_rn(1.f), zero = __float2half_rn(0.f);
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < Npad + M; r += stride) {
        const bool des = r < Npad;
        const int64_t rr = des ? r : r - Npad;
        for (int k = 0; k < K; k++) row[k] = zero;
        if (!des || rr < N) {
            const int32_t *perm = des ? order.row : order.query;
            centred_coords(des ? X : Xr, perm ? perm[rr] : rr, p, dt, c, y);
            float n2 = 0.f;  // |y 2^-e|^2: the FP32 chain of the unscaled norm, scaled exactly
            for (int i = 0; i < p; i++) {
                y[i] *= scale;
                n2 = fmaf(y[i], y[i], n2);
            }
            __half nh, nl;
            f16_split(n2, nh, nl);
            for (int i = 0; i < p; i++) {
                __half vh, vl;
                f16_split(des ? y[i] : -2.f * y[i], vh, vl);  // -2 y_q: an exact scaling
                row[i] = vh;
                row[p + i] = des ? vh : vl;
                row[2 * p + i] = des ? vl : vh;
            }
            if (!(n2 < CUDART_INF_F)) {  // a NaN or infinite coordinate: an infinite distance, not a NaN of some sign
                for (int i = 0; i < 3 * p; i++) row[i] = zero;
                nh = __ushort_as_half(0x7c00), nl = zero;
            }
            row[3 * p] = des ? one : nh;
            row[3 * p + 1] = des ? one : nl;
            row[3 * p + 2] = des ? nh : one;
            row[3 * p + 3] = des ? nl : one;
        }
        __half *dst = des ? A : Q + rr * K;
        for (int k = 0; k < K; k += 8) {
            uint4 v;
            __half *hv = reinterpret_cast<__half *>(&v);
            for (int j = 0; j < 8; j++) hv[j] = row[k + j];
            *reinterpret_cast<uint4 *>(des ? dst + tc_off(rr, k, K) : dst + k) = v;
        }
    }
}

struct TcArgs {
    const __half *A;  // design operand, nmb * 128 rows
    const __half *Q;  // query operand rows, M x K
    int64_t N, M;
    int p, K, nmb;
    KnnOrder order;
    const void *Xref;  // locations (for the blocks' bounding boxes)
    lagp_dtype dt;
    int *counter;      // blocks of queries taken
    const float *tau0;  // per query: sampled threshold, NaN = not screened
    float *rcol;        // per query out: the radius collected in full (rounded down; NaN: not collected)
    const int32_t *Np;
    int32_t Npmax;
    const unsigned long long *kmax, *kmin;
    int32_t *cand, Cmax;
    int32_t *cand_count, *status, *retry;
    int nq, nblocks;  // queries per block, blocks
    int stages;       // shared-memory stages of a group's design ring
    float *dump;      // diagnostic: every value s (M x N) instead of the collection
    int stall;        // test hook: the producer stops after the first design block
    int *err;         // raised when a bounded wait gave up (the block's queries go to the retry)
};

__global__ void __launch_bounds__(TC_THREADS, 1) knn_screen_tc(TcArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int K = a.K, S = a.stages;
    const int stage_halves = TC_MROWS * K;
    __half *sA = reinterpret_cast<__half *>(smem_raw);         // S stages a group x 128 rows
    __half *sQ = sA + (size_t)TC_EPI_GROUPS * S * stage_halves;                // TC_QMAX rows
    float *s_tau2 = reinterpret_cast<float *>(sQ + (size_t)TC_QMAX * K);  // TC_QMAX
    int *s_cnt = reinterpret_cast<int *>(s_tau2 + TC_QMAX);    // TC_QMAX
    uint16_t *s_list = reinterpret_cast<uint16_t *>(s_cnt + TC_QMAX);  // TC_CHUNK design blocks
    uint64_t *bar = reinterpret_cast<uint64_t *>(s_list + TC_CHUNK);
    uint64_t *full = bar, *tfull = bar + TC_EPI_GROUPS * S, *tempty = tfull + TC_NACC;
    __shared__ uint32_t s_tmem;
    __shared__ int s_err, s_blk, s_nlist;
    __shared__ int32_t s_q[TC_QMAX];  // the block's locations
    __shared__ int32_t *s_cand[TC_QMAX];  // and their candidate lists
    __shared__ double s_c[64], s_B;
    __shared__ uint32_t s_qlo[20], s_qhi[20], s_tmax;  // order-preserving keys of floats
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < TC_EPI_GROUPS * S; s++) mbar_init(full + s, 1);
        for (int c = 0; c < TC_NACC; c++) {
            mbar_init(tfull + c, 1);
            mbar_init(tempty + c, 4);  // the four warps of the group that reads it (group c / 2)
        }
        mbar_init_fence();
        s_err = 0;
        centre_and_bound(a.kmax, a.kmin, a.p, s_c, s_B);
    }
    if (warp == 1) {
        __syncwarp();
        tmem_alloc(&s_tmem, TC_TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = s_tmem;
    volatile int *err = &s_err;
    const uint32_t stage_bytes = (uint32_t)stage_halves * 2u;
    const uint32_t sbo = 8u * (uint32_t)K * 2u;  // bytes between 8-row groups
    // the operands carry 2^-e, the accumulators 2^-2e
    const float s2 = ldexpf(1.f, -2 * tc_scale_exp(s_B));

    // the warp's group (copies and MMAs: warp g; epilogue: four warps), and the
    // design blocks that it has seen, modulo 2^32 (its position in its ring)
    const int g = warp < TC_EPI_WARP ? warp : (warp - TC_EPI_WARP) >> 2;
    uint32_t round0 = 0;
    int ld_slot = 0, mma_slot = 0;  // the copying thread's: ring positions, and the phase of the copies awaited
    uint32_t mma_phase = 0;
    for (;;) {
        if (tid == 0) s_blk = atomicAdd(a.counter, 1);
        if (tid < 20) s_qlo[tid] = 0xFFFFFFFFu, s_qhi[tid] = 0u;
        if (tid == 20) s_tmax = 0u;
        __syncthreads();
        const int blk = s_blk;
        if (blk >= a.nblocks) break;
        const int64_t q0 = (int64_t)blk * a.nq;
        const int nqb = (int)min((int64_t)a.nq, a.M - q0);
        const int nmma = (nqb + 15) & ~15;  // MMA N: a multiple of 16
        // query operand and thresholds of this block
        for (int e = tid; e < nmma * K; e += TC_THREADS) {
            const int r = e / K, k = e - r * K;
            sQ[tc_off(r, k, K)] = r < nqb ? a.Q[(q0 + r) * K + k] : __float2half_rn(0.f);
        }
        for (int c = tid; c < TC_QMAX; c += TC_THREADS) {
            float t2 = CUDART_NAN_F;  // NaN: no row ever compares below
            if (c < nqb) {
                const int64_t q = a.order.query ? a.order.query[q0 + c] : q0 + c;
                const int k = a.Np ? a.Np[q] : a.Npmax;
                const float tq = a.tau0[q];
                if (k >= 1 && k <= a.Npmax && tq == tq) {
                    // the sampled threshold widened by 2 E_tc (rows at the
                    // sample's boundary fall inside whatever the rounding of
                    // either pass), then by the collection margin
                    const float t0 = __double2float_ru((double)tq + 2.0 * tc_error_bound(a.p, K, s_B));
                    t2 = __double2float_rd(tc_margin(t0, a.p, K, s_B));
                }
            }
            s_tau2[c] = t2 * s2;  // an exact scaling
            s_cnt[c] = 0;
            s_q[c] = c < nqb ? (int32_t)(a.order.query ? a.order.query[q0 + c] : q0 + c) : 0;
            s_cand[c] = a.cand + s_q[c] * (int64_t)a.Cmax;
            if (a.order.box && t2 == t2) atomicMax(&s_tmax, fkey(t2));
        }
        // the bounding box of the block's queries
        if (a.order.box)
            for (int e = tid; e < nqb * a.p; e += TC_THREADS) {
                const int c = e / a.p, i = e - c * a.p;
                const float y = (float)(load_coord64(a.Xref, a.order.query[q0 + c], a.p, i, a.dt) - s_c[i]);
                if (y == y) {
                    atomicMin(&s_qlo[i], fkey(y));
                    atomicMax(&s_qhi[i], fkey(y));
                }
            }
        __syncthreads();
        // the thresholds folded into the queries' norms, n_q - tau2, so that an
        // accumulator is negative exactly for a row to collect (a query that
        // is not screened: infinite, never negative)
        if (!a.dump)
            for (int c = tid; c < nqb; c += TC_THREADS) {
                __half *nh = sQ + tc_off(c, 3 * a.p, K), *nl = sQ + tc_off(c, 3 * a.p + 1, K);
                const float t2 = s_tau2[c];
                __half h = __ushort_as_half(0x7c00), l = __float2half_rn(0.f);
                if (t2 == t2) f16_split((__half2float(*nh) + __half2float(*nl)) - t2 * (1.f + 0x1p-20f), h, l);
                *nh = h;
                *nl = l;
            }
        fence_proxy_async_smem();
        // Design blocks that may hold a row to collect, a chunk at a time: with
        // boxes, those whose box lies within the largest threshold of the
        // queries' box.  Every row of another block is further from every
        // query than sqrt(tau2) (the FP32 evaluation's relative error is below
        // 1e-5), outside the radius that tau2 guarantees collected.
        for (int chunk = 0; chunk < a.nmb; chunk += TC_CHUNK) {
        // (every role of the chunk before is done: a block-uniform verdict)
        if (__syncthreads_or(*err != 0)) break;
        if (tid == 0) s_nlist = 0;
        __syncthreads();
        for (int m0 = chunk; m0 < min(chunk + TC_CHUNK, a.nmb); m0 += TC_THREADS) {
            const int mb = m0 + tid;
            bool take = mb < min(chunk + TC_CHUNK, a.nmb);
            if (a.order.box && take) {
                float lb = 0.f;
                for (int i = 0; i < a.p; i++) {
                    const float lo = a.order.box[(int64_t)i * a.nmb + mb], hi = a.order.box[(int64_t)(a.p + i) * a.nmb + mb];
                    const float gap = fmaxf(fmaxf(fkey_inv(s_qlo[i]) - hi, lo - fkey_inv(s_qhi[i])), 0.f);
                    lb = fmaf(gap, gap, lb);
                }
                take = !(lb * (1.f - 1e-5f) > fkey_inv(s_tmax));
            }
            const uint32_t vote = __ballot_sync(LAGP_FULL_MASK, take);
            int at = 0;
            if (lane == 0 && vote) at = atomicAdd(&s_nlist, __popc(vote));
            at = __shfl_sync(LAGP_FULL_MASK, at, 0);
            if (take) s_list[at + __popc(vote & ((1u << lane) - 1u))] = (uint16_t)(mb - chunk);
        }
        __syncthreads();
        const int nlist = s_nlist;
        const int cnt = (nlist - g + TC_EPI_GROUPS - 1) / TC_EPI_GROUPS;  // the group's: g, g + 4, ...

        if (warp < TC_EPI_WARP) {
            if (lane == 0) {  // one thread: the group's copies and MMAs
                const uint32_t idesc = idesc_f16_f32(TC_MROWS, nmma);
                const uint64_t qdesc = smem_desc_kmajor(smem_u32(sQ), 128u, sbo);
                __half *ring = sA + (size_t)g * S * stage_halves;
                const uint64_t adesc = smem_desc_kmajor(smem_u32(ring), 128u, sbo);
                uint64_t *const gfull = full + g * S;
                int loaded = 0, landed = 0, issued = 0;
                auto load = [&]() {  // the next design block into the ring
                    const int li = g + loaded * TC_EPI_GROUPS;
                    if (loaded >= cnt || (a.stall && li >= 1)) return;  // (stall: the wait on it then runs out)
                    mbar_arrive_expect_tx(gfull + ld_slot, stage_bytes);
                    bulk_g2s(ring + (size_t)ld_slot * stage_halves, a.A + (size_t)(chunk + s_list[li]) * stage_halves,
                             stage_bytes, gfull + ld_slot);
                    loaded++;
                    if (++ld_slot == S) ld_slot = 0;
                };
                auto land = [&](volatile int *e) {  // waits for the next copy
                    if (!mbar_wait(gfull + mma_slot, mma_phase, e, 32)) return false;
                    landed++;
                    return true;
                };
                auto next = [&]() {
                    if (++mma_slot == S) mma_slot = 0, mma_phase ^= 1u;
                };
                for (int k = 0; k < S; k++) load();
                for (int k = 0; k < cnt; k++) {
                    const uint32_t round = round0 + (uint32_t)k, ac = (uint32_t)g * 2u + (round & 1u);
                    if (!mbar_wait(tempty + ac, ((round >> 1) & 1u) ^ 1u, err, 32)) break;
                    // the accumulator was read, so the block two before this one
                    // is through its MMAs: its stage takes the next copy
                    if (k > 1) load();
                    if (!land(err)) break;
                    tc_fence_after_sync();
                    // (descriptors address shared memory in 16-byte units)
                    const uint64_t ad = adesc + ((uint32_t)mma_slot * stage_bytes >> 4);
                    for (int ks = 0; ks < K / 16; ks++)  // 16 halves (two core matrices) per MMA
                        mma_f16(tmem + ac * TC_ACC_COLS, ad + 16u * ks, qdesc + 16u * ks, idesc, ks > 0 ? 1u : 0u);
                    mma_commit(tfull + ac);  // the accumulator is ready
                    issued = k + 1;
                    next();
                }
                if (*err) {  // the copies in flight land and the MMAs issued finish before the CTA moves on
                    int quiet = 0;
                    if (landed > issued) next();
                    for (; landed < loaded; next())
                        if (!land(&quiet)) break;
                    if (issued) {
                        const uint32_t round = round0 + (uint32_t)issued - 1u;
                        mbar_wait(tfull + g * 2 + (round & 1u), (round >> 1) & 1u, &quiet);
                    }
                }
            }
        } else {
            // epilogue: group g reads accumulators 2g and 2g + 1 in turn, of the listed
            // design blocks g, g + 4, ...; each warp its TMEM lane quarter (32 design rows)
            const int quarter = warp & 3;
            // the columns that are queries, the first one's bit on top
            const unsigned long long cols = nqb < 64 ? ~(~0ull >> nqb) : ~0ull;
            for (int k = 0; k < cnt; k++) {
                const uint32_t round = round0 + (uint32_t)k, ac = (uint32_t)g * 2u + (round & 1u);
                const int li = g + k * TC_EPI_GROUPS;
                const int mb = chunk + s_list[li];
                // every lane waits; the warp goes on only together (the TMEM
                // loads are warp-collective)
                const bool ready = mbar_wait(tfull + ac, (round >> 1) & 1u, err, 64);
                if (!__all_sync(LAGP_FULL_MASK, ready)) break;
                tc_fence_after_sync();
                const int64_t row = (int64_t)mb * TC_MROWS + quarter * 32 + lane;
                uint32_t v[64];
                tmem_ld64(tmem + ((uint32_t)(quarter * 32) << 16) + ac * TC_ACC_COLS, v);
                tmem_wait_ld64(v);
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty + ac);  // every column read: release the accumulator
                if (a.dump) {
#pragma unroll
                    for (int c = 0; c < 64; c++)
                        if (c < nqb && row < a.N) a.dump[(q0 + c) * a.N + row] = __uint_as_float(v[c]) / s2;
                    __syncwarp();
                    continue;
                }
                uint32_t m0 = 0, m1 = 0;  // the sign bits, the first column's on top
#pragma unroll
                for (int i = 0; i < 32; i++) {
                    m0 = __funnelshift_l(v[i], m0, 1);
                    m1 = __funnelshift_l(v[32 + i], m1, 1);
                }
                for (unsigned long long m = row < a.N ? ((unsigned long long)m0 << 32 | m1) & cols : 0ull; m;) {
                    const int c = __clzll((long long)m);
                    m &= ~(0x8000000000000000ull >> c);
                    const int pos = atomicAdd(&s_cnt[c], 1);
                    if (pos < a.Cmax) s_cand[c][pos] = (int32_t)row;
                }
                __syncwarp();
            }
        }
        round0 += (uint32_t)cnt;
        }
        __syncthreads();
        // per-query results: the collected rows and the threshold they were
        // collected under (the rank checks that the N'-th of them lies within
        // the radius that threshold guarantees); an overflowing or
        // unscreened query goes to the exact retry
        const bool failed = *err != 0;
        for (int c = tid; c < nqb; c += TC_THREADS) {
            const int64_t q = s_q[c];
            const int k = a.Np ? a.Np[q] : a.Npmax;
            const bool kvalid = k >= 1 && k <= a.Npmax;
            const bool ok = kvalid && s_tau2[c] == s_tau2[c];
            const bool done = !failed && ok && s_cnt[c] >= k && s_cnt[c] <= a.Cmax;
            a.retry[q] = (kvalid && !done) ? 1 : 0;
            a.cand_count[q] = done ? s_cnt[c] : 0;
            a.rcol[q] = done ? __double2float_rd(tc_collected_radius(s_tau2[c] / s2, a.p, K, s_B)) : CUDART_NAN_F;
            if (a.status) a.status[q] = kvalid ? LAGP_OK : LAGP_EINVAL;
        }
        __syncthreads();
        if (failed) {
            // this CTA's block goes to the exact retry, and whatever blocks it
            // can still take (the others may be failing too)
            for (;;) {
                if (tid == 0) s_blk = atomicAdd(a.counter, 1);
                __syncthreads();
                const int b2 = s_blk;
                __syncthreads();
                if (b2 >= a.nblocks) break;
                for (int c = tid; c < a.nq && (int64_t)b2 * a.nq + c < a.M; c += TC_THREADS) {
                    const int64_t q = a.order.query ? a.order.query[(int64_t)b2 * a.nq + c] : (int64_t)b2 * a.nq + c;
                    const int k = a.Np ? a.Np[q] : a.Npmax;
                    const bool kvalid = k >= 1 && k <= a.Npmax;
                    a.retry[q] = kvalid ? 1 : 0;
                    a.cand_count[q] = 0;
                    a.rcol[q] = CUDART_NAN_F;
                    if (a.status) a.status[q] = kvalid ? LAGP_OK : LAGP_EINVAL;
                }
            }
            break;
        }
    }
    if (tid == 0 && *err) atomicExch(a.err, 1);
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem, TC_TMEM_COLS);
    }
}

}  // namespace

bool knn_tc_supported(int p) { return p >= 1 && tc_k(p) <= 64; }

size_t knn_tc_workspace(int64_t N, int64_t M, int p) {
    const int K = tc_k(p);
    const int64_t Npad = round_up(std::max<int64_t>(N, 1), TC_MROWS);
    return (size_t)(Npad + M) * K * 2 + (size_t)M * 8 + 256;
}

// Design and query operands, the sampled thresholds (tau0, filled by knn_sample
// between the two launches), and the collection pass.  ws: knn_tc_workspace(N, M, p) bytes.
lagp_status launch_knn_tc_prep(lagp_ctx *ctx, void *ws, const void *X, int64_t N, int p, lagp_dtype dtype,
                               const void *Xref, int64_t M, const unsigned long long *kmax,
                               const unsigned long long *kmin, const KnnOrder &order, float **tau0, float **rcol) {
    const int K = tc_k(p);
    const int64_t Npad = round_up(std::max<int64_t>(N, 1), TC_MROWS);
    __half *A = static_cast<__half *>(ws);
    __half *Q = A + Npad * K;
    *tau0 = reinterpret_cast<float *>(Q + M * K);
    *rcol = *tau0 + M;
    knn_tc_prep<<<ctx->num_sms * 4, 128, 0, ctx->stream>>>(X, N, Npad, Xref, M, p, dtype, kmax, kmin, order, A, Q);
    ctx->launches++;
    return lagp_cuda_check(ctx, cudaGetLastError(), "knn_tc_prep");
}

lagp_status launch_knn_tc_collect(lagp_ctx *ctx, void *ws, int64_t N, int p, const void *Xref, lagp_dtype dtype,
                                  int64_t M, const int32_t *Np, int32_t Npmax, const unsigned long long *kmax,
                                  const unsigned long long *kmin, const KnnOrder &order, int32_t *cand, int32_t Cmax,
                                  int32_t *cand_count, int32_t *status, int32_t *retry, int *err, int *counter,
                                  float *rcol, float *dump) {
    const int K = tc_k(p);
    const int64_t Npad = round_up(std::max<int64_t>(N, 1), TC_MROWS);
    TcArgs a;
    a.A = static_cast<const __half *>(ws);
    a.Q = a.A + Npad * K;
    a.N = N;
    a.M = M;
    a.p = p;
    a.K = K;
    a.nmb = (int)(Npad / TC_MROWS);
    a.order = order;
    a.Xref = Xref;
    a.dt = dtype;
    a.counter = counter;
    a.tau0 = reinterpret_cast<const float *>(a.Q + M * K);
    a.rcol = rcol;
    a.Np = Np;
    a.Npmax = Npmax;
    a.kmax = kmax;
    a.kmin = kmin;
    a.cand = cand;
    a.Cmax = Cmax;
    a.cand_count = cand_count;
    a.status = status;
    a.retry = retry;
    a.err = err;
    a.dump = dump;
    a.stall = ctx->knn_tc_stall;
    ctx->knn_tc_stall = 0;
    // blocks: a multiple of the SM count (balanced waves), at most TC_QMAX
    // queries each, taken from a counter (with boxes they cost unevenly)
    const int64_t sms = ctx->num_sms;
    const int64_t nb_min = (M + TC_QMAX - 1) / TC_QMAX;
    const int64_t nb = std::min<int64_t>(M, round_up(nb_min, sms));
    a.nq = (int)((M + nb - 1) / nb);
    a.nblocks = (int)((M + a.nq - 1) / a.nq);
    // as many stages as fit: the CTA then has the SM (and its tensor memory)
    // to itself
    const size_t fixed = (size_t)TC_QMAX * K * 2 + (2 * TC_QMAX + TC_CHUNK / 2) * 4;
    const size_t stage_bytes = (size_t)TC_MROWS * K * 2;
    auto smem_of = [&](int stages) {
        return fixed + TC_EPI_GROUPS * stages * stage_bytes + (TC_EPI_GROUPS * (size_t)stages + 2 * TC_NACC) * 8;
    };
    a.stages = TC_STAGES_MAX;
    while (a.stages > 2 && smem_of(a.stages) + 4096 > ctx->smem_optin) a.stages--;
    size_t smem = smem_of(a.stages);
    if (smem + 4096 > ctx->smem_optin) return lagp_fail(ctx, LAGP_EINVAL, "lagp_knn: tensor-core screen exceeds shared memory");
    // more than half of the SM's shared memory: one CTA per SM, which then
    // holds the whole tensor memory
    smem = std::max(smem, ctx->smem_optin / 2 + 4096);
    LAGP_CUDA(ctx, cudaFuncSetAttribute(knn_screen_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int grid = (int)std::min<int64_t>(a.nblocks, sms);
    knn_screen_tc<<<grid, TC_THREADS, smem, ctx->stream>>>(a);
    ctx->launches++;
    return lagp_cuda_check(ctx, cudaGetLastError(), "knn_screen_tc");
}
