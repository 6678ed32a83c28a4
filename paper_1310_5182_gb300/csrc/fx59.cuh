// 64-bit fixed point on the integer pipe, for the small Cholesky factors of
// local correlation matrices.
//
// A value x, |x| < 4, is held as an integer v = x 2^59 (64 bits).  For the
// inner products v is cut into two signed limbs, v = h 2^30 + l with |l| <=
// 2^29, and the product of two values is
//     x y 2^59 = 2 h h' + (h l' + l h') 2^-29 + l l' 2^-59,
// three 32 x 32 -> 64 bit multiply-adds with the last term (below 2^-1 units
// of 2^-59) left out; |x|, |c| < 2 where a high limb is doubled.
//
// Why it is there: this GPU's FP64 unit takes a warp instruction every 64
// cycles of a sub-partition, whatever its lanes; the integer pipe takes a
// 32 x 32 -> 64 multiply-add every 4 (both measured), so a product costs
// about 12 cycles instead of 64.  Why it is exact enough: a correlation
// matrix with nugget g < 1 has a diagonal of 1 + g < 2, so the rows of its
// factor have norm < sqrt(2) and every entry and every inner product is of
// order one; a fixed 2^-59 is then finer than FP64's rounding of those sums
// (2^-53 of the partial sums).  Where it is not: whatever is small as a whole
// (means, criteria and derivatives far below the entries that they are made
// of).  Each kernel says which of those it leaves to FP64.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

constexpr int FX_FRAC = 59;
constexpr long long FX_ONE = 1ll << FX_FRAC;

struct Fx {
    int h, l;
};

__device__ __forceinline__ Fx fx_split(long long v) {
    Fx f;
    f.l = (int)((unsigned)v << 2) >> 2;        // the low 30 bits, signed
    f.h = (int)((v + (1ll << 29)) >> 30);      // v = h 2^30 + l
    return f;
}

__device__ __forceinline__ long long fx_join(Fx f) { return ((long long)f.h << 30) + f.l; }

// c + a b.  In PTX: the compiler takes the same C expression apart into
// products and 64-bit additions, twice the instructions (18 of them in a row:
// 78 cycles a warp against 40).
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// Sums of products start from FX_HALF, take fx_mid of every product, are
// shifted once (fx_sum adds that to `base`), and end with fx_hi of every
// product: base + sum x c.  Three multiply-adds a product and one shift a sum.
constexpr long long FX_HALF = 1ll << 28;
__device__ __forceinline__ long long fx_mid(long long mid, Fx x, Fx c) {
    return fx_mad(x.l, c.h, fx_mad(x.h, c.l, mid));
}
__device__ __forceinline__ long long fx_sum(long long base, long long mid) { return base + (mid >> 29); }
__device__ __forceinline__ long long fx_hi(long long sum, Fx x, Fx c) { return fx_mad(x.h, 2 * c.h, sum); }

// Range of the middle sum: a product adds up to (|x| + |c|) 2^58 to it, and it
// wraps at 2^63.  Where nothing bounds the norms of both factors, what is above
// its low bits moves to the high sum now and then (exact); hi is doubled at the
// end where it is a sum of h h' alone.
__device__ __forceinline__ void fx_fold_half(long long &hi, long long &mid) {
    hi += mid >> 30;
    mid &= (1ll << 30) - 1;
}
__device__ __forceinline__ void fx_fold(long long &sum, long long &mid) {
    sum += mid >> 29;
    mid &= (1ll << 29) - 1;
}

__device__ __forceinline__ long long fx_mul(Fx a, Fx b) { return fx_hi(fx_mid(FX_HALF, a, b) >> 29, a, b); }

__device__ __forceinline__ Fx fx_neg(Fx a) { return Fx{-a.h, -a.l}; }
__device__ __forceinline__ Fx fx_twice(Fx a) { return Fx{2 * a.h, 2 * a.l}; }

// Nonzero unless |v| < 2^(32 + k).
__device__ __forceinline__ unsigned fx_beyond(long long v, int k) {
    return (unsigned)((int)(v >> 32) + (1 << k)) >> (k + 1);
}

// x 2^59 rounded to nearest, |x| < 4, on the integer pipe.
__device__ __forceinline__ long long fx_from(double x) {
    const int hi = __double2hiint(x);
    const int s = ((hi >> 20) & 0x7ff) - (1075 - FX_FRAC);  // mantissa 2^s
    long long m = ((long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
    if (s >= 0) {
        m <<= s;
    } else {
        const int r = -s < 62 ? -s : 62;
        m = (m + (1ll << (r - 1))) >> r;
    }
    return hi < 0 ? -m : m;
}

// v 2^(e - 59) as a double (one conversion on the FP64 unit).
__device__ __forceinline__ double fx_double(long long v, int e = 0) {
    const double x = (double)v;
    // the power of two by the exponent field (v = 0 stays 0)
    return v == 0 ? 0.0 : __hiloint2double(__double2hiint(x) + ((e - FX_FRAC) << 20), __double2loint(x));
}

// 1 / sqrt(s 2^-59) for 0 < s < 2^60 as y 2^t, y in (0.7, 1.42] (fixed
// point): the hardware's FP32 estimate and one third-order step.  *root
// receives sqrt(s 2^-59).
__device__ __forceinline__ Fx fx_rsqrt(long long s, int *t, long long *root) {
    const int b = 63 - __clzll(s);
    const int sh = (59 - b) >> 1;
    const long long u = s << (2 * sh);  // in [2^58, 2^60)
    const float y0 = rsqrtf((float)(int)(u >> 29) * 0x1p-30f);
    const long long Y = (long long)__float2int_rn(y0 * 0x1p30f) << 29;
    const Fx Yf = fx_split(Y), uf = fx_split(u);
    const Fx Y2 = fx_neg(fx_split(fx_mul(Yf, Yf)));
    const long long e = fx_hi(fx_sum(FX_ONE, fx_mid(FX_HALF, uf, Y2)), uf, Y2);  // 1 - u y0^2
    const Fx ef = fx_split(e);
    const Fx c = fx_split((e >> 1) + ((3 * fx_mul(ef, ef)) >> 3));
    const Fx y = fx_split(fx_hi(fx_sum(Y, fx_mid(FX_HALF, Yf, c)), Yf, c));
    *t = sh;
    *root = fx_mul(uf, y) >> sh;
    return y;
}
