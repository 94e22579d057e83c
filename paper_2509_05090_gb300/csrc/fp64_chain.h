// Short chains for the latency-bound FP64 kernels (QR, corner spectrum).
//
// An SM sub-partition of GB300 finishes one FP64 warp instruction per 64 cycles whether or
// not the next one depends on it (measured: one chain of FMAs 65 cycles per step, two
// interleaved 129, four 257), its FP64 square root takes ~600 and its division ~565.  What
// counts on a serial path is therefore the number of FP64 warp instructions, including
// conversions from and to FP64, and integer instructions (4 to 5 cycles) are nearly free
// beside them.  The scalars of a Householder reflector -- a square root and a division, the
// longest part of every column -- are formed in 64-bit fixed point instead: one third-order
// iteration (Halley's for 1/sqrt, the geometric series for 1/x) from an FP32 seed each.
#pragma once

#include <cuda_runtime.h>

struct HouseholderScalars {
    double nrm, beta;   // |x| and 1 / (|x| (|x| + |x_0|))
};

namespace fp64_chain {
typedef unsigned long long u64;
typedef long long i64;

// a float in (2^-8, 2) as Q63 fixed point, and the float of a Q61 value in [0, 8) (24 bits kept)
__device__ __forceinline__ u64 q63_of_float(float f)
{
    const unsigned b = __float_as_uint(f);
    return (u64)((b & 0x7FFFFFu) | 0x800000u) << (40 + (int)(b >> 23) - 127);
}
// t0 (1 + c) for a Q63 t0 and a small signed Q59 c
__device__ __forceinline__ u64 q63_correct(u64 t0, i64 c)
{
    return t0 + (u64)(__mul64hi((i64)(t0 >> 1), c << 4) << 2);
}
__device__ __forceinline__ i64 q59_square(i64 h) { return ((h >> 8) * (h >> 8)) >> 43; }   // |h| < 2^39
}  // namespace fp64_chain

// s = |x|^2 > 0 and x0 = |x_0| <= |x| (up to rounding).  The seeds are accurate to ~2^-21, an
// iteration cubes that, and the fixed-point values carry 57 bits or more: both results are
// within one ulp.  ~1160 -> 590 cycles against sqrt and division.
__device__ __forceinline__ HouseholderScalars householder_scalars(double s, double x0)
{
    using namespace fp64_chain;
    const int hs = __double2hiint(s), ex = (hs >> 20) & 0x7FF;
    // outside the range where the exponent arithmetic below is exact (tiny and huge sums,
    // infinities, NaN): the plain functions
    if (ex < 64 || ex > 1982) {
        const double nrm = sqrt(s);
        return {nrm, 1.0 / (nrm * (nrm + x0))};
    }
    const int k = (ex - 1023) >> 1, odd = (ex - 1023) & 1;   // s = S 2^(2k), S in [1, 4)
    const u64 ms = ((u64)__double_as_longlong(s) & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);
    const u64 S = ms << (9 + odd);                           // Q61
    const u64 bx = (u64)__double_as_longlong(x0);
    const int sx = k - ((int)(bx >> 52) - 1023);             // x0 = mant 2^-52 2^(k - sx), sx >= 0
    const u64 mx = ((bx & 0xFFFFFFFFFFFFFULL) | (1ULL << 52)) << 10;
    const u64 X = sx >= 62 ? 0 : (sx < 0 ? mx : (mx >> 1) >> sx);   // |x_0| 2^-k in Q61
    const float Sf = __uint_as_float((unsigned)((127 + odd) << 23) | (unsigned)((ms >> 29) & 0x7FFFFFu));
    const float Xf = (float)(unsigned)(X >> 32) * 0x1p-29f;
    const float yf = rsqrtf(Sf), rf = __fdividef(1.0f, fmaf(Sf * yf, Xf, Sf));
    const u64 y0 = q63_of_float(yf), r0 = q63_of_float(rf);
    // y = 1/sqrt(S): h = 1 - S y0^2, y = y0 (1 + h/2 + 3/8 h^2)
    const i64 h = (i64)((1ULL << 59) - __umul64hi(S, __umul64hi(y0, y0)));
    const u64 y = q63_correct(y0, (h >> 1) + ((3 * q59_square(h)) >> 3));
    const u64 N = __umul64hi(S, y);                          // |x| 2^-k in Q60, [1, 2)
    const u64 D = (S >> 1) + __umul64hi(N << 3, X);          // |x| (|x| + |x_0|) 2^(-2k) in Q60
    // r = 1/D: e = 1 - D r0, r = r0 (1 + e + e^2)
    const i64 e = (i64)((1ULL << 59) - __umul64hi(D, r0));
    const u64 r = q63_correct(r0, e + q59_square(e));
    const u64 mn = (N + 128) >> 8;                           // 53 bits, 2^52 <= mn <= 2^53
    const int lz = __clzll((i64)r);
    const u64 rn = r << lz, mr = (rn >> 11) + ((rn >> 10) & 1);
    return {__longlong_as_double((i64)(((u64)(1022 + k) << 52) + mn)),
            __longlong_as_double((i64)(((u64)(1022 - lz - 2 * k) << 52) + mr))};
}

// The sum of a value per lane, the same in every lane: block floating point on the largest
// exponent (58 bits kept of the largest, so the rounding is finer than that of FP64 additions),
// three integer reductions, one rounding.  ~520 -> 344 cycles against five shuffle-and-add
// levels.  All lanes of the warp call it.
__device__ __forceinline__ double warp_sum(double v)
{
    using namespace fp64_chain;
    const u64 b = (u64)__double_as_longlong(v);
    const int ex = (int)(b >> 52) & 0x7FF;
    const int top = (int)__reduce_max_sync(0xffffffffu, (unsigned)ex);
    if (top < 64 || top == 0x7FF) {   // near the bottom of the range, or not finite
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    const int sh = top - ex;
    const u64 mag = ex == 0 || sh > 57 ? 0 : (((b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52)) << 5) >> sh;
    const i64 f = (i64)b < 0 ? -(i64)mag : (i64)mag;
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)(f & 0x1FFFFF));
    const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)((f >> 21) & 0x1FFFFF));
    const int hi = __reduce_add_sync(0xffffffffu, (int)(f >> 42));
    const i64 t = ((i64)hi << 42) + ((i64)mid << 21) + (i64)lo;   // |t| < 2^63, in units of 2^(top - 1080)
    const u64 a = t < 0 ? (u64)-t : (u64)t;
    const int lz = __clzll((i64)a);
    const u64 n = a << lz, m = (n >> 11) + ((n >> 10) & 1);       // 53 bits
    const u64 r = ((u64)(top + 5 - lz) << 52) + m;                // exponent field top - 1080 + 63 - lz + 1023 - 1
    if (a == 0 || top + 5 - lz <= 0) return 0.0;
    return __longlong_as_double((i64)(r | (t < 0 ? 1ULL << 63 : 0)));
}
