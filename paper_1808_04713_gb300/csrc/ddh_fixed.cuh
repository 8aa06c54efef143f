// FP64-accurate dot products on the integer pipe.
//
// GB300 completes 2 FP64 FMA per SM and clock (0.60 T/s timed) and about 26 integer multiply-adds
// 32 x 32 + 64 bits (IMAD.WIDE; timed with both factors changing from one to the next), so a dense product
// whose operands are put on a common power-of-two scale beforehand runs four to five times faster as
// three integer multiply-adds per real product than as one FP64 FMA.
//
// A number v with |v| < 2^e is held as X = round(v 2^(55 - e)), a signed integer of 55 bits, in two
// limbs X = h 2^27 + l, l in [-2^26, 2^26), |h| <= 2^28.  The exponent e is shared: by
// one row of the matrix (fixed when the matrix is laid out) and by one staged vector (its largest
// component, found while it is staged).  A product a x contributes ah xh 2^54 + (ah xl + al xh) 2^27;
// al xl is left out.  Sums of the two kinds are exact in 64 bits, so a result does not depend on the
// order of its terms or on how many threads share a row.
//
// Error against the exact dot product of length K: rounding of both operands (2^-56 of their scales)
// and the omitted al xl (at most 2^-58 of the product of the scales), i.e. about
// 2^-55 sqrt(K) max|a| max|x| -- the size of the FP64 sum's own rounding, 2^-53 of its partial sums.
//
// Infinities and NaN: a row or vector that holds one has exponent 2047 and every result formed with
// it is NaN.  Magnitudes below 2^-1022 count as zero.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ddh {

constexpr int kFxBits = 55, kFxLow = 27;
// complex terms (two products per component) that a thread may add before it flushes: each high
// product is at most 2^56
constexpr int kFxChain = 63;

// biased exponent field; |v| < 2^(field - 1022)
__device__ __forceinline__ int fx_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v as an integer of 55 bits on the scale of exponent field ef >= fx_field(v)
__device__ __forceinline__ long long fx_int(double v, int ef) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int e = (hi >> 20) & 0x7ff;
    long long m = (long long)(((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)lo);
    const int sh = ef - e + (53 - kFxBits);            // 53-bit mantissa to 55 bits, then down the scale
    if (sh > 0) m = sh <= 54 ? (m + (1ll << (sh - 1))) >> sh : 0;
    else m <<= -sh;
    if (e == 0 || ef == 0x7ff) m = 0;
    return hi < 0 ? -m : m;
}
__device__ __forceinline__ void fx_split(long long X, int& h, int& l) {
    l = ((int)X << (32 - kFxLow)) >> (32 - kFxLow);
    h = (int)((X - l) >> kFxLow);
}
// complex value in four limbs (re h, re l, im h, im l)
__device__ __forceinline__ int4 fx_cpx(double x, double y, int ef) {
    int4 r;
    fx_split(fx_int(x, ef), r.x, r.y);
    fx_split(fx_int(y, ef), r.z, r.w);
    return r;
}

struct FxAcc {
    long long h, l;
};
__device__ __forceinline__ void fx_mac(FxAcc& s, int ah, int al, int xh, int xl) {
    s.h += (long long)ah * xh;
    s.l += (long long)ah * xl;
    s.l += (long long)al * xh;
}
// (re, im) += a x, complex; nah, nal = the negated imaginary limbs of a
__device__ __forceinline__ void fx_cmac(FxAcc& re, FxAcc& im, const int4& a, int nah, int nal, const int4& x) {
    fx_mac(re, a.x, a.y, x.x, x.y);
    fx_mac(im, a.x, a.y, x.z, x.w);
    fx_mac(re, nah, nal, x.z, x.w);
    fx_mac(im, a.z, a.w, x.x, x.y);
}

// A sum over chains and lanes is a pair (h, l): h 2^8 + l 2^-16 in units of 2^54.
// Adds the sums of at most kFxChain complex terms to (h, l) and clears them: the low one is carried
// into the high one, and the result split so that up to 256 of them can be added (what is dropped
// lies 2^-70 below the product of the scales).
__device__ __forceinline__ void fx_flush(FxAcc& s, long long& h, unsigned& l) {
    const long long t = s.h + (s.l >> kFxLow);
    h += t >> 8;
    l += ((unsigned)(t & 255) << 16) | (unsigned)((int)(s.l & ((1ll << kFxLow) - 1)) >> (kFxLow - 16));
    s.h = s.l = 0;
}
// 2^s, -1022 <= s <= 1023
__device__ __forceinline__ double fx_pow2(int s) { return __longlong_as_double((long long)(1023 + s) << 52); }
// d 2^s; results below 2^-1022 become zero.  On the 64-bit pattern: written on its two 32-bit halves
// (__double2hiint, __hiloint2double) the build lost the low half of one of two sums in k_gemv_fx, an
// error of 2^-21.
__device__ __forceinline__ double fx_scale(double d, int s) {
    const long long b = __double_as_longlong(d);
    const int e = (int)(b >> 52) & 0x7ff, t = e + s;
    long long r = b + ((long long)s << 52);
    if (t <= 0) r = 0;
    if (t >= 0x7ff) r = (b & (1ll << 63)) | (0x7ffll << 52);
    if (e == 0 || e == 0x7ff) r = b;                   // zero, infinity, NaN
    return __longlong_as_double(r);
}
// Column scaling: a column whose largest entry has exponent field c is divided by 2^(c - 1023) before the
// rows get their exponents, and the vector's entry multiplied by it (exactly) before it is staged.  The
// error of a sum then goes with the largest |a_ij x_j| and not with max |a| max |x|.
__device__ __forceinline__ int fx_even(int c) { return c == 0 || c == 0x7ff ? 0 : c - 1023; }

// The sum (h + l 2^-24) 2^62 on the scales of exponent fields ea (matrix row) and ex (vector)
__device__ __forceinline__ double fx_value(long long h, unsigned l, int ea, int ex) {
    if (ea == 0x7ff || ex == 0x7ff) return __longlong_as_double(0x7ff8000000000000ll);
    h += l >> 24;
    l &= (1u << 24) - 1;
    int k = __clzll(h ^ (h >> 63)) - 1;                // headroom of h
    k = k < 24 ? k : 24;
    const long long v = (h << k) + (l >> (24 - k));
    const int s = 2 * kFxLow + 8 - k + ea + ex - 2044 - 2 * kFxBits, a = max(min(s, 1000), -1000);
    const double d = __dmul_rn(__ll2double_rn(v), fx_pow2(a));
    return s == a ? d : __dmul_rn(d, fx_pow2(max(s - a, -1000)));
}

// A sum with its al xl products kept, s + ll, split in two FP64 numbers that hold it to 2^-96 of the
// product of the scales: the sum is (hi + lo) 2^e with e = fx_exact_exp(ea, ex).
__device__ __forceinline__ void fx_exact(const FxAcc& s, long long ll, double& hi, double& lo) {
    const long long mask = (1ll << kFxLow) - 1;
    long long l = s.l + (ll >> kFxLow), h = s.h + (l >> kFxLow);
    l &= mask;
    ll &= mask;
    hi = (double)(h & ~1023ll);                        // at most 53 bits
    lo = (double)(((h & 1023) << 42) | (l << 15) | (ll >> 12)) * 0x1p-42;
}
__device__ __forceinline__ int fx_exact_exp(int ea, int ex) { return 2 * kFxLow + ea + ex - 2044 - 2 * kFxBits; }

// the larger |hi word| of a complex number: its exponent field above bit 20
__device__ __forceinline__ unsigned fx_mag(const double2& v) {
    const unsigned a = (unsigned)__double2hiint(v.x) & 0x7fffffffu, b = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
    return a > b ? a : b;
}

}  // namespace ddh
