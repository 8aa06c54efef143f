// FP64-accurate dot products on the integer and FP32 pipes.
//
// GB300 completes 2 FP64 FMA per SM and clock (0.60 T/s timed), about 26 integer multiply-adds
// 32 x 32 + 64 bits (IMAD.WIDE; timed with both factors changing from one to the next) and 128 FP32 FMA.  A
// real product is formed here as three integer multiply-adds and three FP32 FMA.
//
// A number v with |v| < 2^e is held as X = v 2^(52 - e) = h 2^26 + l + f: -2^26 <= h < 2^26, 0 <= l < 2^26,
// 0 <= f < 1.  The exponent e is shared: by one row of the matrix (fixed when the matrix is laid
// out) and by one staged vector (its largest component, found while it is staged).  A matrix is kept in this
// form (24 bytes an entry, or packed in 16) beside its complex128 one.  Then
//   a x = ah xh 2^52 + (ah xl + al xh) 2^26 + [ (ah xf + af xh) 2^26 + al xl ] + (al xf + af xl + af xf)
// and the last part is below 2^-25 of the bracket's bound (af xf is kept where ah = 0, so that nothing is left
// of a product only where a factor is zero).
// The first two kinds are summed in 64-bit integers, without error; the bracket in FP32.  The bracket is at most
// 2^-51 of the scale 2^(ea + ex) of a row and a vector, whatever the size of the term itself, and FP32
// rounds each of its additions, so a sum comes out to 2^-72 (30 terms) to 2^-69 (255) of the scale.
//
// FP64 has 2^-53 of P = sum |a x| (of the products in the same component).  P can lie far below the scale: the
// large entries of a row may meet small ones of the vector.  So a component is kept where P >= 2^-16 of
// the scale, which makes it as accurate as the FP64 sum, and formed again in FP64 from the complex128 data
// elsewhere, and wherever a row or vector holds an infinity or a NaN, or nothing above 2^-895.  |sum| >=
// 2^-16 of the scale settles that for nearly all components (fx_value); for the rest fx_again forms P.
// (Splitting operands on a common exponent, so that partial products add without error, is the idea of
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication", 2012.)
//
// Everything here but fx_again compiles for the host as well, where ddh_fixed_dot calls it.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#ifndef __CUDA_ARCH__
#include <string.h>
#endif

namespace ddh {

#define DDH_FX __host__ __device__ __forceinline__

constexpr int kFxBits = 52, kFxLow = 26;
// complex terms that a thread may add before it flushes: each adds at most 2^54 to either integer sum
constexpr int kFxChain = 255;
// flushes that a sum may collect, over all its lanes
constexpr int kFxFlushes = 255;

DDH_FX unsigned long long fx_bits(double v) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long b;
    memcpy(&b, &v, 8);
    return b;
#endif
}
DDH_FX double fx_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    memcpy(&v, &b, 8);
    return v;
#endif
}
// the low word of (hi:lo) >> (s mod 32)
DDH_FX unsigned fx_funnel(unsigned lo, unsigned hi, unsigned s) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, s);
#else
    return (unsigned)((((unsigned long long)hi << 32) | lo) >> (s & 31));
#endif
}

// the high word of |v|: its exponent field above bit 20.  The shared exponent of a row or vector is
// fx_exp of the largest: the field e with |v| < 2^(e - 1022), or 2047 where the fixed form does not serve
// (infinities, NaN, and magnitudes so small that entries below 2^-1022, which the split takes for zero,
// could count)
DDH_FX unsigned fx_mag(double v) { return (unsigned)(fx_bits(v) >> 32) & 0x7fffffffu; }
DDH_FX unsigned fx_mag(const double2& v) {
    const unsigned a = fx_mag(v.x), b = fx_mag(v.y);
    return a > b ? a : b;
}
DDH_FX int fx_exp(unsigned mag) { return mag && mag < (128u << 20) ? 0x7ff : (int)(mag >> 20); }

// one component, split
struct FxNum {
    int h, l;
    float f;                             // f 2^26
};
DDH_FX FxNum fx_split(double v, int ef) {
    const unsigned long long b = fx_bits(v);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const int e = (int)((hi >> 20) & 0x7ff), n = ef - e + 1;
    // the mantissa at the top of (w1, w0), moved down by n bits (one for the sign) in (b1, b0, bm)
    const unsigned w1 = fx_funnel(lo, (hi & 0xfffff) | 0x100000, 21), w0 = lo << 11;
    unsigned b1, b0, bm;
    if (n < 32) {
        b1 = w1 >> n;
        b0 = fx_funnel(w0, w1, n);
        bm = fx_funnel(0, w0, n);
    } else {
        const bool far = n >= 64;
        b1 = 0;
        b0 = far ? 0 : w1 >> (n & 31);
        bm = far ? (n >= 96 ? 0 : w1 >> (n & 31)) : fx_funnel(w0, w1, n);
    }
    // the ones' complement of a negative number: off by 2^-85 of the scale
    const unsigned s = (unsigned)((int)hi >> 31);
    b1 ^= s; b0 ^= s; bm ^= s;
    FxNum r;
    r.h = (int)b1 >> 5;
    r.l = (int)(fx_funnel(b0, b1, 11) & ((1u << kFxLow) - 1));
    // the last of 32 bits is set in every number but zero: a product is zero only where a factor is
    r.f = (float)(fx_funnel(bm, b0, 11) | 1) * 0x1p-6f;
    if (e == 0) { r.h = r.l = 0; r.f = 0.f; }
    return r;
}

// two FP32 numbers and fused multiply-adds of both (one instruction on the device)
struct FxPair {
    unsigned long long v;
};
DDH_FX unsigned fx_word(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned u;
    memcpy(&u, &x, 4);
    return u;
#endif
}
DDH_FX float fx_float(unsigned u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x;
    memcpy(&x, &u, 4);
    return x;
#endif
}
DDH_FX FxPair fx_pair(float x, float y) { return {(unsigned long long)fx_word(y) << 32 | fx_word(x)}; }
DDH_FX float fx_first(FxPair p) { return fx_float((unsigned)p.v); }
DDH_FX float fx_second(FxPair p) { return fx_float((unsigned)(p.v >> 32)); }
DDH_FX void fx_fma2(FxPair& c, FxPair a, FxPair b) {
#ifdef __CUDA_ARCH__
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c.v) : "l"(a.v), "l"(b.v));
#else
    c = fx_pair(fmaf(fx_first(a), fx_first(b), fx_first(c)), fmaf(fx_second(a), fx_second(b), fx_second(c)));
#endif
}

// a staged vector entry: limbs (re h, re l, im h, im l), fractions and high limbs in FP32
struct FxVec {
    int4 i;
    float4 f;
};
DDH_FX FxVec fx_vec(const double2& v, int ef) {
    const FxNum a = fx_split(v.x, ef), b = fx_split(v.y, ef);
    FxVec r;
    r.i.x = a.h; r.i.y = a.l; r.i.z = b.h; r.i.w = b.l;
    r.f.x = a.f; r.f.y = b.f; r.f.z = (float)a.h; r.f.w = (float)b.h;
    return r;
}
// A matrix is laid out split (limbs in .i, fractions in .f; fx_put), beside its complex128 form.  An entry in
// registers: limbs; in FP32, twice each, h (with f where h is zero, so that a product leaves a trace), l and f
struct FxMat {
    int4* i = nullptr;
    float2* f = nullptr;
    DDH_FX FxMat at(int64_t k) const { return {i + k, f + k}; }
};
struct FxRealMat {
    int2* i = nullptr;
    float* f = nullptr;
    DDH_FX FxRealMat at(int64_t k) const { return {i + k, f + k}; }
};
DDH_FX void fx_put(const FxMat& m, int64_t k, const double2& v, int ef) {
    const FxNum a = fx_split(v.x, ef), b = fx_split(v.y, ef);
    int4 i;
    i.x = a.h; i.y = a.l; i.z = b.h; i.w = b.l;
    m.i[k] = i;
    m.f[k] = make_float2(a.f, b.f);
}
DDH_FX void fx_put(const FxRealMat& m, int64_t k, double v, int ef) {
    const FxNum a = fx_split(v, ef);
    m.i[k] = make_int2(a.h, a.l);
    m.f[k] = a.f;
}
// The same in 16 bytes, 11 bits of f left: for a matrix that is read faster than its products are formed.  A
// sum comes out to 2^-64 (60 terms) to 2^-63 (255) of the scale, so P must reach 2^-kFxSmallPacked of it.
DDH_FX long long fx_pack(double v, int ef) {
    const FxNum a = fx_split(v, ef);
    const long long f = (long long)(a.f * 0x1p-15f);       // f 2^11, rounded down
    return v != 0.0 ? (((((long long)a.h << kFxLow) + a.l) << 11) + f) | 1 : 0;
}
DDH_FX void fx_unpack(const longlong2& p, int4& i, float2& f) {
    const unsigned xl = (unsigned)p.x, xh = (unsigned)(p.x >> 32), yl = (unsigned)p.y, yh = (unsigned)(p.y >> 32);
    constexpr unsigned mask = (1u << kFxLow) - 1;
    i.x = (int)xh >> 5;
    i.y = (int)(fx_funnel(xl, xh, 11) & mask);
    i.z = (int)yh >> 5;
    i.w = (int)(fx_funnel(yl, yh, 11) & mask);
    f = make_float2((float)(int)(xl & 2047) * 0x1p15f, (float)(int)(yl & 2047) * 0x1p15f);
}
struct FxReal {
    int h, l;
    FxPair fh, fl, f;
};
DDH_FX FxReal fx_real(int h_, int l_, float f_) {
    FxReal r;
    r.h = h_;
    r.l = l_;
    const float h = (float)h_ + f_ * 0x1p-52f, l = (float)l_;
    r.fh = fx_pair(h, h);
    r.fl = fx_pair(l, l);
    r.f = fx_pair(f_, f_);
    return r;
}
struct FxEntry {
    FxReal x, y;
    int nh, nl;
};
DDH_FX FxEntry fx_entry(const int4& i, const float2& f) {
    FxEntry r;
    r.x = fx_real(i.x, i.y, f.x);
    r.y = fx_real(i.z, i.w, f.y);
    r.nh = -i.z;
    r.nl = -i.w;
    return r;
}

// a lane's complex sum of at most kFxChain terms: rh 2^52 + rl 2^26 + c1.x - c2.y, ih 2^52 + il 2^26 + c1.y + c2.x
struct FxSum {
    long long rh, rl, ih, il;
    FxPair c1, c2;
};
DDH_FX void fx_clear(FxSum& s) {
    s.rh = s.rl = s.ih = s.il = 0;
    s.c1.v = s.c2.v = 0;
}
DDH_FX void fx_imac(long long& h, long long& l, int ah, int al, int xh, int xl) {
    h += (long long)ah * xh;
    l += (long long)ah * xl;
    l += (long long)al * xh;
}
// s += a x: complex, and real times complex
DDH_FX void fx_mac(FxSum& s, const FxEntry& a, const int4& x, const float4& xf) {
    fx_imac(s.rh, s.rl, a.x.h, a.x.l, x.x, x.y);
    fx_imac(s.ih, s.il, a.x.h, a.x.l, x.z, x.w);
    fx_imac(s.rh, s.rl, a.nh, a.nl, x.z, x.w);
    fx_imac(s.ih, s.il, a.y.h, a.y.l, x.x, x.y);
    const FxPair f = fx_pair(xf.x, xf.y), h = fx_pair(xf.z, xf.w), l = fx_pair((float)x.y, (float)x.w);
    fx_fma2(s.c1, a.x.fh, f);
    fx_fma2(s.c2, a.y.fh, f);
    fx_fma2(s.c1, a.x.f, h);
    fx_fma2(s.c2, a.y.f, h);
    fx_fma2(s.c1, a.x.fl, l);
    fx_fma2(s.c2, a.y.fl, l);
}
DDH_FX void fx_mac(FxSum& s, const FxReal& a, const int4& x, const float4& xf) {
    fx_imac(s.rh, s.rl, a.h, a.l, x.x, x.y);
    fx_imac(s.ih, s.il, a.h, a.l, x.z, x.w);
    fx_fma2(s.c1, a.fh, fx_pair(xf.x, xf.y));
    fx_fma2(s.c1, a.f, fx_pair(xf.z, xf.w));
    fx_fma2(s.c1, a.fl, fx_pair((float)x.y, (float)x.w));
}

// Sums over chains and lanes are pairs (h, l): h 2^60 + l 2^24, with the number of flushes that held anything
// but zero above bit 50 of l, so that a sum of nothing but zeros is told from one that cancels.
// Adds component c of a lane's sum to (h, l).
DDH_FX void fx_flush(const FxSum& s, int c, long long& h, long long& l) {
    const long long sh = c ? s.ih : s.rh, sl = c ? s.il : s.rl, t = sh + (sl >> kFxLow);
    const float p = c ? fx_second(s.c1) : fx_first(s.c1), q = c ? fx_first(s.c2) : fx_second(s.c2);
    h += t >> 8;
    l += ((t & 255) << 28) + ((sl & ((1ll << kFxLow) - 1)) << 2) + (long long)rintf((c ? p + q : p - q) * 0x1p-24f);
    if (p != 0.f || q != 0.f || sl != 0) l += 1ll << 50;
}
// 2^-kFxSmall of the scale: results and weights below it (of a packed matrix 2^-kFxSmallPacked)
constexpr int kFxSmall = 16, kFxSmallPacked = 10;
// The value of a sum on the scales of exponents ea (matrix row) and ex (vector).  False: it is small, or
// not a number (fx_again decides what it is to be).
DDH_FX bool fx_carry(long long& h, long long& l, int ea, int ex, int bits) {
    const long long any = (l + (1ll << 49)) >> 50;
    l -= any << 50;
    h += l >> 36;
    l &= (1ll << 36) - 1;
    const long long small = 1ll << (2 * kFxBits - 60 - bits);                     // the scale is 2^104, h counts 2^60
    return ea != 0x7ff && ex != 0x7ff && (any == 0 || h >= small || h < -small);
}
DDH_FX double fx_pow2(int s) { return fx_double((unsigned long long)(1023 + s) << 52); }       // -1022 <= s <= 1023
DDH_FX double fx_ldexp(double d, int s) {
    const int a = s > 1000 ? 1000 : (s < -1000 ? -1000 : s), r = s - a;
    d *= fx_pow2(a);
    return r ? d * fx_pow2(r > 1000 ? 1000 : (r < -1000 ? -1000 : r)) : d;
}
DDH_FX int fx_scale_exp(int ea, int ex) { return ea + ex - 2044 - 2 * kFxBits; }                // of a unit of the sum
DDH_FX bool fx_value(long long h, long long l, int ea, int ex, double& v, int bits = kFxSmall) {
    const bool ok = fx_carry(h, l, ea, ex, bits);
    const unsigned long long m = (unsigned long long)(h ^ (h >> 63));
#ifdef __CUDA_ARCH__
    int k = __clzll((long long)m) - 1;                     // headroom of h
#else
    int k = m ? __builtin_clzll(m) - 1 : 63;
#endif
    k = k < 36 ? k : 36;
    v = fx_ldexp((double)((long long)((unsigned long long)h << k) + (l >> (36 - k))), 60 - k + fx_scale_exp(ea, ex));
    return ok;
}
// the same as hi + lo, each of at most 53 bits
DDH_FX bool fx_value2(long long h, long long l, int ea, int ex, double& hi, double& lo) {
    const bool ok = fx_carry(h, l, ea, ex, kFxSmall);
    hi = fx_ldexp((double)(h & ~2047ll), 60 + fx_scale_exp(ea, ex));
    lo = fx_ldexp((double)(((h & 2047) << 36) | l), 24 + fx_scale_exp(ea, ex));
    return ok;
}
// P of both components in units of the scale, from the high limbs (and so from below): w += the term's
struct FxWeight {
    float x, y;
};
DDH_FX void fx_weigh(FxWeight& w, int ah, int bh, const int4& x) {
    const float ax = fabsf((float)ah), ay = fabsf((float)bh), xx = fabsf((float)x.x), xy = fabsf((float)x.z);
    w.x += ax * xx + ay * xy;
    w.y += ax * xy + ay * xx;
}
DDH_FX bool fx_heavy(float w, int bits) { return w >= (float)(1ll << (2 * kFxLow - bits)); }  // the scale is 2^52

#ifdef __CUDACC__
// What is to become of the components that fx_value turned down, of one row and one vector, by the G lanes
// that share the row (a power of two; G > 1: every lane of the warp calls).  bad: this lane's, bit 0 real, bit
// 1 imaginary.  a(j), x(j): entries; ah(j), xi(j): the high limbs of a (real, imaginary), the limbs of x.  Returns which of the group's stay as they
// are; d holds the FP64 sums for the others.
template <class FA, class FH, class FI, class FX>
__device__ __noinline__ unsigned fx_again(int G, unsigned bad, int n, int ea, int ex, const FA& a, const FH& ah, const FI& xi,
                                          const FX& x, double2& d, int bits = kFxSmall) {
    const int j0 = threadIdx.x & (G - 1);
    for (int o = G >> 1; o > 0; o >>= 1) bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    FxWeight w = {0.f, 0.f};
    if (bad && ea != 0x7ff && ex != 0x7ff)
#pragma unroll 4
        for (int j = j0; j < n; j += G) {
            const int2 u = ah(j);
            fx_weigh(w, u.x, u.y, xi(j));
        }
    for (int o = G >> 1; o > 0; o >>= 1) {
        w.x += __shfl_xor_sync(0xffffffffu, w.x, o);
        w.y += __shfl_xor_sync(0xffffffffu, w.y, o);
    }
    const unsigned keep = (fx_heavy(w.x, bits) ? 1 : 0) | (fx_heavy(w.y, bits) ? 2 : 0);
    const bool need = (bad & ~keep) != 0;
    if (G > 1 ? !__any_sync(0xffffffffu, need) : !need) return keep;
    double sx = 0, sy = 0;
    if (need)
#pragma unroll 4
        for (int j = j0; j < n; j += G) {
            const double2 u = a(j), v = x(j);
            sx = fma(u.x, v.x, fma(-u.y, v.y, sx));
            sy = fma(u.x, v.y, fma(u.y, v.x, sy));
        }
    for (int o = G >> 1; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    d = make_double2(sx, sy);
    return keep;
}
#endif

}  // namespace ddh
