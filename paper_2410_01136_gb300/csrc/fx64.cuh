// fx64.cuh -- FP64 elementary functions evaluated in 64-bit fixed point.
//
// Why: an SM of sm_103a executes 2 FP64 operations per clock (a warp-wide
// FP64 instruction occupies its pipe for 16 clocks) against 64 to 128 integer
// ones, so a function of 10 to 40 FP64 instructions costs 160 to 640 clocks
// of the pipe that bounds the FP64 march.  Here the argument's mantissa is
// taken apart with integer instructions, the reduction and the polynomial run
// on unsigned 64-bit fractions (a product's high half is 3 wide integer
// multiplies and 2 additions), and the result is rounded once to FP64: no
// FP64 instruction at all.  The FP64 march keeps 73 FP64 instructions per
// sample (the grid model; pipe 70 % active, issue 35 %).  Measured against
// CUDA's functions: a map of a 256 x 256 x 64 grid (Nside 64, 512 steps)
// 14.5 -> 4.0 ms, WMAP-type maps and gradient (Nside 16, 128 steps, 2
// frequencies) 1.33 -> 0.58 ms (4.2 and 0.64 ms before the lane count followed),
// at the same error against 64-bit values; CUDA's functions are specified to
// 1 ulp.
//
// Accuracy: 60 to 63 correct bits before the final rounding, i.e. at most 0.53
// ulp of the result, where division and square root round correctly in
// hardware.  Beside a zero of the function:
//  * log, atan2 and sincos (at non-zero multiples of pi/2) keep this relative
//    accuracy with ZEROS (the default), and without it have an absolute error
//    of 2^-60.  The march goes without (10 to 20 integer instructions per call):
//    there these values enter sums, phases and products of order one.  Fields
//    evaluated for the caller take ZEROS, as a component may be nothing but
//    such a value;
//  * the tanh of sech2_tanh and the weights of trilinear_weights have an
//    absolute error of 2^-60 (formed in FP64 from e^-2x and from 1 - f they had
//    2^-53).
// Arguments outside each function's ordinary range (non-normal, huge, zero or
// negative where that is special, NaN) go to the CUDA function.
//
// Method: the polynomials interpolate 2^f, atanh, sin, cos and atan at
// Chebyshev nodes of the reduced range (in 400-bit arithmetic, each coefficient
// cut to its word; the interpolation is off by less than 2^-64 of the result);
// the reciprocal and the reciprocal square root are a 22-bit FP32 seed and one
// Newton-Raphson step with its second-order term.
// Qa.b below: an unsigned 64-bit word whose unit is 2^-b.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define SYNAX_FX_FN __device__ __forceinline__
#else   // plain C++: the same integer arithmetic, for tests on the host
#include <cmath>
#include <cstring>
#define SYNAX_FX_FN static inline
#endif

namespace synax {
namespace fx {

typedef unsigned long long u64;
typedef uint32_t u32;

#ifdef __CUDACC__
SYNAX_FX_FN u64 bits_of(double x) { return (u64)__double_as_longlong(x); }
SYNAX_FX_FN double of_bits(u64 b) { return __longlong_as_double((long long)b); }
SYNAX_FX_FN int clz(u64 v) { return __clzll((long long)v); }
SYNAX_FX_FN u64 mulhi(u64 a, u64 b) { return __umul64hi(a, b); }
// bits of the FP32 approximations of 1/x and 1/sqrt(x), x in [1, 4)
SYNAX_FX_FN u32 rcp_seed(u32 xbits) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(xbits)));
    return __float_as_uint(y);
}
SYNAX_FX_FN u32 rsqrt_seed(u32 xbits) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(xbits)));
    return __float_as_uint(y);
}
#else
SYNAX_FX_FN u64 bits_of(double x) {
    u64 b;
    std::memcpy(&b, &x, 8);
    return b;
}
SYNAX_FX_FN double of_bits(u64 b) {
    double x;
    std::memcpy(&x, &b, 8);
    return x;
}
SYNAX_FX_FN int clz(u64 v) { return v ? __builtin_clzll(v) : 64; }
SYNAX_FX_FN u64 mulhi(u64 a, u64 b) { return (u64)(((unsigned __int128)a * b) >> 64); }
SYNAX_FX_FN u32 rcp_seed(u32 xbits) {
    float x, y;
    std::memcpy(&x, &xbits, 4);
    y = 1.0f / x;
    u32 b;
    std::memcpy(&b, &y, 4);
    return b;
}
SYNAX_FX_FN u32 rsqrt_seed(u32 xbits) {
    float x, y;
    std::memcpy(&x, &xbits, 4);
    y = 1.0f / std::sqrt(x);
    u32 b;
    std::memcpy(&b, &y, 4);
    return b;
}
#endif

SYNAX_FX_FN int biased_exp(u64 b) { return (int)(b >> 52) & 0x7FF; }
// The mantissa as Q1.63, in [1, 2) (0 for zero and subnormals).
SYNAX_FX_FN u64 mantissa(u64 b) { return (b & 0x7FF0000000000000ull) ? (b << 11) | 0x8000000000000000ull : 0ull; }

// High half of a product without the low x low term: too small by less than 3.
SYNAX_FX_FN u64 mh(u64 a, u64 b) {
    const u32 ah = (u32)(a >> 32), al = (u32)a, bh = (u32)(b >> 32), bl = (u32)b;
    return (u64)ah * bh + (((u64)ah * bl) >> 32) + (((u64)al * bh) >> 32);
}

// v 2^k (v unsigned) rounded to FP64, with the given sign bit; flushed to zero
// below the normal range.  The caller keeps the result below 2^1024.
SYNAX_FX_FN double pack(u64 v, int k, u64 sign) {
    const int lz = clz(v);
    const u64 m = v << (lz & 63);
    const u64 r = (m >> 11) + ((m >> 10) & 1);              // 53 bits, carry included
    const int ex = 1023 + 62 + k - lz;                        // biased exponent less one (r carries the leading one)
    const u64 out = ((u64)(u32)ex << 52) + r;
    return of_bits((v == 0 || ex < 0 ? 0ull : out) | sign);
}

// (hi:lo) >> s for s >= 0, returning the low 64 bits and, in top, the next ones.
SYNAX_FX_FN u64 shr128(u64 hi, u64 lo, int s, u64& top) {
    const u64 w0 = s < 64 ? lo : hi, w1 = s < 64 ? hi : 0ull;
    const int t = s & 63;
    top = w1 >> t;
    const u64 r = (w0 >> t) | ((w1 << 1) << (63 - t));
    return s < 128 ? r : 0ull;
}

// 2^f - 1 for f in [0, 1) (Q0.64), Q0.64.
SYNAX_FX_FN u64 exp2m1_core(u64 f) {
    // (2^f - 1) / f; the last sum stays below 2^64 (the coefficients add up to 1 - 2^-61)
    u64 p = 0x000000000214D124ull;
    p = 0x000000001A7C5766ull + mh(p, f);
    p = 0x00000001EBCC1444ull + mh(p, f);
    p = 0x0000001E49A967DFull + mh(p, f);
    p = 0x000001B527AA4152ull + mh(p, f);
    p = 0x0000162C00EAEA04ull + mh(p, f);
    p = 0x0000FFE5FE97CE77ull + mh(p, f);
    p = 0x000A184897AAA791ull + mh(p, f);
    p = 0x005761FF9E2D427Cull + mh(p, f);
    p = 0x0276556DF7497D09ull + mh(p, f);
    p = 0x0E35846B8250637Full + mh(p, f);
    p = 0x3D7F7BFF058B1D3Full + mh(p, f);
    p = 0xB17217F7D1CF79ABull + mh(p, f);
    return mh(p, f);
}
// 2^t for t = n + f 2^-64, as FP64; n within the normal range.
SYNAX_FX_FN double exp2_core(int n, u64 f) {
    const u64 p = exp2m1_core(f);
    return of_bits(((u64)(u32)(n + 1023) << 52) + (p >> 12) + ((p >> 11) & 1));
}

// |x| L 2^ke = n + f 2^-64 for |x| below about 700 (so that n fits), with
// the mantissa of the factor as L1 (Q1.63) and L2 (the next 64 bits).
SYNAX_FX_FN int scaled_split(u64 b, u64 L1, u64 L2, int ke, u64& f) {
    const u64 M = mantissa(b);
    u64 hi = mulhi(M, L1), lo = M * L1;                       // Q2.126
    const u64 c = mh(M, L2);
    lo += c;
    hi += lo < c ? 1 : 0;
    u64 top;
    f = shr128(hi, lo, 62 + 1023 - ke - biased_exp(b), top);
    return (int)top;
}
constexpr u64 kLog2e1 = 0xB8AA3B295C17F0BBull, kLog2e2 = 0xBE87FED0691D3E88ull;   // log2 e
constexpr u64 kLog2e05_1 = 0x93BB62877CDFF3C9ull, kLog2e05_2 = 0x653998A6BA7DCBA0ull;   // 16 (0.05 log2 e)
SYNAX_FX_FN bool exp_in_range(u64 b) { return ((u32)(b >> 32) & 0x7FFFFFFFu) < 0x4085E000u; }   // |x| < 700

// e^x (NATURAL) or 2^x.
template <bool NATURAL>
SYNAX_FX_FN double exp_any(double x) {
    const u64 b = bits_of(x);
    if (!exp_in_range(b)) {
#ifdef __CUDACC__
        return NATURAL ? ::exp(x) : ::exp2(x);
#else
        return NATURAL ? std::exp(x) : std::exp2(x);
#endif
    }
    u64 f;
    int n;
    if (NATURAL) {
        n = scaled_split(b, kLog2e1, kLog2e2, 0, f);
    } else {
        u64 top;
        f = shr128(mantissa(b), 0, 63 + 1023 - biased_exp(b), top);
        n = (int)top;
    }
    if (b >> 63) {                                            // x < 0
        n = f ? -n - 1 : -n;
        f = 0ull - f;
    }
    return exp2_core(n, f);
}
// e^(-x / 20) (FIFTH false) or e^(-x / 5) for x >= 0: the scale of the argument
// joins the constant, so the argument is not rounded.
template <bool FIFTH>
SYNAX_FX_FN double exp_radial(double x) {
    const u64 b = bits_of(x);
    if (!exp_in_range(b) || (b >> 63)) return exp_any<true>(x * (FIFTH ? -0.2 : -0.05));
    u64 f;
    const int n = scaled_split(b, kLog2e05_1, kLog2e05_2, FIFTH ? -2 : -4, f);
    return exp2_core(f ? -n - 1 : -n, 0ull - f);
}

// 1/d for d in [1, 2) as Q1.63: Q1.63 in (1/2, 1], error below 2^-61.
SYNAX_FX_FN u64 rcp_core(u64 D) {
    // 24-bit seed r0 (Q0.32, < 1) from the FP32 reciprocal of the leading bits
    u32 s = rcp_seed(0x3F800000u | (u32)((D << 1) >> 41));
    s = s > 0x3F7FFFFFu ? 0x3F7FFFFFu : s;
    s = s < 0x3F000000u ? 0x3F000000u : s;                  // in [1/2, 1)
    const u32 r0 = (s << 8) | 0x80000000u;
    const u32 Dh = (u32)(D >> 32), Dl = (u32)D;
    // e = 1 - d r0 in units of 2^-63, |e| < 2^42; 1/d = r0 (1 + e + e^2 + ...)
    const long long e = (long long)(0x8000000000000000ull - ((u64)Dh * r0 + (((u64)Dl * r0) >> 32)));
    const int eh = (int)(e >> 12);
    const long long g = e + (((long long)eh * eh) >> 39);
    const long long gh = g >> 32;
    return ((u64)r0 << 31) + (u64)(((long long)r0 * gh + (long long)(((u64)r0 * (u32)g) >> 32)));
}

// a / b
SYNAX_FX_FN double div(double a, double b) {
    const u64 ab = bits_of(a), bb = bits_of(b);
    const int ea = biased_exp(ab), eb = biased_exp(bb), de = ea - eb;
    if (eb == 0 || eb == 0x7FF || ea == 0x7FF || de > 1000 || (ea != 0 && de < -1000) || (ea == 0 && (ab << 1) != 0))
        return a / b;
    return pack(mulhi(mantissa(ab), rcp_core(mantissa(bb))), de - 62, (ab ^ bb) & 0x8000000000000000ull);
}
SYNAX_FX_FN double rcp(double x) {
    const u64 b = bits_of(x);
    const int ex = biased_exp(b);
    if (ex < 2 || ex > 2040) return 1.0 / x;
    return pack(rcp_core(mantissa(b)), 1023 - ex - 63, b & 0x8000000000000000ull);
}

// 1/sqrt(m) for m in [1, 4) as Q2.62: the seed r0 (Q0.32) and the correction
// g (units of 2^-62), 1/sqrt(m) = r0 (1 + g).
SYNAX_FX_FN void rsqrt_core(u64 m, u32& r0, long long& g) {
    const int two = (m >> 63) != 0;                           // m >= 2
    const u32 xb = two ? 0x40000000u | (u32)((m << 1) >> 41) : 0x3F800000u | (u32)((m << 2) >> 41);
    u32 s = rsqrt_seed(xb);
    s = s > 0x3F7FFFFFu ? 0x3F7FFFFFu : s;                  // in [1/2, 1)
    r0 = s < 0x3F000000u ? 0x80000000u : (s << 8) | 0x80000000u;
    const u64 sq = (u64)r0 * r0;                              // r0^2, Q0.64, exact
    const long long h = (long long)(0x4000000000000000ull - mulhi(m, sq));   // 1 - m r0^2, |h| < 2^42
    const int hh = (int)(h >> 12);
    // (1 - h)^(-1/2) = 1 + h/2 + 3 h^2/8 + ...
    g = (h >> 1) + ((3 * (((long long)hh * hh) >> 21)) >> 20);
}
// v (1 + g), g in units of 2^-62
SYNAX_FX_FN u64 mul_1pg(u64 v, long long g) {
    const u64 ag = (u64)(g < 0 ? -g : g) << 20;
    const u64 c = mulhi(v, ag) >> 18;
    return g < 0 ? v - c : v + c;
}
SYNAX_FX_FN double sqrt(double x) {
    const u64 b = bits_of(x);
    const int ex = biased_exp(b);
    if ((b >> 63) || ex == 0 || ex == 0x7FF) {
#ifdef __CUDACC__
        return ::sqrt(x);
#else
        return std::sqrt(x);
#endif
    }
    const int e = ex - 1023, half = e >> 1;                   // floor
    const u64 m = mantissa(b) >> ((e & 1) ? 0 : 1);           // m in [1, 4), Q2.62
    u32 r0;
    long long g;
    rsqrt_core(m, r0, g);
    const u64 z = (u64)(u32)(m >> 32) * r0 + (((u64)(u32)m * r0) >> 32);   // m r0, Q2.62
    return pack(mul_1pg(z, g), half - 62, 0);
}
SYNAX_FX_FN double rsqrt(double x) {
    const u64 b = bits_of(x);
    const int ex = biased_exp(b);
    if ((b >> 63) || ex == 0 || ex == 0x7FF) {
#ifdef __CUDACC__
        return ::rsqrt(x);
#else
        return 1.0 / std::sqrt(x);
#endif
    }
    const int e = ex - 1023, half = e >> 1;
    const u64 m = mantissa(b) >> ((e & 1) ? 0 : 1);
    u32 r0;
    long long g;
    rsqrt_core(m, r0, g);
    return pack(mul_1pg((u64)r0 << 31, g), -half - 63, 0);
}

// log2(m) for m = M in [1, 2): log2(m) = l, or 1 - l with up = 1, so that
// 0 <= l <= 1/2.  Returns 2^lz l as Q2.62: lz normalises |m - 1| (or 2 - m) where
// ZEROS, so that a small l keeps all its bits (else lz = 0).
template <bool ZEROS>
SYNAX_FX_FN u64 log2_core(u64 M, int& up, int& lz) {
    up = M > 0xB504F333F9DE6484ull;                           // m > sqrt 2: log2(m / 2) < 0
    const u64 a = up ? 0ull - M : M - 0x8000000000000000ull;   // |m - 1| or 2 - m, Q1.63
    const u64 D = (M >> 1) + (up ? 0x8000000000000000ull : 0x4000000000000000ull);
    // D is (m + 2)/2 or (m + 1)/2 in [1, 2); s = a / (2 D), Q0.64
    const u64 R = rcp_core(D);
    lz = ZEROS ? clz(a) & 63 : 0;
    const u64 sn = mulhi(a << lz, R) << 1;
    const u64 s = sn >> lz;
    const u64 u = mh(s, s);
    u64 p = 0x0C3EC75D74CD7069ull;                            // (2 / ln 2) atanh(s) / s, Q2.62
    p = 0x0C3BA01CC4BFBA70ull + mh(p, u);
    p = 0x0E3514BCF0189B7Dull + mh(p, u);
    p = 0x10C9A5991B72D86Full + mh(p, u);
    p = 0x1484B14487386E78ull + mh(p, u);
    p = 0x1A61762A7085B953ull + mh(p, u);
    p = 0x24EED8A1DF3F9890ull + mh(p, u);
    p = 0x3D8E13B87407F8C2ull + mh(p, u);
    p = 0xB8AA3B295C17F0BBull + mh(p, u);
    return mh(sn, p);
}
// ln x (NATURAL) or log2 x.
template <bool NATURAL, bool ZEROS = true>
SYNAX_FX_FN double log_any(double x) {
    const u64 b = bits_of(x);
    const int ex = biased_exp(b);
    if ((b >> 63) || ex == 0 || ex == 0x7FF) {
#ifdef __CUDACC__
        return NATURAL ? ::log(x) : ::log2(x);
#else
        return NATURAL ? std::log(x) : std::log2(x);
#endif
    }
    int up, lzl;
    const u64 ln = log2_core<ZEROS>(mantissa(b), up, lzl);
    const int e = ex - 1023 + up;
    // |log2 x| as v 2^k: l alone (2^lzl l, Q2.62), or |e| +- l with as many fraction bits as |e| leaves
    const u32 ae = (u32)(e < 0 ? -e : e);
    const int sh = 64 - clz(ae);
    const u64 ls = (ln >> lzl) >> sh;
    u64 v = ((u64)ae << (62 - sh)) + ((e < 0) == (up != 0) ? ls : 0ull - ls);
    v = ae == 0 ? ln : v;
    const u64 sign = (ae == 0 ? up != 0 : e < 0) ? 0x8000000000000000ull : 0ull;
    int k = (ae == 0 ? -lzl : sh) - 62;
    if (NATURAL) {
        const int lz = clz(v);
        v = mulhi(v << (lz & 63), 0xB17217F7D1CF79ABull);       // ln 2, Q0.64
        k -= lz;
    }
    return pack(v, k, sign);
}

// The 64 bits below (hi:lo) >> s, s in [0, 128).
SYNAX_FX_FN u64 below128(u64 hi, u64 lo, int s) {
    const int t = s & 63;
    const u64 w0 = s < 64 ? 0ull : lo, w1 = s < 64 ? lo : hi;
    return (w0 >> t) | ((w1 << 1) << (63 - t));
}

// sin and cos of x radians, or (REV) of x revolutions.
template <bool REV, bool ZEROS = true>
SYNAX_FX_FN void sincos_any(double x, double* sn, double* cs) {
    const u64 b = bits_of(x);
    const int ex = biased_exp(b);
    // Huge, subnormal or not finite.  The product with 4 / (2 pi) is off by up to 2^(e - 125) for
    // |x| in [2^e, 2^(e + 1)), which below 2^14 radians is 2^-59.5 of the distance to the nearest
    // multiple of pi/2 or less (29 pi/2 is 2^-60.5 from a double, and so its doubles in proportion).
    // Any fraction of 2^60 revolutions is exact.
    if (ex > 1023 + (REV ? 60 : (ZEROS ? 13 : 30)) || (ex == 0 && (b << 1) != 0)) {
#ifdef __CUDACC__
        if (REV) ::sincospi(2.0 * x, sn, cs);
        else ::sincos(x, sn, cs);
#else
        const double a = REV ? 6.283185307179586476925 * x : x;
        *sn = std::sin(a);
        *cs = std::cos(a);
#endif
        return;
    }
    const u64 M = mantissa(b);
    const int e = ex - 1023;
    // |x| in revolutions 2^(REV ? -e : 2 - e), Q1.127
    u64 hi, lo;
    if (REV) {
        hi = M;
        lo = 0;
    } else {
        const u64 K1 = 0xA2F9836E4E441529ull, K2 = 0xFC2757D1F534DDC0ull;   // 4 / (2 pi), Q0.64 and beyond
        hi = mulhi(M, K1);
        lo = M * K1;
        const u64 c = mh(M, K2);
        lo += c;
        hi += lo < c ? 1 : 0;
    }
    const int e4 = REV ? e : e - 2;
    u64 top;
    const u64 phi = shr128(hi, lo, 63 - e4, top);             // revolutions mod 1, Q0.64
    const u32 quad = (u32)((phi + 0x2000000000000000ull) >> 62);
    const u64 r = phi - ((u64)quad << 62);                    // signed, |r| <= 1/8
    const u64 rs = r >> 63;
    u64 a = rs ? 0ull - r : r;
    a -= a >> 61;                                             // 1/8 itself: the largest word below it
    const u64 w = a << 3;                                     // 8 |r| = |angle| 4 / pi, Q0.64
    const u64 u = mh(w, w);
    u64 ps = 0x000000000005B16Eull;                           // sin(pi w / 4) / w, Q0.64
    ps = 0x0000000007A3BB44ull - mh(ps, u);
    ps = 0x000000078C1D2D3Full - mh(ps, u);
    ps = 0x00000541E0D2172Full - mh(ps, u);
    ps = 0x000265A599CC5584ull - mh(ps, u);
    ps = 0x00A335E33BAD56C9ull - mh(ps, u);
    ps = 0x14ABBCE625BE52BBull - mh(ps, u);
    ps = 0xC90FDAA22168C234ull - mh(ps, u);
    u64 pc = 0x000000000000479Dull;                           // (1 - cos(pi w / 4)) / u, Q0.64
    pc = 0x00000000006DB7A2ull - mh(pc, u);
    pc = 0x000000007E74E1C2ull - mh(pc, u);
    pc = 0x00000069B47CA821ull - mh(pc, u);
    pc = 0x00003C3EA0D1235Dull - mh(pc, u);
    pc = 0x00155D3C7E3CBFF6ull - mh(pc, u);
    pc = 0x040F07C206D6B0ECull - mh(pc, u);
    pc = 0x4EF4F326F9177969ull - mh(pc, u);
    // an unreduced angle keeps its full mantissa (8 |x| = hi 2^(e4 + 3 - 63))
    const bool whole = quad == 0 && e4 < -3;
    u64 wn = w;                                               // 8 |r| 2^lz
    int lz = 0;
    if (ZEROS) {
        // |r| with the 64 bits below it, normalised
        const u64 rl = below128(hi, lo, 63 - e4);
        const u64 h = rs ? ~r + (rl == 0 ? 1 : 0) : r, l = rs ? 0ull - rl : rl;
        const u64 h1 = h ? h : l, l1 = h ? l : 0ull;
        const int z = clz(h1);
        wn = (h1 << (z & 63)) | ((l1 >> 1) >> ((63 - z) & 63));
        lz = (h ? z : z + 64) - 3;
    }
    const double s0 = whole ? pack(mh(hi, ps), e4 + 3 - 63, rs << 63) : pack(mh(wn, ps), -64 - lz, rs << 63);
    const double c0 = pack(0x8000000000000000ull - (mh(u, pc) >> 1), -63, 0);
    const bool swap = quad & 1;
    const u64 ss = bits_of(swap ? c0 : s0) ^ ((u64)(quad >> 1) << 63) ^ (b & 0x8000000000000000ull);
    const u64 cc = bits_of(swap ? s0 : c0) ^ ((u64)((quad + 1) & 2) << 62);
    *sn = of_bits(ss);
    *cs = of_bits(cc);
}

// atan2(y, x)
template <bool ZEROS = true>
SYNAX_FX_FN double atan2(double y, double x) {
    const u64 yb = bits_of(y), xb = bits_of(x);
    const u64 sign_bit = 0x8000000000000000ull;
    const u64 ya = yb & ~sign_bit, xa = xb & ~sign_bit;
    const bool steep = ya > xa;                               // |y| > |x| (the bits of FP64 magnitudes are ordered)
    const u64 big = steep ? ya : xa, small = steep ? xa : ya;
    const int eb = biased_exp(big), de = eb - biased_exp(small);
    // (a quotient that may fall below the normal range included)
    if (eb == 0 || eb == 0x7FF || (small != 0 && (biased_exp(small) == 0 || (ZEROS && de > 1000)))) {
#ifdef __CUDACC__
        return ::atan2(y, x);
#else
        return std::atan2(y, x);
#endif
    }
    // w = small / big in [0, 1], Q0.64 (1 itself as the largest word)
    const u64 q = mulhi(mantissa(small), rcp_core(mantissa(big)));          // mantissa ratio, Q2.62
    u64 w = de > 63 ? 0ull : (de >= 2 ? q >> (de - 2) : (q >> 62 && (de == 0 || q >> 63) ? ~0ull : q << (2 - de)));
    const u64 u = mh(w, w);
    u64 p = 0x000013B06050D7CAull;                            // atan(w) / w, Q1.63
    p = 0x00010AFB5DFA4FF9ull - mh(p, u);
    p = 0x0006C0FAD7A13A79ull - mh(p, u);
    p = 0x001BE49BCD43B438ull - mh(p, u);
    p = 0x0052E2F3B6D9E8FCull - mh(p, u);
    p = 0x00BDF70523BCA88Full - mh(p, u);
    p = 0x01607C09CDCFA333ull - mh(p, u);
    p = 0x0226E02ECEF13905ull - mh(p, u);
    p = 0x02EFDA08E589AF70ull - mh(p, u);
    p = 0x03A02B6236FADB86ull - mh(p, u);
    p = 0x042FB842DFBF29ACull - mh(p, u);
    p = 0x04A79AFB4D5CA315ull - mh(p, u);
    p = 0x0517CDBBCC35C989ull - mh(p, u);
    p = 0x058EE9268F13C20Aull - mh(p, u);
    p = 0x061801BE51559B9Aull - mh(p, u);
    p = 0x06BC919BE1B86F56ull - mh(p, u);
    p = 0x0787856861092217ull - mh(p, u);
    p = 0x0888885173291AB2ull - mh(p, u);
    p = 0x09D89D85AEC3E1B6ull - mh(p, u);
    p = 0x0BA2E8B9F4F03019ull - mh(p, u);
    p = 0x0E38E38E36CA11CEull - mh(p, u);
    p = 0x1249249249187AA0ull - mh(p, u);
    p = 0x1999999999997478ull - mh(p, u);
    p = 0x2AAAAAAAAAAAAA7Dull - mh(p, u);
    p = 0x7FFFFFFFFFFFFFFFull - mh(p, u);
    u64 t = mh(w, p) >> 1;                                    // radians, Q2.62
    const u64 pi = 0xC90FDAA22168C234ull;                     // Q2.62
    t = steep ? (pi >> 1) - t : t;
    t = (xb & sign_bit) ? pi - t : t;
    // beside zero, from the quotient before its shift: q 2^-de atan(w) / w
    const bool near0 = ZEROS && !steep && de >= 2 && !(xb & sign_bit);
    return pack(near0 ? mulhi(q << 1, p) : t, -62 - (near0 ? de : 0), yb & sign_bit);
}

// sech^2 x and tanh x for 0 <= x < 300, from e = e^(-2x): 4 e / (1 + e)^2 and (1 - e) / (1 + e).
SYNAX_FX_FN void sech2_tanh(double x, double& sech2, double& th) {
    const u64 b = bits_of(x);
    if (biased_exp(b) > 1023 + 7 || (b >> 63)) {              // x >= 256, or NaN
        const double e = exp_any<true>(-2.0 * x), inv = rcp(1.0 + e);
        sech2 = 4.0 * e * inv * inv;
        th = (1.0 - e) * inv;
        return;
    }
    u64 f;
    const int t = scaled_split(b, kLog2e1, kLog2e2, 1, f);
    const int n = f ? t + 1 : t;                              // e = 2^-n m
    const u64 m = 0x8000000000000000ull + (exp2m1_core(0ull - f) >> 1);   // in [1, 2), Q1.63
    u64 e = n > 63 ? 0ull : m >> (n & 63);                    // Q1.63
    e -= e >> 63;                                             // (e = 1: keep 1 + e below 2)
    const u64 inv = rcp_core(0x8000000000000000ull + e);
    sech2 = pack(mulhi(mulhi(m, inv), inv), -n + 2 - 61, 0);
    th = pack(mulhi(0x8000000000000000ull - e, inv), -62, 0);
}
// a > b for a >= 0 (the bits of FP64 magnitudes are ordered); true for NaN.
SYNAX_FX_FN bool above(double a, double b) { return bits_of(a) > bits_of(b); }
// floor(v) (clamped to +-2^30) and v - floor(v), the fraction exact to 2^-64.
SYNAX_FX_FN double split_floor(double v, int& whole) {
    const u64 b = bits_of(v);
    const int ex = biased_exp(b);
    const bool neg = b >> 63;
    if (ex > 1023 + 29) {                                     // huge or not finite
        whole = v != v ? 0 : (neg ? -(1 << 30) : 1 << 30);
        return v - v;                                         // (0, or NaN)
    }
    u64 top;
    u64 f = shr128(mantissa(b), 0, 1086 - ex, top);
    whole = neg ? (f ? -(int)top - 1 : -(int)top) : (int)top;
    f = neg ? 0ull - f : f;
    return pack(f, -64, 0);
}
// f in [0, 1] as Q1.63 (a number: NaN has no fixed-point form).
SYNAX_FX_FN u64 unit_q63(double f) {
    const u64 b = bits_of(f);
    const int s = 1023 - biased_exp(b);
    return s > 63 ? 0ull : mantissa(b) >> (s & 63);
}
// A small integer as FP64.
SYNAX_FX_FN double from_int(int k) {
    return pack((u64)(u32)(k < 0 ? -k : k), 0, k < 0 ? 0x8000000000000000ull : 0ull);
}
// The 8 trilinear weights prod (d ? f : 1 - f) of a cell, node q = (q & 1,
// (q >> 1) & 1, q >> 2) along (x, y, z).
SYNAX_FX_FN void trilinear_weights(double fx, double fy, double fz, double w[8]) {
    const u64 one = 0x8000000000000000ull;
    const u64 x1 = unit_q63(fx), y1 = unit_q63(fy), z1 = unit_q63(fz);
    const u64 x[2] = {one - x1, x1}, y[2] = {one - y1, y1}, z[2] = {one - z1, z1};
    for (int q = 0; q < 4; ++q) {
        const u64 yz = mh(y[q & 1], z[q >> 1]) << 1;          // Q1.63
        w[2 * q] = pack(mh(x[0], yz), -62, 0);
        w[2 * q + 1] = pack(mh(x[1], yz), -62, 0);
    }
}

}  // namespace fx
}  // namespace synax
