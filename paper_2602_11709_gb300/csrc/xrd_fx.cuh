// 64-bit fixed-point exp and sin/cos for the FP64 structure-factor loop.
//
// One FP64 operation costs as much as about 70 integer ones on this part (1.7
// lane operations per clock and SM), so the FP64 loop's exponentials and
// phase factors are formed in integers: a table (1024 exponentials, 513 phase
// factors of a quarter turn) and a short Taylor series, every product a 32 x 32
// bit multiplication or three of them. exp(-x) errs by less than (1/2 + x/128)
// 2^-53 of itself before it is rounded to a double (rounding x itself to a
// double costs up to x 2^-53). sin and cos err by less than 6.5e-18 absolute
// (3.7e-18 seen), a 17th of a rounding at 1, but not relative to themselves
// next to a zero as the library's do: in a structure factor's sum the
// rounding of the phase, which is exact here, weighed more.
//
// Host and device: tests/test_fx_host.py compares both functions, compiled for
// the host, with a 60-digit evaluation.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace xrd {

#define XRD_HD __host__ __device__ __forceinline__

XRD_HD uint32_t fx_hi32(uint64_t x) { return (uint32_t)(x >> 32); }
XRD_HD uint32_t fx_mulhi(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
// high 64 bits of a b, the low halves' product left out (below by at most 3 units)
XRD_HD uint64_t fx_mulhi64(uint64_t a, uint64_t b)
{
    const uint32_t ah = fx_hi32(a), al = (uint32_t)a, bh = fx_hi32(b), bl = (uint32_t)b;
    return (uint64_t)ah * bh + fx_mulhi(ah, bl) + fx_mulhi(al, bh);
}
XRD_HD uint64_t fx_umul64hi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    const uint32_t ah = fx_hi32(a), al = (uint32_t)a, bh = fx_hi32(b), bl = (uint32_t)b;
    const uint64_t mid = (uint64_t)ah * bl + fx_mulhi(al, bl), low = (uint64_t)al * bh + (uint32_t)mid;
    return (uint64_t)ah * bh + fx_hi32(mid) + fx_hi32(low);
#endif
}
XRD_HD int fx_clz64(uint64_t x)  // x != 0
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}
XRD_HD double fx_as_double(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    __builtin_memcpy(&d, &b, 8);
    return d;
#endif
}
XRD_HD uint64_t fx_as_bits(double d)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(d);
#else
    uint64_t b;
    __builtin_memcpy(&b, &d, 8);
    return b;
#endif
}

constexpr int kFxExpN = 1024;  // 2^(-j / 1024), 64 fractional bits
constexpr int kFxScN = 512;    // cos and sin of (j / 512) quarter turns, 62 fractional bits, j = 0 .. 512

// A positive double as m 2^(e - 63), m in [2^63, 2^64). Zero has m = 0 and an exponent below any other's: fx_exp2_neg
// takes a product's size from the exponents, and a product of zero is small whatever the other factor.
struct FxNum {
    uint64_t m;
    int e;
};
constexpr int kFxZero = -4096;
constexpr int kFxSlow = 1 << 20;  // exponent of an exponent coefficient that the fixed-point form does not cover

// v >= 0 (a normal double, or zero)
XRD_HD FxNum fx_num(double v)
{
    const uint64_t b = fx_as_bits(v);
    FxNum r;
    r.e = (int)(b >> 52) - 1023;
    r.m = ((b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11;
    if (v == 0.0) {
        r.m = 0;
        r.e = kFxZero;
    }
    return r;
}

// b log2(e) for an exponent coefficient b >= 0, to about 2^-64 relative; e = kFxSlow where b is negative, not
// finite or outside [2^-300, 2^300] (and not zero): the caller takes the library's exp there.
XRD_HD FxNum fx_log2e(double b)
{
    if (b == 0.0) return FxNum{0ull, kFxZero};
    if (!(b >= 0x1p-300 && b <= 0x1p300)) return FxNum{0ull, kFxSlow};
    constexpr uint64_t L = 0xB8AA3B295C17F0BCull;  // log2(e) 2^63
    const FxNum n = fx_num(b);
    const uint64_t hi = fx_umul64hi(n.m, L);  // in [0.72 2^62, 1.45 2^63): the product 2^(e - 62) / 2^64
    const uint64_t lo = n.m * L;
    if (hi >> 63) return FxNum{hi + (lo >> 63), n.e + 1};
    return FxNum{(hi << 1) | (lo >> 63), n.e};
}

// exp(-b s2) for bl2 = b log2(e) and s2, as (m, n): the value is m 2^(-64 - n), m in [2^63, 2^64), or m = 0 (and n >= 1021)
// where it is below 2^-1021. tab: kFxExpN entries.
XRD_HD uint64_t fx_exp2_neg(uint64_t bm, int be, uint64_t sm, int se, const uint64_t* __restrict__ tab, int& n)
{
    const uint64_t P = fx_mulhi64(bm, sm);
    const int sh = 9 - be - se;  // T = b s2 log2(e) with 53 fractional bits
    n = 2048;
    if (sh < 0) return 0ull;
    const uint64_t T = sh == 0 ? P : (sh <= 64 ? ((P >> (sh - 1)) + 1ull) >> 1 : 0ull);
    n = (int)(T >> 53);
    if (n >= 1021) return 0ull;
    const uint32_t j = (uint32_t)(T >> 43) & (kFxExpN - 1);
    // y = ln2 r for the remaining 43 bits r 2^-53 < 2^-10: y < 6.8e-4, 74 fractional bits
    constexpr uint32_t Lh = 0xB17217F7u, Ll = 0xD1CF79ACu;  // ln 2, 64 fractional bits
    const uint32_t rh = (uint32_t)(T >> 11), rl = (uint32_t)T << 21;
    const uint64_t y = (uint64_t)rh * Lh + fx_mulhi(rh, Ll) + fx_mulhi(rl, Lh);
    const uint32_t yh = fx_hi32(y), yl = (uint32_t)y;
    // exp(-y) = 1 - (y - y^2/2 + y^3/6 - y^4/24), next term below 2^-59
    const uint64_t y2 = (uint64_t)yh * yh + ((uint64_t)fx_mulhi(yh, yl) << 1);  // y^2, 84 fractional bits
    const uint32_t y3 = fx_mulhi(fx_hi32(y2), yh);                               // y^3, 62
    const uint32_t y4 = fx_mulhi(y3, yh);                                        // y^4, 72
    const uint64_t c3 = (uint64_t)fx_mulhi(y3, 0x2AAAAAABu) << 12;               // y^3/6, 74
    const uint32_t c4 = fx_mulhi(y4, 715827883u);                                // y^4/6, 72 = y^4/24, 74
    const uint64_t p = y - (y2 >> 11) + c3 - c4;
    const uint64_t t = tab[j];
    return t - (fx_mulhi64(t, p) >> 10);
}

// (m, n) of fx_exp2_neg as a double (rounded to nearest; results below 2^-1021 are 0)
XRD_HD double fx_exp_double(uint64_t m, int n)
{
    if (m == 0ull) return 0.0;
    return fx_as_double(((uint64_t)(1021 - n) << 52) + (m >> 11) + ((m >> 10) & 1ull));
}

// A normal double as (-1)^(e & 1) am 2^((e >> 1) - 60), am in [2^60, 2^61); zero has am = 0 and an exponent below any other's.
XRD_HD uint64_t fx_signed(double v, int& e)
{
    const FxNum n = fx_num(v < 0.0 ? -v : v);
    e = 2 * n.e + (v < 0.0);
    return n.m >> 3;
}

// sum of four such numbers (am, ae) times exp(-b_i s2), the exponentials as in fx_exp2_neg, to 2^-58 of the largest term:
// terms are aligned to that one, not to the largest coefficient, whose term may have decayed.
XRD_HD double fx_exp_sum(const uint64_t* am, const int16_t* ae, const uint64_t* bm, const int16_t* be, FxNum S,
                         const uint64_t* __restrict__ tab)
{
    uint64_t v[4];
    int e[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        int n;
        const uint64_t m = fx_exp2_neg(bm[i], be[i], S.m, S.e, tab, n);
        v[i] = fx_mulhi64(am[i], m);  // v 2^(e - 60), below 2^61
        e[i] = (ae[i] >> 1) - n;
    }
    const int t0 = e[0] > e[1] ? e[0] : e[1], t1 = e[2] > e[3] ? e[2] : e[3], top = t0 > t1 ? t0 : t1;
    int64_t sum = 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int sh = top - e[i];
        const int64_t w = (int64_t)(v[i] >> (sh < 63 ? sh : 63)), neg = -(int64_t)(ae[i] & 1);
        sum += (w ^ neg) - neg;
    }
    const uint64_t sign = (uint64_t)sum & 0x8000000000000000ull;
    const uint64_t a = sum < 0 ? 0ull - (uint64_t)sum : (uint64_t)sum;
    const int z = fx_clz64(a | 1ull);
    const int f = 1023 + 62 + top - 60 - z;  // exponent field less one: the significand's top bit carries into it
    const uint64_t m = a << z;
    if (a == 0ull || f < 0) return 0.0;  // below 2^-1022
    return fx_as_double(sign | (((uint64_t)f << 52) + (m >> 11) + ((m >> 10) & 1ull)));
}

// A signed fixed-point number with F fractional bits as a double (rounded to nearest)
template <int F>
XRD_HD double fx_to_double(int64_t v)
{
    const uint64_t sign = (uint64_t)v & 0x8000000000000000ull;
    const uint64_t a = v < 0 ? 0ull - (uint64_t)v : (uint64_t)v;
    if (a == 0ull) return 0.0;
    const int z = fx_clz64(a);
    const uint64_t m = a << z;  // in [2^63, 2^64)
    return fx_as_double(sign | (((uint64_t)(1023 + 62 - F - z) << 52) + (m >> 11) + ((m >> 10) & 1ull)));
}

// cos and sin of 2 pi P / 2^64 with 62 fractional bits. tab: kFxScN + 1 pairs (cos, sin) of the first quarter turn.
XRD_HD void fx_sincos(uint64_t P, const ulonglong2* __restrict__ tab, int64_t& c, int64_t& s)
{
    const uint32_t q = (uint32_t)(P >> 62);
    const uint32_t j = (uint32_t)(P >> 53) & (kFxScN - 1);
    const uint64_t d = P & ((1ull << 53) - 1);  // turns 2^-64, below 2^-11 turn
    // x = 2 pi d 2^-64 < 3.07e-3, 71 fractional bits
    constexpr uint64_t kTwoPi61 = 0xC90FDAA22168C235ull;  // 2 pi, 61 fractional bits
    const uint64_t x = fx_mulhi64(d << 10, kTwoPi61);
    const uint32_t xh = fx_hi32(x), xl = (uint32_t)x;
    const uint64_t x2 = (uint64_t)xh * xh + ((uint64_t)fx_mulhi(xh, xl) << 1);  // x^2, 78 bits (< 2^61.3)
    const uint32_t a2 = (uint32_t)(x2 >> 30), a1 = (uint32_t)(x >> 31);          // x^2 with 48 bits, x with 40
    const uint64_t x3 = (uint64_t)a2 * a1;                                       // x^3, 88 bits (< 2^63)
    const uint32_t a3 = fx_hi32(x3);                                             // 56 bits
    const uint32_t a5 = fx_mulhi(a3, a2);                                        // x^5, 72 bits
    // sin x = x - x^3/6 + x^5/120 (next term below 2^-71); 71 bits
    const uint64_t sx = x - (((uint64_t)a3 * 0x2AAAAAABu) >> 17) + (fx_mulhi(a5, 35791394u) >> 1);
    // 1 - cos x = x^2/2 - x^4/24 + x^6/720 (1.2e-18); 78 bits
    const uint32_t a4 = fx_mulhi(a2, a2);                                        // x^4, 64 bits
    const uint64_t cx = (x2 >> 1) - ((uint64_t)fx_mulhi(a4, 178956971u) << 14) +
                        ((uint64_t)fx_mulhi(fx_mulhi(a4, a2), 5965232u) >> 2);  // a4 a2: x^6 with 80 bits
    const ulonglong2 t = tab[j];
    const int64_t c0 = (int64_t)(t.x - (fx_mulhi64(t.x, cx << 2) >> 16) - (fx_mulhi64(t.y, sx) >> 7));
    const int64_t s0 = (int64_t)(t.y - (fx_mulhi64(t.y, cx << 2) >> 16) + (fx_mulhi64(t.x, sx) >> 7));
    // (cos, sin) of x + q quarter turns
    const int64_t c1 = q & 1u ? s0 : c0, s1 = q & 1u ? c0 : s0;
    c = (q + 1u) & 2u ? -c1 : c1;
    s = q & 2u ? -s1 : s1;
}

}  // namespace xrd
