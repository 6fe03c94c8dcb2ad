// qex_fix64.cuh -- FP64 hops on the integer pipe.
//
// An FP64 FMA takes 64 clocks a warp on a GB300 SM quarter, a 32x32+64-bit
// integer multiply-add and every other integer instruction 2 (measured; the
// two kinds of integer instruction share those clocks).  A 3x3 complex
// mat-vec is 36 FP64 FMAs, 2304 clocks; here it takes 1180: the link and the
// vector are brought into fixed point (a common exponent each, 60 bits, as
// two signed 32-bit digits), a product is three multiply-adds (hi hi, hi lo,
// lo hi; the lo lo product is below the last bit kept) and the sums are exact
// 64-bit integers.  About half of the 600 instructions convert the link.
//
// Accuracy.  One unit of the accumulators is 2^-56 of the largest product
// |U| |v| (largest real of the link times largest real of the vectors, each
// rounded up to a power of two); a hop rounds by about 0.3 units and by 2.75 at
// most, and the running exponent carries kFixSlack spare bits.  FP64 arithmetic
// rounds every partial sum by 2^-54 of its value.  Norm-wise error of a sum of
// eight hops against 113 bits, Gaussian vectors: 0.64e-16 here, 2.3e-16 for FMAs
// (unit links: 0.71e-16 and 1.05e-16; vectors of very different size from
// hop to hop: 0.88e-16 and 2.2e-16).
//
// That is against the largest product of the site.  A real whose own terms are all
// far smaller (a colour, or imaginary parts, decades below the others, in links
// that do not mix them) would lose bits that FMAs keep.  So each hop also adds up,
// in packed halves and a little above its truth, what the magnitudes of every
// real's terms come to, and a colour with a real whose terms do not reach kFixTerms
// is formed again with FMAs.  The rest are within 18 x 2^-53 of their terms' sum, where
// the 48 FMAs they stand for are within 48, and rms at 0.1 to 0.9 of those.
// Gaussian vectors meet no such site (1e-4 of them with Gaussian links); where
// every site is one (unit links, or colours 1e-2 apart with links that do not mix
// them) the operator takes 330-430 us at 32^4 in place of 141.  The bound's 80
// instructions a hop cost 8 % (byte magnitudes through __dp4a: 40 %, it takes as
// long as an FP64 FMA).
//
// A hop whose link or vector holds an Inf or NaN, or whose largest real lies
// outside 2^-470 .. 2^470 (zeros apart), makes the site fall back to FP64 FMAs as
// well, so such values come out as they do there.
#pragma once

#include <math.h>
#include <string.h>

#include <cuda_fp16.h>

#include "qex_common.cuh"

namespace qex {

constexpr int kFixShift = 4;   // high digits are at most 2^28
constexpr int kFixSlack = 1;   // spare bits of the running exponent
constexpr int kFixLow = 553;    // exponent fields accepted: 2^-470 <= ...
constexpr int kFixHigh = 1493;  // ... < 2^470
constexpr float kFixTerms = 0x1p-11f;  // what FixSum::terms has to come to: 2^54 units, 2^53 at least in truth

struct Digits {
    int hi, lo;  // hi 2^32 + lo
};

QEX_HD uint64_t fix_shr(uint64_t x, uint32_t n) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));  // 0 for n > 63
    return r;
#else
    return n > 63 ? 0 : x >> n;
#endif
}

QEX_HD uint64_t fix_shl(uint64_t x, uint32_t n) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));  // 0 for n > 63
    return r;
#else
    return n > 63 ? 0 : x << n;
#endif
}

QEX_HD int64_t fix_sar(int64_t x, uint32_t n) { return x >> (n > 63 ? 63 : n); }

// a b + c, one IMAD.WIDE
QEX_HD int64_t fix_mad(int a, int b, int64_t c) { return (int64_t)a * b + c; }

QEX_HD uint64_t fix_bits(double d) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(d);
#else
    uint64_t u;
    memcpy(&u, &d, 8);
    return u;
#endif
}

QEX_HD double fix_double(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    memcpy(&d, &u, 8);
    return d;
#endif
}

QEX_HD uint32_t fix_mag(double d) { return (uint32_t)(fix_bits(d) >> 32) & 0x7FFFFFFFu; }

// |d| in units of 2^(e - 1023 - 63 + kFixShift), truncated; key = ((e +
// kFixShift) << 20) | 0xFFFFF with e at least d's exponent field.  Zero (and
// anything 64 bits below 2^(e - 1023)) gives 0.
QEX_HD uint64_t fix_abs(uint32_t h, uint32_t l, uint32_t key) {
    const uint32_t n = (key - (h & 0x7FFFFFFFu)) >> 20;
#ifdef __CUDA_ARCH__
    const uint32_t t = __funnelshift_l(l, h, 11);
#else
    const uint32_t t = (h << 11) | (l >> 21);
#endif
    return fix_shr(((uint64_t)(t | 0x80000000u) << 32) | (l << 11), n);
}

QEX_HD Digits fix_digits(uint32_t hi, uint32_t lo) {
    Digits d;
    d.lo = (int)lo;
    d.hi = (int)(hi + (lo >> 31));
#ifdef __CUDA_ARCH__
    // Opaque from here on: seen through, the products below become 64-bit
    // multiplications of what the digits were made from.
    asm("" : "+r"(d.hi), "+r"(d.lo));
#endif
    return d;
}

// Magnitudes of a complex value by the leading 12 bits n of its high digits, read
// as the bits of two halves: n 2^-24 up to n = 2^11, at most twice that above.
#ifdef __CUDA_ARCH__
typedef __half2 FixMag;
#else
struct FixMag {
    float x, y;
};
inline float fix_half(uint32_t n) {
    return n < 0x400 ? ldexpf((float)n, -24) : ldexpf((float)((n & 0x3FF) | 0x400), (int)(n >> 10) - 25);
}
#endif

QEX_HD FixMag fix_mag2(uint32_t re, uint32_t im) {
#ifdef __CUDA_ARCH__
    const uint32_t w = __byte_perm(re, im, 0x7632);
    FixMag m;
    memcpy(&m, &w, 4);
    return m;
#else
    return {fix_half(re >> 16), fix_half(im >> 16)};
#endif
}

QEX_HD FixMag fix_const2(float x) {
#ifdef __CUDA_ARCH__
    return __float2half2_rn(x);
#else
    return {x, x};
#endif
}

QEX_HD FixMag fix_min2(FixMag a, FixMag b) {
#ifdef __CUDA_ARCH__
    return __hmin2(a, b);
#else
    return {a.x < b.x ? a.x : b.x, a.y < b.y ? a.y : b.y};
#endif
}

QEX_HD FixMag fix_mul2(FixMag a, FixMag b) {
#ifdef __CUDA_ARCH__
    return __hmul2(a, b);
#else
    return {a.x * b.x, a.y * b.y};
#endif
}

QEX_HD FixMag fix_swap2(FixMag a) {
#ifdef __CUDA_ARCH__
    return __lowhigh2highlow(a);
#else
    return {a.y, a.x};
#endif
}

// c + (a.x + i a.y's magnitudes)(b.x + i b.y's): re and im; bx: b swapped.
QEX_HD FixMag fix_terms2(FixMag a, FixMag b, FixMag bx, FixMag c) {
#ifdef __CUDA_ARCH__
    return __hfma2(__high2half2(a), bx, __hfma2(__low2half2(a), b, c));
#else
    return {a.x * b.x + a.y * bx.x + c.x, a.x * b.y + a.y * bx.y + c.y};
#endif
}

QEX_HD FixMag fix_add2(FixMag a, FixMag b) {
#ifdef __CUDA_ARCH__
    return __hadd2(a, b);
#else
    return {a.x + b.x, a.y + b.y};
#endif
}

QEX_HD float fix_least(FixMag a) {
#ifdef __CUDA_ARCH__
    return fminf(__low2float(a), __high2float(a));
#else
    return a.x < a.y ? a.x : a.y;
#endif
}

// Link real: a negative one is complemented instead of negated (one unit of
// 2^-60 off), a zero of either sign stays 0.
QEX_HD Digits fix_link_real(double d, uint32_t key, uint32_t &lead) {
    const uint64_t b = fix_bits(d);
    const uint32_t h = (uint32_t)(b >> 32);
    const uint64_t x = fix_abs(h, (uint32_t)b, key);
    uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
    lead = hi;
    if (h > 0x80000000u) {
        hi = ~hi;
        lo = ~lo;
    }
    return fix_digits(hi, lo);
}

// Vector real times (neg ? -1 : 1), exactly negated.
QEX_HD uint64_t fix_vec_real(double d, uint32_t key, bool neg, uint32_t &lead) {
    const uint64_t b = fix_bits(d);
    const uint32_t h = (uint32_t)(b >> 32);
    const uint64_t x = fix_abs(h, (uint32_t)b, key);
    lead = (uint32_t)(x >> 32);
    return ((int32_t)h < 0) != neg ? 0 - x : x;
}

// Sum of the hops so far: value a[.] 2^(e - kFixUnit); re/im of colours 0..2.
// |a| < 2^62 for up to 8 hops: |U1| |V1| <= 2^56, 6 products a hop.
constexpr int kFixUnit = 2 * 1023 + 2 * (63 - kFixShift) - 64;
struct FixSum {
    int64_t a[6];
    int e;
    FixMag terms[3];  // what the terms of colour a come to, re and im, in units of 2^65: within [0.9, 2] of the truth
    bool some;        // a hop was not all zeros
    bool bad;
};

// terms 2^-n (nothing left past 14)
QEX_HD FixMag fix_lower(FixMag t, uint32_t n) {
#ifdef __CUDA_ARCH__
    const uint32_t w = n < 15u ? (15u - n) * 0x04000400u : 0u;
    FixMag p;
    memcpy(&p, &w, 4);
    return __hmul2(t, p);
#else
    const float p = n < 15u ? ldexpf(1.f, -(int)n) : 0.f;
    return {t.x * p, t.y * p};
#endif
}

QEX_HD bool fix_few(FixMag terms, float least = kFixTerms) { return fix_least(terms) < least; }

// |c| 2^e <= 2^f: a sum in units of c 2^e loses no more than one in units of 2^f.  With
// terms of twice kFixTerms in the second they are enough for both.
QEX_HD bool fix_below(double c, int e, int f) { return (int)(fix_mag(c) >> 20) - 1022 + e <= f; }

QEX_HD void fix_clear(FixSum &s) {
    for (int k = 0; k < 6; ++k) s.a[k] = 0;
    s.e = 0;
    for (int a = 0; a < 3; ++a) s.terms[a] = fix_const2(0.f);
    s.some = false;
    s.bad = false;
}

QEX_HD uint32_t fix_max(uint32_t a, uint32_t b) { return a > b ? a : b; }

// The largest magnitude m (high word) of a link or vector, raised to the
// smallest accepted one if all of it is zero (any() is the OR of its words),
// which sets zero; bad is set if it is out of range.
template <typename Any>
QEX_HD uint32_t fix_range(uint32_t m, bool &bad, bool &zero, const Any &any) {
    if (m >= (uint32_t)kFixHigh << 20) bad = true;
    if (m < (uint32_t)kFixLow << 20) {
        if (any() << 1) bad = true;  // a sign bit alone is a zero
        zero = true;
        m = (uint32_t)kFixLow << 20;
    }
    return m;
}

QEX_HD uint64_t fix_any(const Vec3<double> &v) {
    uint64_t any = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) any |= fix_bits(v.c[a].re) | fix_bits(v.c[a].im);
    return any;
}

// s += (neg ? -1 : 1) U v (DAG: U^+ v).  side(a), a = 0, 1, 2: FP64 work of
// the caller placed between the integer instructions of the three rows.
struct NoSide {
    QEX_HD void operator()(int) const {}
};
template <bool DAG, int SLACK = kFixSlack, typename Side = NoSide>
QEX_HD void fix_hop(FixSum &s, const Mat3<double> &u, const Vec3<double> &v, bool neg, const Side &side = Side()) {
    uint32_t mu = 0, mv = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) mu = fix_max(mu, fix_max(fix_mag(u.e[k].re), fix_mag(u.e[k].im)));
#pragma unroll
    for (int a = 0; a < 3; ++a) mv = fix_max(mv, fix_max(fix_mag(v.c[a].re), fix_mag(v.c[a].im)));
    bool zero = false;
    mu = fix_range(mu, s.bad, zero, [&] {
        uint64_t any = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k) any |= fix_bits(u.e[k].re) | fix_bits(u.e[k].im);
        return any;
    });
    mv = fix_range(mv, s.bad, zero, [&] { return fix_any(v); });
    const int eu = (int)(mu >> 20), eh = eu + (int)(mv >> 20);
    if (eh > s.e) {  // a larger product than the unit allows for: raise the unit
        const int e = eh + SLACK;
#pragma unroll
        for (int k = 0; k < 6; ++k) s.a[k] = fix_sar(s.a[k], (uint32_t)(e - s.e));
#pragma unroll
        for (int a = 0; a < 3; ++a) s.terms[a] = fix_lower(s.terms[a], (uint32_t)(e - s.e));
        s.e = e;
    }
    const uint32_t ku = ((uint32_t)(eu + kFixShift) << 20) | 0xFFFFFu;
    const uint32_t kv = ((uint32_t)(s.e - eu + kFixShift) << 20) | 0xFFFFFu;
    Digits vr[3], vi[3], vn[3];  // vn: -vi (DAG: -vr)
    FixMag vm[3], vx[3];         // |vr|, |vi| times 2^15 (at most 4: exact), and swapped
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        uint32_t lr, li;
        const uint64_t re = fix_vec_real(v.c[b].re, kv, neg, lr), im = fix_vec_real(v.c[b].im, kv, neg, li);
        vm[b] = fix_mul2(fix_min2(fix_mag2(lr, li), fix_const2(0x1p-13f)), fix_const2(0x1p15f));
        vx[b] = fix_swap2(vm[b]);
        vr[b] = fix_digits((uint32_t)(re >> 32), (uint32_t)re);
        vi[b] = fix_digits((uint32_t)(im >> 32), (uint32_t)im);
        const uint64_t n = 0 - (DAG ? re : im);
        vn[b] = fix_digits((uint32_t)(n >> 32), (uint32_t)n);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        side(a);
        int64_t hr = s.a[2 * a], hi = s.a[2 * a + 1];
        int64_t mr = 0x80000000ll, mi = 0x80000000ll;  // the half that rounds the fold below
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int k = DAG ? 3 * b + a : 3 * a + b;
            uint32_t lr, li;
            const Digits ur = fix_link_real(u.e[k].re, ku, lr), ui = fix_link_real(u.e[k].im, ku, li);
            s.terms[a] = fix_terms2(fix_mag2(lr, li), vm[b], vx[b], s.terms[a]);
            // U: (ur vr - ui vi, ur vi + ui vr);  U^+: (ur vr + ui vi, ur vi - ui vr)
            const Digits x = DAG ? vi[b] : vn[b], y = DAG ? vn[b] : vr[b];
            hr = fix_mad(ur.hi, vr[b].hi, hr);
            mr = fix_mad(ur.hi, vr[b].lo, mr);
            mr = fix_mad(ur.lo, vr[b].hi, mr);
            hr = fix_mad(ui.hi, x.hi, hr);
            mr = fix_mad(ui.hi, x.lo, mr);
            mr = fix_mad(ui.lo, x.hi, mr);
            hi = fix_mad(ur.hi, vi[b].hi, hi);
            mi = fix_mad(ur.hi, vi[b].lo, mi);
            mi = fix_mad(ur.lo, vi[b].hi, mi);
            hi = fix_mad(ui.hi, y.hi, hi);
            mi = fix_mad(ui.hi, y.lo, mi);
            mi = fix_mad(ui.lo, y.hi, mi);
        }
        s.a[2 * a] = fix_mad((int)(mr >> 32), 1, hr);
        s.a[2 * a + 1] = fix_mad((int)(mi >> 32), 1, hi);
    }
    s.some |= !zero;
}

// The unit of a sum as a double (a power of two in range for a sum that is
// not bad: exponent fields 2 kFixLow .. 2 kFixHigh + kFixSlack).
QEX_HD double fix_unit(int e) { return fix_double((uint64_t)(uint32_t)(e - kFixUnit + 1023) << 52); }

// ---------------------------------------------- reals with an exponent each
// hi 2^32 + lo, 2^59 to 2^60 in magnitude, times 2^(e - kFixNum); zero: kFixNone.
constexpr int kFixNum = 1023 + 63 - kFixShift;
constexpr int kFixNone = -1000000;
struct FixNum {
    Digits d;
    int e;
};

QEX_HD FixNum fix_num(double d) {  // d normal or zero
    const uint64_t b = fix_bits(d);
    const uint32_t h = (uint32_t)(b >> 32), f = (h >> 20) & 0x7FFu;
    const uint64_t x = f ? (((b << 11) | 0x8000000000000000ull) >> kFixShift) : 0;
    const uint64_t y = (int32_t)h < 0 ? 0 - x : x;
    return {fix_digits((uint32_t)(y >> 32), (uint32_t)y), f ? (int)f : kFixNone};
}

QEX_HD int fix_clz(uint64_t x) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

QEX_HD FixNum fix_num(int64_t x, int e) {  // x 2^(e - kFixUnit), |x| < 2^62
    const int n = fix_clz((uint64_t)(x ^ (x >> 63)));
    const int64_t y = (int64_t)fix_shl((uint64_t)x, (uint32_t)(n - 1)) >> (kFixShift - 1);
    return {fix_digits((uint32_t)((uint64_t)y >> 32), (uint32_t)y),
            x ? e - kFixUnit + kFixNum + kFixShift - n : kFixNone};
}

// a b / 2^64 in units of 2^(a.e + b.e - 2 kFixNum + 64), within 0.75; shifted down n.
QEX_HD int64_t fix_product(const FixNum &a, const FixNum &b, int n) {
    int64_t m = fix_mad(a.d.hi, b.d.lo, 0x80000000ll);
    m = fix_mad(a.d.lo, b.d.hi, m);
    return fix_sar(fix_mad((int)(m >> 32), 1, fix_mad(a.d.hi, b.d.hi, 0)), (uint32_t)n);
}

// x 2^(e - kFixUnit) as a double, rounded to the nearest (half away from zero), for
// results in the normal range: about 46 clocks, where a conversion and a product
// with the unit take 128 on the FP64 pipe.
QEX_HD double fix_to_double(int64_t x, int e) {
    const uint64_t mag = x < 0 ? 0 - (uint64_t)x : (uint64_t)x;
    const int n = fix_clz(mag);
    const uint64_t top = fix_shl(mag, (uint32_t)n);  // leading bit at 63
    const uint64_t r = (top >> 11) + ((top >> 10) & 1);
    const uint64_t d = r + ((uint64_t)(uint32_t)(e - kFixUnit + 63 - n + 1022) << 52);  // a carry raises the exponent
    return fix_double(mag ? d | ((uint64_t)x & 0x8000000000000000ull) : 0);
}

}  // namespace qex
