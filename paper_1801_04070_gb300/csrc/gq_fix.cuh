// gq_fix.cuh -- 64-bit fixed-point arithmetic on the integer pipe for sums that
// need FP64's accuracy.
//
// GB300 issues one FP64 instruction of a warp every 64 (multiply-add) to 76
// (add, multiply) cycles per SM sub-partition, but a 32 x 32 + 64 bit integer
// multiply-add every 4 and another integer instruction every 2 on the second
// pipe (measured with 16 independent warps).  A 64 x 64 bit product rounded to
// its upper half takes three multiply-adds, a complex one twelve: about 60 cycles
// for a complex multiply-accumulate against 430 on the FP64 pipe.  Where the
// operands have a known range (|r/w| <= 1, a shared exponent for the strengths)
// fixed point loses nothing: sums are exact and a product is rounded at 2^-60 of
// the largest term, below FP64's own 2^-53 of each term.
//
// A number is held as value = h 2^32 + l with both words signed ("balanced"),
// so that every partial product is a signed mad.wide.  The functions also
// compile for the host (the CPU checks of their error).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define GQ_HD __host__ __device__ __forceinline__
#else
#define GQ_HD inline
#endif

struct gfx {
    int h, l;
};

// a b + c.  Written as the carry chain that becomes one multiply-add; mad.wide
// itself is split into a product and a 64-bit addition.
GQ_HD long long fx_mw(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    unsigned l, h;
    asm("mad.lo.cc.s32 %0, %2, %3, %4; madc.hi.s32 %1, %2, %3, %5;"
        : "=&r"(l), "=r"(h)
        : "r"(a), "r"(b), "r"((unsigned)c), "r"((unsigned)(c >> 32)));
    return (long long)((unsigned long long)h << 32 | l);
#else
    return (long long)a * b + c;
#endif
}
// (the wrapping conversions below are two's complement on every target)
GQ_HD long long fx_shl(long long v, int s) { return (long long)((unsigned long long)v << s); }

GQ_HD gfx fx_bal(long long v) {
    gfx r;
    r.l = (int)v;
    r.h = (int)(v >> 32) + (int)((unsigned)r.l >> 31);
    return r;
}

// a b / 2^64, rounded (the product of the two low words, below 2^-2 units, is dropped)
GQ_HD long long fx_mul(gfx a, gfx b) {
    const long long mid = fx_mw(a.h, b.l, fx_mw(a.l, b.h, 1LL << 31));
    return fx_mw(a.h, b.h, (long long)(int)(mid >> 32));
}

// A factor split at bit 30: v = h 2^30 + l / 4 (l holds four times the low part,
// with its sign), so that v u / 2^62 has whole words as its partial products'
// places and needs no shift.  |v| < 2^61.
struct gfx30 {
    int h, l;
};
GQ_HD gfx30 fx_split30(long long v) {
    gfx30 r;
    r.l = (int)((unsigned)v << 2);
    r.h = (int)(v >> 30) + (int)((unsigned)r.l >> 31);
    return r;
}
// complex a b / 2^62 with b = (x, y) and ny = -y; |a| < 2^60, |b| < 2^62.1 (the
// four middle products stay below 2^63)
GQ_HD void fx_cmul30(gfx30 ar, gfx30 ai, gfx x, gfx y, gfx ny, long long &re, long long &im) {
    const long long mr = fx_mw(ar.h, x.l, fx_mw(ar.l, x.h, fx_mw(ai.h, ny.l, fx_mw(ai.l, ny.h, 1LL << 31))));
    const long long mi = fx_mw(ar.h, y.l, fx_mw(ar.l, y.h, fx_mw(ai.h, x.l, fx_mw(ai.l, x.h, 1LL << 31))));
    re = fx_mw(ar.h, x.h, fx_mw(ai.h, ny.h, (long long)(int)(mr >> 32)));
    im = fx_mw(ar.h, y.h, fx_mw(ai.h, x.h, (long long)(int)(mi >> 32)));
}

GQ_HD uint64_t fx_bits(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}
// v >> s for any unsigned count (64 and above give 0)
GQ_HD uint64_t fx_shr(uint64_t v, int s) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));   // the count is clamped, not wrapped
    return r;
#else
    return (unsigned)s > 63u ? 0 : v >> s;
#endif
}

// the 53-bit significand of a normal double
GQ_HD uint64_t fx_mant(uint64_t bits) { return (bits & 0xfffffffffffffull) | 0x10000000000000ull; }
GQ_HD int fx_expo(uint64_t bits) { return (int)(bits >> 52) & 0x7ff; }

// the biased exponent of x: 0 for zero only (1 for a subnormal number)
GQ_HD int fx_expo1(double x) {
    const uint64_t b = fx_bits(x);
    const int e = fx_expo(b);
    return e > 0 ? e : (b << 1) != 0;
}

// x 2^(1022 - e) 2^62 for |x| < 2^(e - 1022) (e: a biased exponent no smaller than x's), truncated
GQ_HD long long fx_from_double(double x, int e) {
    const uint64_t b = fx_bits(x);
    const int ex = fx_expo(b);
    const uint64_t m = ex ? fx_mant(b) : b & 0xfffffffffffffull;
    const long long v = (long long)fx_shr(m << 10, e + 1 - (ex ? ex : 1));
    return (long long)b < 0 ? -v : v;
}

// 2^62 / M for the significand M = m / 2^52 of m in [2^52, 2^53): an FP32
// reciprocal of M's leading 24 bits (22 bits kept as an integer Y) and one
// third-order step y (1 - e + e^2), e = M y - 1.  m Y is a 75-bit number whose
// leading bits are 2^74, so e comes exactly out of its low 64 bits.  Relative
// error below 2^-57.
GQ_HD long long fx_rcp(uint64_t m) {
    const unsigned mh = (unsigned)(m >> 32), ml = (unsigned)m;
    const unsigned fb = ((((mh << 3) | (ml >> 29))) & 0x7fffffu) | 0x3f800000u;
    unsigned Y;
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(fb)));
    Y = __float_as_uint(y + 2.0f) & 0x7fffffu;      // y + 2 in [2.5, 3]: y 2^22 in the fraction
#else
    float f, s;
    memcpy(&f, &fb, 4);
    s = 1.0f / f + 2.0f;
    memcpy(&Y, &s, 4);
    Y &= 0x7fffffu;
#endif
    const long long E = (long long)((uint64_t)ml * Y + ((uint64_t)(mh * Y) << 32));   // e 2^74
    const int e = (int)(E >> 37);                                                     // e 2^37
    const gfx c = fx_bal(fx_mw(e, e, -E));
    const long long t = fx_mw((int)Y, c.h, (long long)(int)(fx_mw((int)Y, c.l, 1LL << 31) >> 32));
    return fx_shl((long long)Y, 40) + (t >> 2);
}

// u = (re / w) 2^62 from w, |w|^2 = n2 and the radius' significand (R, 2^61) and
// biased exponent: re / M2 by fx_rcp, each component's significand shifted into
// the common format (a right shift for |u| < 2), complemented for a negative w (a
// unit of 2^-62 off) and multiplied.  The lowest bit of u is set so that no low
// word is -2^31, which has no negative.
GQ_HD void fx_ratio(double wx, double wy, uint64_t nb, gfx R, int er, gfx &ux, gfx &uy, gfx &nuy) {
    const gfx G = fx_bal(fx_shl(fx_mul(R, fx_bal(fx_rcp(fx_mant(nb)))), 2));   // 2^61 r / M
    const int k = er - fx_expo(nb) - 1023 - 1;
    auto comp = [&](uint64_t b) {
        const gfx x = fx_bal((long long)fx_shr(fx_mant(b) << 10, -(k + fx_expo(b))) ^ ((long long)b >> 63));
        return fx_bal(fx_shl(fx_mul(x, G), 4) | 1);
    };
    ux = comp(fx_bits(wx));
    nuy = comp(fx_bits(wy));
    uy.h = -nuy.h;
    uy.l = -nuy.l;
}

// (1/2) log x 2^57 relative to 2^(e_ref - 1023), for the bits of a normal x:
// Tang's table method (see gq_math.cuh) with t_j a 16-bit integer T_j / 2^16, so
// that r = m t_j - 1 comes exactly out of the low 64 bits of m T_j; then
// log1p(r) to r^4 with |r| < 2^-9.97, and the mean of the r^5 term as r^3 2^-20/30
// (what is left of it is below 2^-53.8, 2^-56 in the mean).  Each of the shifts
// truncates by half a unit on average; the table holds the compensation.
constexpr int kFxLogJ = 512;
struct FxLogTable {
    long long hl[kFxLogJ];   // -(1/2) log(T_j / 2^16) 2^57
    int t[kFxLogJ];
};
constexpr int kFxLogWords = kFxLogJ * 3;   // 32-bit words
GQ_HD long long fx_log_half(uint64_t bits, int e_ref, const long long *hl, const int *tj) {
    const uint64_t m = fx_mant(bits);
    const int j = (int)(bits >> 43) & (kFxLogJ - 1);
    const unsigned T = (unsigned)tj[j];
    const long long R = (long long)((uint64_t)(unsigned)m * T + ((uint64_t)((unsigned)(m >> 32) * T) << 32));   // r 2^68
    const gfx r = fx_bal(R);
    const long long S2 = fx_mw((int)(fx_mw(r.h, r.l, 0) >> 32), 2, fx_mw(r.h, r.h, 0));   // r^2 2^72
    const int p = 357913941 + 68 - (r.h >> 8);                                           // (1/6 - r/8 + 2^-20/30) 2^31
    const int rp = (int)(fx_mw(r.h, p, 0) >> 28);                                        // r p 2^39
    const int tail = (int)(fx_mw((int)(S2 >> 22), rp, 0) >> 32);                         // r^3 p 2^57
    long long f = hl[j] + (R >> 12) - (S2 >> 17) + tail;
    const int e = fx_expo(bits) - e_ref;
    // (log 2 / 2) 2^57 = 49946518145322874 (rounded)
    constexpr long long kC = 49946518145322874LL;
    constexpr int kCl = (int)(unsigned)(kC & 0xffffffff), kCh = (int)(kC >> 32) + (int)((unsigned)kCl >> 31);
    f = fx_mw(e, kCl, f);
    return f + fx_shl((long long)((unsigned)e * (unsigned)kCh), 32);
}

inline void fx_log_table_host(FxLogTable *T) {
    for (int j = 0; j < kFxLogJ; ++j) {
        const long double c = 1.0L + (j + 0.5L) / (long double)kFxLogJ;
        T->t[j] = (int)(65536.0L / c + 0.5L);
        T->hl[j] = (long long)floorl(-0.5L * logl((long double)T->t[j] / 65536.0L) * 0x1p57L + 1.0L);
    }
}
