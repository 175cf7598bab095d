// hg_pair64.cuh -- the FP64 path's pair law (acceleration, jerk and snap of a pair) and a
// pair's potential (host and device; the host form serves the CPU tests).
//
// GB300 has two FP64 lanes per SM: a warp-wide FP64 instruction holds its
// sub-partition's unit for 64 cycles, so a pair law of ~55 FP64 instructions takes
// ~3500 cycles per warp.  A 32 x 32 + 64-bit integer multiply-add takes two.  Hence only
//   the differences r, v, a, w = v - 3 alpha r and the sums of q r, q w and q u
// are FP64 instructions (21), and the rest runs on the integer pipes beside them:
//   R^2 = r^2 + eps^2, q = m / R^3, alpha = r.v / R^2,
//   u = a - 6 alpha v - gamma r, gamma = 3 (v^2 + r.a) / R^2 - 15 alpha^2.
//
// Integer numbers are 64-bit sizes with a sign and a binary exponent of their own: every
// product of a dot product and every component of u has its exponent, and the terms of
// a sum are shifted to the largest of them.  So a component of the sums is as good
// whatever the others are (thin discs, nearly aligned pairs).  The integers lose 2^-55 or
// so of the sizes of a component's terms and are rounded to FP64 once: a pair's terms are
// within 3 2^-53 of these sizes, where FP64 instructions throughout reach 8 (q r), 15
// (q w) and 16 (q u) 2^-53 (10^6 random pairs each, of seven kinds).  A factor of a product is
// split at its 32nd bit, X = h 2^32 + l, and X Y / 2^64 = h h' + (h l' + l h') / 2^32:
// three multiply-adds (l l' is below the last place).  Infinities, NaN and
// numbers near the ends of FP64's range are left to FP64 instructions (vectors_fp64); a
// component of u all of whose terms are below 2^-762 may count as zero.
//
// An evaluation of N = 32768 particles: 45.6 ms, the FP64 unit 83 % busy; with w in integers
// too (18 FP64 instructions) 49.1 ms; with u in FP64 instructions as well the unit alone would
// take 48 ms.  (One exponent for the three components of a vector and of a sum takes 36 ms,
// but holds small components in fewer bits than FP64 does.)
//
// The potential of a pair is one positive number, m / R: integers after the three
// differences, sums over kFold64 pairs in block fixed point.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "hg_internal.cuh"

namespace hg {
namespace p64 {

#if defined(__CUDACC__)
#define HG_P64 __device__ __forceinline__
#else
#define HG_P64 inline
#endif

constexpr int kSVec = 62;                 // scale of the potential's separation
constexpr int kSMass = 63;                // of its mass, in [1/4, 1/2)
constexpr int kSR2 = 2 * kSVec - 64;      // of r^2 and eps^2
constexpr int kSY = 61;                   // of y, in (1, 2]
constexpr int kFold64 = 32;               // pairs between additions to the total sums
constexpr int kSlack = 2;                 // its exponent is raised by this much more than needed
constexpr int kExpNone = -(1 << 28);      // exponent of zero

struct Limbs {
    int32_t h, l;
};

// Shifts by any count >= 0 (counts of 64 and more give zero or the sign).
HG_P64 int64_t sar(int64_t x, int s)
{
#if defined(__CUDA_ARCH__)
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return x >> (s < 63 ? s : 63);
#endif
}
HG_P64 uint64_t shr(uint64_t x, int s)
{
#if defined(__CUDA_ARCH__)
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return s < 64 ? x >> s : 0;
#endif
}
HG_P64 int clz32(uint32_t x)
{
#if defined(__CUDA_ARCH__)
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}
HG_P64 uint64_t dbits(double x)
{
    return (uint64_t)bits_of(x);
}
HG_P64 int imax(int a, int b) { return a > b ? a : b; }
HG_P64 int imin(int a, int b) { return a < b ? a : b; }
HG_P64 uint32_t umin(uint32_t a, uint32_t b) { return a < b ? a : b; }

// a b + c, one instruction (stated as such: from the C expression the compiler
// proves low limbs non-negative and falls back to 64 x 64-bit products).
HG_P64 int64_t mad(int32_t a, int32_t b, int64_t c)
{
#if defined(__CUDA_ARCH__)
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (int64_t)a * b + c;
#endif
}
HG_P64 uint64_t madu(uint32_t a, uint32_t b, uint64_t c)
{
#if defined(__CUDA_ARCH__)
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (uint64_t)a * b + c;
#endif
}
HG_P64 int32_t lo32(int64_t x) { return (int32_t)x; }
HG_P64 int32_t hi32(int64_t x) { return (int32_t)((uint64_t)x >> 32); }
HG_P64 int64_t word(int32_t hi, int32_t lo) { return (int64_t)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo); }
HG_P64 Limbs split(int64_t x) { return Limbs{hi32(x) + (int32_t)((uint32_t)lo32(x) >> 31), lo32(x)}; }
// H + floor(M / 2^32)
HG_P64 int64_t carry(int64_t H, int64_t M) { return mad(hi32(M), 1, H); }
// kRound in the cross sum rounds a product to nearest: errors without a preferred
// sign, since the sums run over many pairs whose terms cancel.
constexpr int64_t kRound = (int64_t)1 << 31;
HG_P64 int64_t mul(Limbs a, Limbs b) { return carry(mad(a.h, b.h, 0), mad(a.h, b.l, mad(a.l, b.h, kRound))); }
HG_P64 int64_t norm2(const Limbs (&a)[3])
{
    return mad(hi32(mad(a[2].h, a[2].l, mad(a[1].h, a[1].l, mad(a[0].h, a[0].l, kRound >> 1)))), 2,
               mad(a[2].h, a[2].h, mad(a[1].h, a[1].h, mad(a[0].h, a[0].h, 0))));
}

// Vector d as X times 2^(returned exponent - kSVec); low collects the smallest
// complemented high word seen (below 2^20: an infinity or NaN).  Components far
// below the largest shift to zero; a vector below 2^-958 counts as zero.
HG_P64 int vec(double d0, double d1, double d2, int64_t (&o)[3], uint32_t &low)
{
    const uint64_t b[3] = {dbits(d0), dbits(d1), dbits(d2)};
    uint32_t nh[3];   // 2047 - biased exponent in the top bits
#pragma unroll
    for (int k = 0; k < 3; ++k) nh[k] = ~(uint32_t)(b[k] >> 32) & 0x7fffffffu;
    const uint32_t nm = umin(umin(nh[0], nh[1]), nh[2]);
    low = umin(low, nm);
    const int ne = (int)(nm >> 20), base = ne > 2047 - 64 ? 192 - ne : -ne;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t hi = (uint32_t)((b[k] << (kSVec - 53)) >> 32);
        const uint64_t m = (uint64_t)word((int32_t)((hi & 0x1fffffffu) | 0x20000000u), (int32_t)((uint32_t)b[k] << (kSVec - 53)));
        const int32_t sg = (int32_t)(b[k] >> 32) >> 31;
        const uint64_t u = shr(m, base + (int)(nh[k] >> 20));
        o[k] = (int64_t)(u ^ (uint64_t)word(sg, sg)) - sg;
    }
    return 2047 - ne - 1022;
}

// eps^2 as a fraction in [1/2, 1) (scale kSR2) and its exponent; zero: fraction 0, no exponent;
// beyond FP64's range: an exponent that leaves q below it.
struct Soft {
    int64_t q;
    int e;
    double eps2;
};
inline
#if defined(__CUDACC__)
    __host__ __device__
#endif
    Soft soft(double eps2)
{
    Soft s{0, kExpNone, eps2};
    if (eps2 > 0.0) {
        int e;
        const bool finite = eps2 < INFINITY;
        const double f = frexp(finite ? eps2 : 1.0, &e);   // [1/2, 1)
        s.q = (int64_t)ldexp(f, kSR2);
        s.e = finite ? e : 8192;
    }
    return s;
}

// y = rho^(-1/2) (scale kSY, in (1, 2]) for rho in [2^62, 2^64) standing for rho / 2^64:
// the hardware FP32 reciprocal square root y0 (24 bits), then with e = 1 - rho y0^2
// (|e| < 2^-20, formed exactly enough modulo 2^64) the binomial series of
// (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + O(e^3), whose rest is below 2^-60.
HG_P64 int64_t rsqrt_q(uint64_t rho)
{
    const uint32_t r1 = (uint32_t)(rho >> 32), r0 = (uint32_t)rho;
#if defined(__CUDA_ARCH__)
    const uint32_t u = (uint32_t)__float2int_rn(rsqrt_approx(__uint2float_rn(r1)) * 0x1p45f);
#else
    const uint32_t u = (uint32_t)lrintf(1.0f / sqrtf((float)r1) * 0x1p45f);
#endif
    const uint64_t uu = madu(u, u, 0);                       // y0^2, scale 58
    const uint32_t a1 = (uint32_t)(uu >> 30), a0 = (uint32_t)uu & 0x3fffffffu;
    const uint64_t lo = madu(r1, a0, madu(r0, a1, 0) >> 2);
    const int64_t e = (int64_t)((1ull << 62) - ((madu(r1, a1, 0) << 2) + (lo >> 28)));   // scale 62
    const int32_t es = (int32_t)(e >> 12);
    const int32_t e2 = (int32_t)(mad(es, es, 0) >> 32);        // e^2, scale 68
    const int64_t d = (e >> 1) + ((3 * e2) >> 9);              // scale 62
    const int32_t dh = (int32_t)(d >> 16), dl = (int32_t)d & 0xffff;
    const int64_t c = mad((int32_t)u, dh, mad((int32_t)u, dl, 0) >> 16) >> 14;   // y0 d
    return word((int32_t)u + hi32(c), lo32(c));
}

// R^2 = r^2 + eps^2 = (rho / 2^64) 2^(2 hx) and y = (rho / 2^64)^(-1/2), from
// r^2 = rr 2^(er2 - kSR2), rr < 2^63.  Returns false (y = 1, hx = 0) for R^2 = 0 or below
// FP64's range.
template <bool GUARD>
HG_P64 bool inverse_radius(int64_t rr, int er2, const Soft &s, int64_t &y, int &hx)
{
    int e2 = imax(er2, s.e);
    uint64_t r2 = shr((uint64_t)rr, e2 - er2) + shr((uint64_t)s.q, e2 - s.e);
    bool ok = true;
    if (GUARD) {
        ok = r2 != 0 && e2 > -1074;
        r2 = ok ? r2 : (uint64_t)1 << kSR2;
        e2 = ok ? e2 : 0;
    }
    const int lz = clz32((uint32_t)(r2 >> 32));
    const int k = lz - ((lz ^ e2) & 1);
    y = rsqrt_q(r2 << k);
    hx = (e2 + 64 - kSR2 - k) >> 1;
    return ok;
}

// Mass in [1/4, 1/2) (scale kSMass) times 2^(returned exponent) (sign kept, zero exact).
HG_P64 int mass_limbs(double m, Limbs &o, uint32_t &low)
{
    const uint64_t b = dbits(m);
    const uint32_t hi = (uint32_t)(b >> 32), ah = hi & 0x7fffffffu;
    low = umin(low, ah ^ 0x7fffffffu);
    const int e = (int)(ah >> 20);
    const uint64_t f = ((uint64_t)((ah & 0xfffffu) | (e > 0 ? 0x100000u : 0u)) << 32) | (uint32_t)b;
    const int64_t u = (int64_t)(f << (kSMass - 54));
    o = split((int32_t)hi < 0 ? -u : u);
    return imax(e, 1) - 1021;
}

// Size of a normal double or zero: x 2^(e - 1085), the top bit of x at bit 62; zero is 0 with
// e = kExpZero, below any product's exponent.  A denormal number (x > 0 with kExpZero)
// counts for nothing beside the others; vectors_int bounds what it could have been.
constexpr int kExpZero = -8192;
struct Size {
    uint64_t x;
    int e;
};
HG_P64 Size size_of(double d)
{
    const uint64_t b = dbits(d);
    const uint32_t lo = (uint32_t)b, ah = (uint32_t)(b >> 32) & 0x7fffffffu;
    const uint32_t top = (ah & 0xfffffu) | umin(ah, 0x100000u);
    return Size{(uint64_t)word((int32_t)((top << 10) | (lo >> 22)), (int32_t)(lo << 10)),
                ah >= 0x100000u ? (int)(ah >> 20) : kExpZero};
}
HG_P64 int max_e(const Size (&s)[3]) { return imax(imax(s[0].e, s[1].e), s[2].e); }

// All bits of a sign: 0 or -1.
HG_P64 int32_t sign_of(double d) { return hi32((int64_t)dbits(d)) >> 31; }
HG_P64 int32_t sign_of(int64_t x) { return hi32(x) >> 31; }
// X + x or, for s = -1, X - x.
HG_P64 int64_t add_signed(int64_t X, uint64_t x, int32_t s) { return X + (int64_t)(x ^ (uint64_t)word(s, s)) - s; }

// x y / 2^64 and x^2 / 2^64 to within a unit, for x, y <= 2^63.
HG_P64 uint64_t mulu(uint64_t x, uint64_t y)
{
    const uint32_t h = (uint32_t)(x >> 32), l = (uint32_t)x, h2 = (uint32_t)(y >> 32), l2 = (uint32_t)y;
    return madu(h, h2, madu(h, l2, madu(l, h2, 0x80000000u)) >> 32);
}
HG_P64 uint64_t squ(uint64_t x)
{
    const uint32_t h = (uint32_t)(x >> 32), l = (uint32_t)x;
    return madu(h, h, madu(h, l, 0x40000000u) >> 31);
}

HG_P64 int clz64(uint64_t x)
{
#if defined(__CUDA_ARCH__)
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

// Number x 2^e (x > 0: top bit at bit 62; zero: any e, kExpNone from normal) with the sign s.
struct Number {
    uint64_t x;
    int e;
    int32_t s;
};
// X 2^e for |X| < 2^63, turned over for s = -1.
HG_P64 Number normal(int64_t X, int e, int32_t s)
{
    Number n;
    const int32_t sx = sign_of(X);
    const uint64_t x = (uint64_t)add_signed(0, (uint64_t)X, sx);
    const int z = clz64(x) - 1;
    n.x = x << z;
    n.e = z < 63 ? e - z : kExpNone;
    n.s = s ^ sx;
    return n;
}

// x 2^e for x = 0 or x in [2^32, 2^63).
HG_P64 Number normal_hi(uint64_t x, int e, int32_t s)
{
    const int z = clz32((uint32_t)(x >> 32)) - 1;
    return Number{x << z, e - z, s};
}

// Rounded to FP64; ok turns false for what is not zero and not a normal number.
HG_P64 double to_fp64(const Number &n, bool &ok)
{
    const int eb = n.e + (62 + 1022);                     // exponent field less one, before rounding
    ok = ok && ((uint32_t)eb < 2045u || hi32((int64_t)n.x) == 0);
    const uint64_t m = (n.x + 0x200u) >> 10;              // the top bit, in place 52, adds one to the field
    const uint64_t b = m + ((uint64_t)((uint32_t)imax(eb, 0) << 20 | ((uint32_t)n.s & 0x80000000u)) << 32);
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)b);
#else
    double d;
    memcpy(&d, &b, 8);
    return d;
#endif
}

// What a pair adds to the sums: q r, q w, q u.
struct Terms {
    double q, w[3], u[3];
};

// In FP64 instructions: any inputs.
template <bool GUARD>
HG_P64 void vectors_fp64(const double (&r)[3], const double (&v)[3], const double (&a)[3], double m, double eps2,
                         Terms &t)
{
    const double r2 = fma(r[2], r[2], fma(r[1], r[1], fma(r[0], r[0], eps2)));
#if defined(__CUDA_ARCH__)
    double rinv = rsqrt(r2);
#else
    double rinv = 1.0 / sqrt(r2);
#endif
    if (GUARD) rinv = (r2 > 0.0) ? rinv : 0.0;
    const double rinv2 = rinv * rinv;
    const double rv = fma(r[2], v[2], fma(r[1], v[1], r[0] * v[0]));
    const double v2ra = fma(r[2], a[2], fma(r[1], a[1], fma(r[0], a[0], fma(v[2], v[2], fma(v[1], v[1], v[0] * v[0])))));
    const double alpha = rv * rinv2;
    const double a3 = -3.0 * alpha, b3 = -3.0 * fma(alpha, alpha, v2ra * rinv2);
    t.q = m * rinv * rinv2;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t.w[k] = fma(a3, r[k], v[k]);
        t.u[k] = fma(b3, r[k], fma(a3 + a3, t.w[k], a[k]));
    }
}

// In integers but for w; returns false for what they do not hold.
template <bool GUARD>
HG_P64 bool vectors_int(const double (&r)[3], const double (&v)[3], const double (&a)[3], double m, const Soft &soft2,
                        Terms &t)
{
    const Size rs[3] = {size_of(r[0]), size_of(r[1]), size_of(r[2])};
    const Size vs[3] = {size_of(v[0]), size_of(v[1]), size_of(v[2])};
    const Size as[3] = {size_of(a[0]), size_of(a[1]), size_of(a[2])};
    const Size ms = size_of(m);
    const int32_t sr[3] = {sign_of(r[0]), sign_of(r[1]), sign_of(r[2])};
    const int32_t sv[3] = {sign_of(v[0]), sign_of(v[1]), sign_of(v[2])};
    const int32_t sa[3] = {sign_of(a[0]), sign_of(a[1]), sign_of(a[2])};
    const int er = max_e(rs), ev = max_e(vs);
    // Here and below, ok holds the numbers to a range in which denormal components (below
    // 2^-1022) have no part of 2^-62 in any sum: components below 2^500, dot products with a
    // term of 2^-460 or more, alpha and gamma below 2^260, u with a term of 2^-700 or more
    // (or all terms zero).
    bool ok = imax(imax(er, ev), max_e(as)) < 1023 + 500 && ms.e < 2047;

    // r^2 = rr 2^(2 er - 2105): products below 2^62 (2^60 or more for the largest), halved.
    uint64_t rr = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) rr += shr(squ(rs[k].x), 2 * (er - rs[k].e) + 1);
    int64_t yi;
    int hx;
    const bool apart = inverse_radius<GUARD>((int64_t)rr, 2 * er - 2045, soft2, yi, hx);
    const uint64_t y = (uint64_t)yi << 1;                  // 1/R = y 2^(-62 - hx), y in (2^62, 2^63]
    const uint64_t y2 = squ(y), y3 = (3 * y2) >> 1;        // 1/R^2 = y2 2^(-60 - 2 hx), 3/R^2 = y3 2^(-59 - 2 hx)

    // r.v, below 3 2^61 in units of 2^(e1 - 2105); v^2 + r.a, below 6 2^60 in units of 2^(e2 - 2104)
    int p[3], c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = rs[k].e + vs[k].e;
        c[k] = rs[k].e + as[k].e;
    }
    const int e1 = imax(imax(p[0], p[1]), p[2]), e2 = imax(imax(imax(c[0], c[1]), c[2]), 2 * ev);
    ok = ok && (uint32_t)e1 >= 2046u - 460u && (uint32_t)e2 >= 2046u - 460u;   // (or negative)
    const int32_t s0 = sr[0] ^ sv[0];
    int64_t X = (int64_t)shr(mulu(rs[0].x, vs[0].x), e1 - p[0] + 1), Z = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (k > 0) X = add_signed(X, shr(mulu(rs[k].x, vs[k].x), e1 - p[k] + 1), sr[k] ^ sv[k] ^ s0);
        Z += (int64_t)shr(squ(vs[k].x), e2 - 2 * vs[k].e + 2);
        Z = add_signed(Z, shr(mulu(rs[k].x, as[k].x), e2 - c[k] + 2), sr[k] ^ sa[k]);
    }
    const Number rv = normal(X, e1 - 2105, s0), va = normal(Z, e2 - 2104, 0);

    // 3 alpha = al3 2^ea, al3 < 3 2^60; alpha = al 2^(ea - 1), al <= 2^61
    const uint64_t al3 = mulu(rv.x, y3), al = mulu(rv.x, y2);
    const int ea = rv.e + 64 - 59 - 2 * hx;
    // gamma = ga 2^eg: its parts below 3 2^60 and 15 2^57
    const int eg1 = va.e + 64 - 59 - 2 * hx, eg2 = 2 * ea + 63, eg = imax(eg1, eg2);
    const int64_t G = add_signed(-(int64_t)shr(mulu((al << 1) + (al >> 1), al3 << 1), eg - eg2),
                                 shr(mulu(va.x, y3), eg - eg1), va.s);
    ok = ok && imax(ea, eg) < 260 - 62;
    const int32_t sg = sign_of(G);
    const uint64_t ga = (uint64_t)add_signed(0, (uint64_t)G, sg);

    const double a3 = to_fp64(normal_hi(al3, ea, ~rv.s), ok);

#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t.w[k] = fma(a3, r[k], v[k]);
        // u: a_k below 2^61, 6 alpha v_k below 3 2^59, gamma r_k below 2^62, in units of 2^(eu + 2)
        const int fa = as[k].e - 1085, fw = ea + vs[k].e + (65 - 1085), fg = eg + rs[k].e + (64 - 1085);
        const int eu = imax(imax(fa, fw - 2), fg - 2);
        ok = ok && (uint32_t)(eu + 4096) >= 4096u - 700u;   // (or below -4096)
        const Number u = normal(add_signed(add_signed((int64_t)shr(as[k].x, eu - fa + 2),
                                                      shr(mulu(al3, vs[k].x), eu - fw + 2), ~(rv.s ^ sv[k] ^ sa[k])),
                                           shr(mulu(ga, rs[k].x), eu - fg + 2), ~(sg ^ sr[k] ^ sa[k])),
                                eu + 2, sa[k]);
        t.u[k] = to_fp64(u, ok);
    }
    // m / R^3 = m (1/R) (1/R^2), below 2^62
    t.q = to_fp64(normal((int64_t)mulu(mulu(ms.x, y), y2 << 1), ms.e - 1080 - 3 * hx, sign_of(m)), ok);
    if (GUARD && !apart) t.q = 0.0;   // a pair at zero distance
    return ok;
}

// i-particle: position, velocity, acceleration.
struct Body {
    double x, y, z, vx, vy, vz, ax, ay, az;
};

// Sums of one i-particle on one lane: c over up to kFold64 pairs, s of the finished ones (so
// that a large term meets few roundings at its own size).
struct Sums {
    double c[9], s[9];
    int cnt;         // pairs in c
#if !defined(__CUDACC__)
    bool bad;        // host checks: an infinity or NaN among the pairs (shown in every sum)
#endif
};

HG_P64 void clear(Sums &a)
{
    for (int k = 0; k < 9; ++k) a.c[k] = a.s[k] = 0.0;
    a.cnt = 0;
#if !defined(__CUDACC__)
    a.bad = false;
#endif
}

// One pair: j-particle (position, mass, velocity, acceleration) on i-particle d.
template <bool GUARD>
HG_P64 void pair(const Body &d, double jx, double jy, double jz, double jm, double jvx, double jvy, double jvz,
                 double jax, double jay, double jaz, const Soft &soft2, Sums &acc)
{
    const double r[3] = {jx - d.x, jy - d.y, jz - d.z};
    const double v[3] = {jvx - d.vx, jvy - d.vy, jvz - d.vz};
    const double a[3] = {jax - d.ax, jay - d.ay, jaz - d.az};
    Terms t;
    if (!vectors_int<GUARD>(r, v, a, jm, soft2, t)) vectors_fp64<GUARD>(r, v, a, jm, soft2.eps2, t);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        acc.c[k] = fma(t.q, r[k], acc.c[k]);
        acc.c[3 + k] = fma(t.q, t.w[k], acc.c[3 + k]);
        acc.c[6 + k] = fma(t.q, t.u[k], acc.c[6 + k]);
    }
#if !defined(__CUDACC__)
    for (int k = 0; k < 3; ++k) acc.bad = acc.bad || !isfinite(r[k]) || !isfinite(v[k]) || !isfinite(a[k]);
    acc.bad = acc.bad || !isfinite(jm);
#endif
}

HG_P64 void fold(Sums &a)
{
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        a.s[k] += a.c[k];
        a.c[k] = 0.0;
    }
    a.cnt = 0;
}
HG_P64 void count_pair(Sums &a)
{
    if (++a.cnt == kFold64) fold(a);
}

// All sums in s.
HG_P64 void finish(Sums &a)
{
    fold(a);
#if !defined(__CUDACC__)
    for (double &x : a.s)
        if (a.bad) x = NAN;
#endif
}

// 2^e for |e| <= 1022.
HG_P64 double exp2i(int e)
{
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)(e + 1023) << 52);
#else
    return ldexp(1.0, e);
#endif
}

// s + H 2^e: one rounding of H and one of the sum for |e| <= 960, else in two
// steps (beyond 2^+-2040 the factor is that).
HG_P64 double add_scaled(double s, int64_t H, int e)
{
    const double h = (double)H;
    if (e >= -960 && e <= 960) return fma(h, exp2i(e), s);
    const int c = imin(imax(e, -2040), 2040), c1 = c >> 1;
    return s + (h * exp2i(c1)) * exp2i(c - c1);
}

// Potential of one pair, m / R (R^2 = r^2 + eps^2): H 2^(E - kSPot) sums the pairs
// since the last fold (rounded to nearest in these units), s the rest.  A term
// enters below 2^(kSPot - kPotHead): kFold64 of them stay below 2^62.
constexpr int kSPot = kSMass + kSY - 64, kPotHead = 4;
struct Potential {
    int64_t H;
    int E;
    double s;
    uint32_t low;
};

HG_P64 void clear(Potential &a)
{
    a.H = 0;
    a.E = kExpNone;
    a.s = 0.0;
    a.low = 0x7fffffffu;
}

// m 2^em: the j-particle's mass (mass_limbs).  Coincident particles without
// softening give infinity, as 1 / r does; skip leaves the pair out.
HG_P64 void pair_potential(double dx, double dy, double dz, Limbs m, int em, bool skip, const Soft &soft2,
                           Potential &acc)
{
    int64_t rx[3];
    const int er = vec(dx, dy, dz, rx, acc.low);
    const Limbs r[3] = {split(rx[0]), split(rx[1]), split(rx[2])};
    int64_t y;
    int hx;
    const bool ok = inverse_radius<true>(norm2(r), 2 * er, soft2, y, hx);
    if (!ok && !skip) acc.s = INFINITY;
    int64_t t = mul(m, split(y));                    // in [1/4, 1], scale kSPot
    t = (ok && !skip) ? t : 0;
    const int e = em - hx, need = e + kPotHead;
    if (need > acc.E && t != 0) {
        acc.H = sar(acc.H, need + kSlack - acc.E);
        acc.E = need + kSlack;
    }
    acc.H += (sar(t, imax(acc.E - e - 1, 0)) + 1) >> 1;
}

HG_P64 void fold_fp64(Potential &a)
{
    a.s = add_scaled(a.s, a.H, a.E - kSPot);
    a.H = 0;
}

}  // namespace p64
}  // namespace hg
