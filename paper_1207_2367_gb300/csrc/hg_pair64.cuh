// hg_pair64.cuh -- the FP64 path's pair law on the integer pipes: acceleration,
// jerk and snap of a pair, and a pair's potential, at FP64 accuracy or better
// without the FP64 unit (host and device; the host form serves the CPU test).
//
// GB300 has two FP64 lanes per SM: a warp-wide FP64 instruction holds its
// sub-partition's unit for 64 cycles, so the ~55 FP64 instructions of a pair are
// ~3500 cycles per warp.  A 32 x 32 + 64-bit integer multiply-add takes two.  Here
// only the differences r_j - r_i, v_j - v_i, a_j - a_i (nine subtractions, whose
// operands have any exponents) are FP64 instructions; everything after them is
// block fixed point.
//
// Numbers are 64-bit integers in units of 2^-58 ("Q58", |x| < 4) beside a binary
// exponent; each of the vectors r, v, a has one exponent (its largest component
// lies in [1/2, 1)), so a component is exact to 2^-58 of the vector's size.  A
// factor of a product is split into limbs x = h 2^29 + l (h: signed, 31 bits), and
// x y = h h' + (h l' + l h') 2^-29 in the same units (l l' is below them): three
// multiply-adds, dot products and sums accumulating inside them.
//
// The pair law, with R^2 = r^2 + eps^2 and n = r / R (so that every factor is
// bounded by the vectors it multiplies):
//   lambda = n.v, nu = n.a, w = v - 3 lambda n,
//   u = a - 3 nu n - (6 lambda w + 3 (v^2 + lambda^2) n) / R,
//   A = q r, J = q w, S = q u with q = m / R^3.
// Sums: three running exponents per i-particle (A, J, S), raised when a larger
// term arrives, so that q is shifted once per sum (rounded to nearest) and the
// products accumulate in 64-bit integers; every kFold64 pairs they are added to
// FP64 sums.  Errors per pair are 2^-55 or less of |A|, |J|, |S|, against a few
// 2^-53 of the FP64 instructions.
#pragma once

#include <math.h>
#include <stdint.h>

#include "hg_internal.cuh"

namespace hg {
namespace p64 {

#if defined(__CUDACC__)
#define HG_P64 __device__ __forceinline__
#else
#define HG_P64 inline
#endif

constexpr int kLimb = 29;                 // bits of the low limb
constexpr int kQ = 2 * kLimb;             // fraction bits
constexpr int32_t kLow = (1 << kLimb) - 1;
constexpr int kFoldM = 8;                 // pairs between carries of the cross sums into the high sums
constexpr int kFold64 = 32;               // pairs between additions to the FP64 sums (a multiple of kFoldM)
// A term enters its sum with |q'| < 2^(58 - kHead): the high sums of kFold64
// terms (|x| < 3.5) stay below 3.5 * 32 * 2^(58 - 3) < 2^62, the cross sums of
// kFoldM below 8 (3.5 + 2^-3) 2^58 < 2^63.
constexpr int kHead = 3;
constexpr int kExpNone = -(1 << 28);      // exponent of an empty sum
constexpr uint32_t kHiInf = 0x7ff00000u;  // high word of an infinity

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
HG_P64 uint32_t umax(uint32_t a, uint32_t b) { return a > b ? a : b; }

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
HG_P64 Limbs split(int64_t x) { return Limbs{(int32_t)(x >> kLimb), (int32_t)x & kLow}; }
// The same with the low limb in [-2^28, 2^28), of x + kEven: the dropped products of
// low limbs then have no preferred sign.
constexpr int64_t kEven = (int64_t)1 << (kLimb - 1);
HG_P64 Limbs split_even(int64_t x) { return Limbs{(int32_t)(x >> kLimb), ((int32_t)x & kLow) - (int32_t)kEven}; }
HG_P64 int64_t join(Limbs x) { return mad(x.h, 1 << kLimb, x.l); }
HG_P64 int64_t carry(int64_t H, int64_t M) { return H + (M >> kLimb); }
// kRound in the cross sum rounds a product to nearest: errors without a preferred
// sign, since the sums run over many pairs whose terms cancel.
constexpr int64_t kRound = (int64_t)1 << (kLimb - 1);
HG_P64 int64_t mul(Limbs a, Limbs b, int64_t round = kRound)
{
    return carry(mad(a.h, b.h, 0), mad(a.h, b.l, mad(a.l, b.h, round)));
}
HG_P64 int64_t sqr(Limbs a) { return mad(a.h, a.h, 0) + (mad(a.h, a.l, 0) >> (kLimb - 1)); }
HG_P64 int64_t dot(const Limbs (&a)[3], const Limbs (&b)[3])
{
    return carry(mad(a[2].h, b[2].h, mad(a[1].h, b[1].h, mad(a[0].h, b[0].h, 0))),
                 mad(a[2].h, b[2].l, mad(a[2].l, b[2].h, mad(a[1].h, b[1].l, mad(a[1].l, b[1].h,
                     mad(a[0].h, b[0].l, mad(a[0].l, b[0].h, kRound)))))));
}
HG_P64 int64_t norm2(const Limbs (&a)[3])
{
    return mad(a[2].h, a[2].h, mad(a[1].h, a[1].h, mad(a[0].h, a[0].h, 0))) +
           (mad(a[2].h, a[2].l, mad(a[1].h, a[1].l, mad(a[0].h, a[0].l, 0))) >> (kLimb - 1));
}

// Vector d as limbs times 2^(returned exponent); top collects the largest high
// word seen (infinities and NaN).  Components far below the largest shift to
// zero; a vector below 2^-958 counts as zero.
HG_P64 int vec(double d0, double d1, double d2, Limbs (&o)[3], uint32_t &top)
{
    const uint64_t b[3] = {dbits(d0), dbits(d1), dbits(d2)};
    uint32_t ah[3];
    for (int k = 0; k < 3; ++k) ah[k] = (uint32_t)(b[k] >> 32) & 0x7fffffffu;
    const uint32_t am = umax(umax(ah[0], ah[1]), ah[2]);
    top = umax(top, am);
    const int e = (int)(am >> 20), es = e < 64 ? 255 : e;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint64_t m = ((uint64_t)((ah[k] & 0xfffffu) | 0x100000u) << 32) | (uint32_t)b[k];
        const uint64_t u = shr(m << (kQ - 53), es - (int)(ah[k] >> 20));
        const int32_t sg = ((int32_t)(b[k] >> 32) >> 31) | 1;
        o[k].h = (int32_t)(u >> kLimb) * sg;
        o[k].l = ((int32_t)u & kLow) * sg;
    }
    return e - 1022;
}

// eps^2 as a fraction in [1/2, 1) (Q58) and its exponent; zero: fraction 0, no exponent.
struct Soft {
    int64_t q;
    int e;
};
inline
#if defined(__CUDACC__)
    __host__ __device__
#endif
    Soft soft(double eps2)
{
    Soft s{0, kExpNone};
    if (eps2 > 0.0) {
        int e;
        const double f = frexp(eps2, &e);   // [1/2, 1)
        s.q = (int64_t)ldexp(f, kQ);
        s.e = e;
    }
    return s;
}

// y = rho^(-1/2) (Q58, in (1, 2]) for rho in [2^62, 2^64) standing for rho / 2^64:
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
    const uint64_t uu = madu(u, u, 0);                       // y0^2, Q58
    const uint32_t a1 = (uint32_t)(uu >> 30), a0 = (uint32_t)uu & 0x3fffffffu;
    const uint64_t lo = madu(r1, a0, madu(r0, a1, 0) >> 2);
    const int64_t e = (int64_t)((1ull << 62) - ((madu(r1, a1, 0) << 2) + (lo >> 28)));   // Q62
    const int32_t es = (int32_t)(e >> 12);
    const int32_t e2 = (int32_t)(mad(es, es, 0) >> 32);        // e^2, Q68
    const int64_t d = (e >> 1) + ((3 * e2) >> 9);              // Q62
    const int32_t dh = (int32_t)(d >> 16), dl = (int32_t)d & 0xffff;
    const int64_t c = mad((int32_t)u, dh, mad((int32_t)u, dl, 0) >> 16);   // y0 d, Q75
    return mad((int32_t)u, 1 << 29, c >> 17);
}

// R^2 = r^2 + eps^2 = (rho / 2^64) 2^(2 hx) and y = (rho / 2^64)^(-1/2), from
// r^2 = rr 2^er2.  Returns false (y = 1, hx = 0) for R^2 = 0 or below FP64's range.
template <bool GUARD>
HG_P64 bool inverse_radius(int64_t rr, int er2, const Soft &s, int64_t &y, int &hx)
{
    int e2 = imax(er2, s.e);
    uint64_t r2 = shr((uint64_t)rr, e2 - er2) + shr((uint64_t)s.q, e2 - s.e);   // < 4
    bool ok = true;
    if (GUARD) {
        ok = r2 != 0 && e2 > -1074;
        r2 = ok ? r2 : (uint64_t)1 << kQ;
        e2 = ok ? e2 : 0;
    }
    const int lz = clz32((uint32_t)(r2 >> 32));
    const int k = lz - ((lz ^ e2) & 1);
    y = rsqrt_q(r2 << k);
    hx = (e2 + 64 - kQ - k) >> 1;
    return ok;
}

// Mass as limbs in [1/4, 1/2) times 2^(returned exponent) (sign kept, zero exact).
HG_P64 int mass_limbs(double m, Limbs &o, uint32_t &top)
{
    const uint64_t b = dbits(m);
    const uint32_t hi = (uint32_t)(b >> 32), ah = hi & 0x7fffffffu;
    top = umax(top, ah);
    const int e = (int)(ah >> 20);
    const uint32_t mh = (ah & 0xfffffu) | (e > 0 ? 0x100000u : 0u);
    const uint32_t ml = (uint32_t)b;
    const int32_t sg = ((int32_t)hi >> 31) | 1;
    // 53 bits times 2^4: limbs of 28 and 29 bits
    o.h = (int32_t)((mh << 7) | (ml >> 25)) * sg;
    o.l = (int32_t)((ml & 0x1ffffffu) << 4) * sg;
    return imax(e, 1) - 1021;
}

// i-particle: position, velocity, acceleration.
struct Body {
    double x, y, z, vx, vy, vz, ax, ay, az;
};

// Sums of one i-particle on one lane.  Component c: (H[c] + M[c] 2^-29) 2^(E[c/3] - 58).
struct Sums {
    int64_t H[9], M[9];
    int E[3];
    double s[9];
    int cnt;         // pairs since the last addition to s
    uint32_t top;    // largest high word of a difference or mass (infinities, NaN)
};

HG_P64 void clear(Sums &a)
{
    for (int c = 0; c < 9; ++c) {
        a.H[c] = a.M[c] = 0;
        a.s[c] = 0.0;
    }
    for (int g = 0; g < 3; ++g) a.E[g] = kExpNone;
    a.cnt = 0;
    a.top = 0;
}

// q 2^-s rounded to nearest (s >= 1), low limb in [-2^28, 2^28).
HG_P64 Limbs scaled(int64_t q, int s)
{
    const int64_t t = sar(q, s - 1) + ((1 << kLimb) + 1);
    return Limbs{(int32_t)(t >> (kLimb + 1)), ((int32_t)((uint32_t)t >> 1) & kLow) - (1 << (kLimb - 1))};
}

HG_P64 void add_term(Sums &a, int g, Limbs q, const Limbs (&x)[3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a.H[3 * g + k] = mad(q.h, x[k].h, a.H[3 * g + k]);
        a.M[3 * g + k] = mad(q.h, x[k].l, mad(q.l, x[k].h, a.M[3 * g + k]));
    }
}

// Rare: a term larger than any before moves the sums to its exponent.
HG_P64 void raise(Sums &a, const int (&need)[3])
{
#pragma unroll
    for (int g = 0; g < 3; ++g) {
        const int d = imax(need[g] - a.E[g], 0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a.H[3 * g + k] = sar(carry(a.H[3 * g + k], a.M[3 * g + k]), d);
            a.M[3 * g + k] = d > 0 ? 0 : (int64_t)(a.M[3 * g + k] & kLow);
        }
        a.E[g] += d;
    }
}

// One pair: j-particle (position, mass, velocity, acceleration) on i-particle d.
template <bool GUARD>
HG_P64 void pair(const Body &d, double jx, double jy, double jz, double jm, double jvx, double jvy, double jvz,
                 double jax, double jay, double jaz, const Soft &soft2, Sums &acc)
{
    Limbs r[3], v[3], a[3], m;
    const int er = vec(jx - d.x, jy - d.y, jz - d.z, r, acc.top);
    const int ev = vec(jvx - d.vx, jvy - d.vy, jvz - d.vz, v, acc.top);
    const int ea = vec(jax - d.ax, jay - d.ay, jaz - d.az, a, acc.top);
    const int em = mass_limbs(jm, m, acc.top);

    int64_t y;
    int hx;
    const bool ok = inverse_radius<GUARD>(norm2(r), 2 * er, soft2, y, hx);
    const Limbs yl = split(y);
    // q = m y^3 2^(em - 3 hx), in [1/4, 4)
    const int64_t q = mul(split(mul(split(mul(m, yl)), yl)), yl);
    if (GUARD && !ok) return;   // a pair at zero distance

    // n = r / R = n' 2^-hn: below R = 2 r or so n' stays of order one (|n'| < 1.75).
    const int s1 = imin(hx - er, 1), hn = hx - er - s1;
    const Limbs ys = split(y >> s1);
    Limbs n[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) n[k] = split_even(mul(r[k], ys, kRound + (kEven << kLimb)));

    // lambda = lam 2^-hn, nu = nu' 2^-hn, |lam| and |nu'| < 3.1 (< 1.75 for hn = 0)
    const int64_t lam = dot(n, v), nu = dot(n, a);
    const Limbs ll = split(lam);
    Limbs w[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)                          // |w| <= 2 |v| < 3.5
        w[k] = split_even(join(v[k]) + kEven - sar(3 * mul(ll, n[k]), 2 * hn));
    // kappa = (v^2 + lambda^2) y / 2 <= 6.  The part of u along 1 / R has the length
    // |6 (lambda y w + kappa n)| <= 6 kappa (its square over y^2 v^4 |n|^2, with c the
    // cosine of v and n, is (3 + 6 c^2 - 15 |n|^2 c^2)^2 + 36 c^2 (1 - c^2)), and at
    // most 32 kappa |n| / |n'|; |a - 3 nu n| <= 2 |a| < 3.5.
    const int64_t kap = mul(split((norm2(v) + sar(sqr(ll), 2 * hn)) >> 1), yl);
    const int64_t lam1 = mul(ll, yl);
    const int bk = 64 - kQ - imin(clz32((uint32_t)((uint64_t)kap >> 32)), 7);   // kappa < 2^bk, bk >= -1
    const int ec = 2 * ev - hx - hn;
    const int eu = imax(ea + 2, ec + bk + 2 + imin(hn, 3));
    const int sa = eu - ea, sz = eu - ec - 1;            // >= 2, >= bk + 1
    const Limbs c1 = split(sar(3 * nu, sa + 2 * hn) + sar(3 * kap, sz) + 1);   // < 2.9
    const Limbs c2 = split(sar(3 * lam1, sz));                            // <= 3
    Limbs u[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {                        // |u| < 2.4
        const int64_t H = mad(c2.h, w[k].h, mad(c1.h, n[k].h, 0));
        const int64_t M = mad(c2.h, w[k].l, mad(c2.l, w[k].h, mad(c1.h, n[k].l, mad(c1.l, n[k].h, 0))));
        u[k] = split_even(sar(join(a[k]), sa) + kEven - carry(H, M));
    }

    // The sums: |q| < 2^b (Q58), brought below 2^-kHead in each sum's units.
    const int eq = em - 3 * hx;
    const uint32_t qh = (uint32_t)((uint64_t)(q < 0 ? -q : q) >> 32);
    const int b = 64 - kQ - imin(clz32(qh), 8) + eq + kHead;
    const int need[3] = {b + er, b + ev, b + eu};
    if (imax(imax(need[0] - acc.E[0], need[1] - acc.E[1]), need[2] - acc.E[2]) > 0) raise(acc, need);
    add_term(acc, 0, scaled(q, acc.E[0] - eq - er), r);
    add_term(acc, 1, scaled(q, acc.E[1] - eq - ev), w);
    add_term(acc, 2, scaled(q, acc.E[2] - eq - eu), u);
}

// Cross sums into the high sums (every kFoldM pairs).
HG_P64 void fold_cross(Sums &a)
{
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        a.H[c] = carry(a.H[c], a.M[c]);
        a.M[c] &= kLow;
    }
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

// The integer sums into the FP64 sums (every kFold64 pairs, and at the end); the
// cross sums have been carried.  x 2^e in two exact steps (the last may round).
HG_P64 void fold_fp64(Sums &a)
{
#pragma unroll
    for (int g = 0; g < 3; ++g) {
        const int e = imin(imax(a.E[g] - kQ, -2040), 2040), e1 = e >> 1;
        const double f1 = exp2i(e1), f2 = exp2i(e - e1);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a.s[3 * g + k] += ((double)a.H[3 * g + k] * f1) * f2;
            a.H[3 * g + k] = 0;
        }
    }
    a.cnt = 0;
}

HG_P64 void count_pair(Sums &a)
{
    a.cnt += 1;
    if ((a.cnt & (kFoldM - 1)) == 0) {
        fold_cross(a);
        if (a.cnt == kFold64) fold_fp64(a);
    }
}

// All sums in s; an infinity or NaN among the inputs gives NaN.
HG_P64 void finish(Sums &a)
{
    fold_cross(a);
    fold_fp64(a);
    if (a.top >= kHiInf)
        for (int c = 0; c < 9; ++c) a.s[c] = NAN;
}

// Potential of one pair, m / R (R^2 = r^2 + eps^2): H 2^(E - 58) sums the pairs
// since the last fold (rounded to nearest in these units), s the rest.
struct Potential {
    int64_t H;
    int E;
    double s;
    uint32_t top;
};

HG_P64 void clear(Potential &a)
{
    a.H = 0;
    a.E = kExpNone;
    a.s = 0.0;
    a.top = 0;
}

// m 2^em: the j-particle's mass (mass_limbs).  Coincident particles without
// softening give infinity, as 1 / r does; skip leaves the pair out.
HG_P64 void pair_potential(double dx, double dy, double dz, Limbs m, int em, bool skip, const Soft &soft2,
                           Potential &acc)
{
    Limbs r[3];
    const int er = vec(dx, dy, dz, r, acc.top);
    int64_t y;
    int hx;
    const bool ok = inverse_radius<true>(norm2(r), 2 * er, soft2, y, hx);
    if (!ok && !skip) acc.s = INFINITY;
    int64_t t = mul(m, split(y));                    // in [1/4, 1]
    t = (ok && !skip) ? t : 0;
    const int e = em - hx, need = e + 1;             // |t| 2^-1 <= 1/2: kFold64 terms stay below 2^62
    if (need > acc.E && t != 0) {
        acc.H = sar(acc.H, need - acc.E);
        acc.E = need;
    }
    acc.H += (sar(t, imax(acc.E - e - 1, 0)) + 1) >> 1;
}

HG_P64 void fold_fp64(Potential &a)
{
    const int e = imin(imax(a.E - kQ, -2040), 2040), e1 = e >> 1;
    a.s += ((double)a.H * exp2i(e1)) * exp2i(e - e1);
    a.H = 0;
}

}  // namespace p64
}  // namespace hg
