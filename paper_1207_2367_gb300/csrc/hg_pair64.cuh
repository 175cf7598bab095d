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
// Numbers are 64-bit integers: x stands for X = x 2^S with a scale S known at each
// place, beside a binary exponent; each of the vectors r, v, a has one exponent (its
// largest component lies in [1/2, 1)), so a component is exact to 2^-62 of the
// vector's size.  A factor of a product is split at its 32nd bit, X = h 2^32 + l with
// l signed (its word as it is; h takes the carry), and X Y / 2^64 = h h' +
// (h l' + l h') / 2^32: the word of a sum is its quotient, so a product is four
// multiply-adds (l l' is below its last place) and no shift, dot products and sums
// accumulating inside them.  The scales below are chosen so that |h| < 2^31 and
// that the cross sums stay below 2^63 (the |h| of the factors add up to < 2^32).
//
// The pair law, with R^2 = r^2 + eps^2 and n = r / R (so that every factor is
// bounded by the vectors it multiplies):
//   lambda = n.v, nu = n.a, w = v - 3 lambda n,
//   u = a - 3 nu n - (6 lambda w + 3 (v^2 + lambda^2) n) / R,
//   A = q r, J = q w, S = q u with q = m / R^3.
// Sums: three running exponents per i-particle (A, J, S), raised when a larger
// term arrives, so that q is shifted once per sum (rounded to nearest) and the
// products accumulate in 96-bit integers; every kFold64 pairs they are added to
// FP64 sums (small blocks: the lanes' integers are added first, hg_eval.cu).  Errors per pair are 2^-55 or less of |A|, |J|, |S|, against a few
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

constexpr int kSVec = 62;                 // scale of r, v, a
constexpr int kSMass = 63;                // of the mass, in [1/4, 1/2)
constexpr int kSR2 = 2 * kSVec - 64;      // of r^2 and eps^2
constexpr int kSY = 61;                   // of y, in (1, 2]
constexpr int kSQ = 61;                   // of q, in [1/4, 4)
constexpr int kFold64 = 32;               // pairs between additions to the FP64 sums
// A term enters its sum with |q'| < 2^kBitsQ: the high sums of kFold64 terms stay
// below 32 * 2^(59 - 32) * 3.5 * 2^29 < 2^63; a dropped l l' is 2^-56 of the largest
// term.  A sum's exponent is raised by kSlack more than a larger term needs, so that
// it moves less often.
constexpr int kBitsQ = 59, kSlack = 2;
constexpr int kExpNone = -(1 << 28);      // exponent of an empty sum
static_assert(kFold64 == 32, "the room of align_sums");

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
HG_P64 int64_t sqr(Limbs a) { return mad(hi32(mad(a.h, a.l, kRound >> 1)), 2, mad(a.h, a.h, 0)); }
HG_P64 int64_t dot(const Limbs (&a)[3], const Limbs (&b)[3])
{
    return carry(mad(a[2].h, b[2].h, mad(a[1].h, b[1].h, mad(a[0].h, b[0].h, 0))),
                 mad(a[2].h, b[2].l, mad(a[2].l, b[2].h, mad(a[1].h, b[1].l, mad(a[1].l, b[1].h,
                     mad(a[0].h, b[0].l, mad(a[0].l, b[0].h, kRound)))))));
}
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

// eps^2 as a fraction in [1/2, 1) (scale kSR2) and its exponent; zero: fraction 0, no exponent.
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
        s.q = (int64_t)ldexp(f, kSR2);
        s.e = e;
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
// r^2 = rr 2^er2.  Returns false (y = 1, hx = 0) for R^2 = 0 or below FP64's range.
template <bool GUARD>
HG_P64 bool inverse_radius(int64_t rr, int er2, const Soft &s, int64_t &y, int &hx)
{
    // The largest component is 2^(kSVec - 1) or more, and so is its share of rr; the
    // dropped l l' of the others must not take rr below that: R >= |r| holds with hx.
    constexpr int64_t kLeast = (int64_t)1 << (2 * (kSVec - 1) - 64);
    rr = rr > 0 && rr < kLeast ? kLeast : rr;
    int e2 = imax(er2, s.e);
    uint64_t r2 = shr((uint64_t)rr, e2 - er2) + shr((uint64_t)s.q, e2 - s.e);   // < 4
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

// i-particle: position, velocity, acceleration.
struct Body {
    double x, y, z, vx, vy, vz, ax, ay, az;
};

// Sums of one i-particle on one lane.  Component c: (H[c] + M[c] / 2^32) in units of
// 2^(E[c/3] - unit(c/3)), beside s.
struct Sums {
    int64_t H[9];
    uint32_t M[9];
    int E[3];
    double s[9];
    int cnt;         // pairs since the last addition to s
    uint32_t low;    // smallest complemented high word of a difference or mass (infinities, NaN)
};
// Scales of r, w, u where they enter the sums; the sums' units.
constexpr int kSW = 61, kSU = 61;
HG_P64 int unit(int g) { return kSQ + (g == 0 ? kSVec : g == 1 ? kSW : kSU) - 64; }

HG_P64 void clear(Sums &a)
{
    for (int c = 0; c < 9; ++c) {
        a.H[c] = 0;
        a.M[c] = 0u;
        a.s[c] = 0.0;
    }
    for (int g = 0; g < 3; ++g) a.E[g] = kExpNone;
    a.cnt = 0;
    a.low = 0x7fffffffu;
}

// q 2^-s rounded to nearest (s >= 1), as limbs.
HG_P64 Limbs scaled(int64_t q, int s) { return split((sar(q, s - 1) + 1) >> 1); }

HG_P64 void add_term(Sums &a, int g, Limbs q, const Limbs (&x)[3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int64_t m = mad(q.h, x[k].l, mad(q.l, x[k].h, (int64_t)(uint64_t)a.M[3 * g + k]));
        a.M[3 * g + k] = (uint32_t)lo32(m);
        a.H[3 * g + k] = carry(mad(q.h, x[k].h, a.H[3 * g + k]), m);
    }
}

// (H, M) 2^-d; from d = 32 on the rest below H's last place is dropped.
HG_P64 void shift_sum(int64_t &H, uint32_t &M, int d)
{
    M = d < 32 ? (uint32_t)lo32((int64_t)shr((uint64_t)word(lo32(H), (int32_t)M), d)) : 0u;
    H = sar(H, d);
}

// A term larger than the sums' units allow moves them to its exponent.
HG_P64 void raise(Sums &a, const int (&need)[3])
{
#pragma unroll
    for (int g = 0; g < 3; ++g) {
        const int d = need[g] > a.E[g] ? need[g] + kSlack - a.E[g] : 0;
        a.E[g] += d;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            shift_sum(a.H[3 * g + k], a.M[3 * g + k], d);
        }
    }
}

// One pair: j-particle (position, mass, velocity, acceleration) on i-particle d.
template <bool GUARD>
HG_P64 void pair(const Body &d, double jx, double jy, double jz, double jm, double jvx, double jvy, double jvz,
                 double jax, double jay, double jaz, const Soft &soft2, Sums &acc)
{
    int64_t rx[3], vx[3], ax[3];
    Limbs r[3], v[3], a[3], m;
    const int er = vec(jx - d.x, jy - d.y, jz - d.z, rx, acc.low);
    const int ev = vec(jvx - d.vx, jvy - d.vy, jvz - d.vz, vx, acc.low);
    const int ea = vec(jax - d.ax, jay - d.ay, jaz - d.az, ax, acc.low);
    const int em = mass_limbs(jm, m, acc.low);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r[k] = split(rx[k]);
        v[k] = split(vx[k]);
        a[k] = split(ax[k]);
    }

    int64_t y;
    int hx;
    const bool ok = inverse_radius<GUARD>(norm2(r), 2 * er, soft2, y, hx);
    if (GUARD && !ok) return;   // a pair at zero distance
    const Limbs yl = split(y);
    // q = m y^3 2^(em - 3 hx), in [1/4, 4): (m y) and y^2 lifted to scales 62 and 60
    const int64_t q = mul(split(mul(m, yl) << 2), split(sqr(yl) << 2)) << 3;

    // n = r / R = n' 2^-hn: below R = 2 r or so n' stays of order one (|n'| < 1.75).
    const int s1 = imin(hx - er, 1), hn = hx - er - s1;
    const Limbs ys = split(y >> s1);
    Limbs n[3];                                          // scale 59
#pragma unroll
    for (int k = 0; k < 3; ++k) n[k] = split(mul(r[k], ys));

    // lambda = lam 2^-hn, nu = nu' 2^-hn, |lam| and |nu'| < 3.1 (< 1.75 for hn = 0), scale 57
    const int64_t lam = dot(n, v), nu = dot(n, a);
    const Limbs ll = split(lam << 4);                    // scale 61
    const Limbs l3 = split(sar(3 * lam, 2 * hn) << 3);   // 3 lambda 2^-hn < 5.3, scale 60
    Limbs w[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)                          // |w| <= 2 |v| < 3.5
        w[k] = split((vx[k] >> (kSVec - kSW)) - (mul(l3, n[k]) << (kSW - 55)));
    // kappa = (v^2 + lambda^2) y / 2 <= 6, scale 58.  The part of u along 1 / R has the
    // length |6 (lambda y w + kappa n)| <= 6 kappa (its square over y^2 v^4 |n|^2, with c
    // the cosine of v and n, is (3 + 6 c^2 - 15 |n|^2 c^2)^2 + 36 c^2 (1 - c^2)), and at
    // most 32 kappa |n| / |n'|; |a - 3 nu n| <= 2 |a| < 3.5.
    const int64_t kap = mul(split(norm2(v) + (sar(sqr(ll), 2 * hn) << 2)), yl);
    const int64_t lam1 = mul(ll, yl);                    // scale 58
    const int bk = 6 - imin(clz32((uint32_t)hi32(kap)), 7);   // kappa < 2^bk, bk >= -1
    const int ec = 2 * ev - hx - hn;
    const int eu = imax(ea + 2, ec + bk + 2 + imin(hn, 3));
    const int sa = eu - ea, sz = eu - ec - 1;            // >= 2, >= bk + 1
    const Limbs c1 = split(sar(12 * nu, sa + 2 * hn - 2) + (sar(3 * kap, sz) << 3) + 4);   // < 2.9, scale 61
    const Limbs c2 = split(sar(3 * lam1, sz) << 1);                                        // <= 3, scale 59
    Limbs u[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {                        // |u| < 2.4, formed at scale 56, lifted
        const int64_t H = mad(c2.h, w[k].h, mad(c1.h, n[k].h, 0));
        const int64_t M = mad(c2.h, w[k].l, mad(c2.l, w[k].h, mad(c1.h, n[k].l, mad(c1.l, n[k].h, kRound))));
        u[k] = split(sar(ax[k], sa + kSVec - kSU) - (carry(H, M) << (kSU - 56)));
    }

    // The sums: |q| < 2^b, brought below 2^kBitsQ in each sum's units.
    const int eq = em - 3 * hx;
    const int b = 64 - imin(clz32((uint32_t)hi32(q < 0 ? -q : q)), 5) - kBitsQ + eq;
    const int need[3] = {b + er, b + ev, b + eu};
    if (imax(imax(need[0] - acc.E[0], need[1] - acc.E[1]), need[2] - acc.E[2]) > 0) raise(acc, need);
    add_term(acc, 0, scaled(q, acc.E[0] - eq - er), r);
    add_term(acc, 1, scaled(q, acc.E[1] - eq - ev), w);
    add_term(acc, 2, scaled(q, acc.E[2] - eq - eu), u);
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

// The high sums into the FP64 sums.
HG_P64 void fold_fp64(Sums &a)
{
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        a.s[c] = add_scaled(a.s[c], a.H[c], a.E[c / 3] - unit(c / 3));
        a.H[c] = 0;
    }
    a.cnt = 0;
}

// Component c of the integer sums alone.
HG_P64 double sum_of(int64_t H, uint32_t M, int E, int c)
{
    const int e = E - unit(c / 3);
    return add_scaled(add_scaled(0.0, H, e), (int64_t)(uint64_t)M, e - 32);
}

// Sums of lanes that together took `all` pairs, the same number each and none folded
// yet: moves this lane's to the exponents E, with room for the total.
HG_P64 void align_sums(Sums &a, const int (&E)[3], int all)
{
    const int room = all > kFold64 ? 32 - clz32((uint32_t)(all - 1)) - 5 : 0;
#pragma unroll
    for (int c = 0; c < 9; ++c) shift_sum(a.H[c], a.M[c], E[c / 3] + room - a.E[c / 3]);
    for (int g = 0; g < 3; ++g) a.E[g] = E[g] + room;
}
HG_P64 void add_sums(int64_t &H, uint32_t &M, int64_t H2, uint32_t M2)
{
    const uint64_t m = (uint64_t)M + M2;
    M = (uint32_t)m;
    H += H2 + (int64_t)(m >> 32);
}

HG_P64 void count_pair(Sums &a)
{
    if (++a.cnt == kFold64) fold_fp64(a);
}

// All sums in s; an infinity or NaN among the inputs gives NaN.
HG_P64 void finish(Sums &a)
{
    fold_fp64(a);
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        a.s[c] = add_scaled(a.s[c], (int64_t)(uint64_t)a.M[c], a.E[c / 3] - unit(c / 3) - 32);
        if (a.low < 0x100000u) a.s[c] = NAN;
    }
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
