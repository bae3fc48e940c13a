// Pair terms of the FP64 real space from tables: force factor and energy of the erfc Coulomb and of the
// Lennard-Jones 12-6 potential as functions of u = r^2, to about 2^-52 per pair;
// the separations in 64-bit fixed point.
//
// Why: GB300 issues an FP64 instruction over about 76 clocks of a warp and scheduler, and sqrt, the
// division, exp and erfc of a pair are about 90 of them (the pair kernels kept the FP64 pipe 85 % busy).
//
// Each octave of u below the cutoff (eight of them) has 128 segments; in a segment the force factor is its
// Taylor polynomial of degree 8 about the centre (half a segment is at most 2^-8 of u, so each further
// term is about 2^-7 smaller, and the first one left out below 2^-58), the constant term in FP64 and the
// rest, at most 2^-5 of it, in float-float with FP32 for the small terms: two FP64 additions.  The
// segment and the argument come from the bits of u, and u from integers: the separation of two coordinates
// in fixed point is exact, box vectors included, and its square is nine 32-bit multiplications to 2^-59 of the
// cutoff's.  With dU/du = -f/2 the energy is the integral of the same polynomial from the segment's centre: the
// value there in FP64, the rest, 2^-8 of it, in float-float.  What is left in FP64 per pair is thirteen
// instructions: the charge product, one FMA and two additions of the force factor, three roundings of separations,
// four FMAs of the force and the virial, two of the energies.  (All of an energy in float-float took eleven, 1137
// against 1185 us for an NPT run of four steps at N = 2e4, with sums 4 to 20 times further off than FP64 pair terms
// give: 1.6e-11 against 1.1e-12 for E_lj there; with the constant terms in FP64 they are as near.)
//
// Coulomb derivatives: with B_0 = erfc(s r)/r and B_n = ((2n-1) B_{n-1} + (2a)^n e^{-a u} / sqrt(pi a)) / u
// (a = alpha, s = sqrt(alpha)) the force factor is B_1 and d B_n / du = -B_{n+1} / 2: a recurrence of
// positive terms.
#pragma once

#include "rbe_fix64.cuh"

namespace rbe {

constexpr int kPairSegBits = 7;                          // segments per octave: 2^7
constexpr int kPairOctaves = 8;
constexpr int kPairSegs = kPairOctaves << kPairSegBits;  // 1024
constexpr int kPairPlanes = 4;                           // 16-byte planes per part
constexpr size_t kPairTabBytes = 16 * (size_t)kPairSegs * 2 * kPairPlanes;

// One 16-byte plane entry, as four words.
struct alignas(16) PairWord {
    uint32_t w[4];
};

__host__ __device__ __forceinline__ void pair_put(PairWord& p, int j, float f) { p.w[j] = fx_bits(f); }

__host__ __device__ inline void pair_split(double x, float& h, float& l)
{
    h = (float)x;
    l = (float)(x - (double)h);
}

__host__ __device__ inline void pair_put_double(PairWord& p, int j, double x)
{
    unsigned long long b;
#ifdef __CUDA_ARCH__
    b = (unsigned long long)__double_as_longlong(x);
#else
    __builtin_memcpy(&b, &x, 8);
#endif
    p.w[j] = (uint32_t)b;
    p.w[j + 1] = (uint32_t)(b >> 32);
}

__host__ __device__ __forceinline__ double pair_get_double(const PairWord& p, int j)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)p.w[j + 1], (int)p.w[j]);
#else
    const unsigned long long b = ((unsigned long long)p.w[j + 1] << 32) | p.w[j];
    double x;
    __builtin_memcpy(&x, &b, 8);
    return x;
#endif
}

// a b for a, b as sums of two doubles.
__host__ __device__ inline double2 pair_dd_mul(double2 a, double2 b)
{
    const double p = a.x * b.x, e = fma(a.x, b.x, -p) + (a.x * b.y + a.y * b.x), s = p + e;
    return make_double2(s, e - (s - p));
}

// Segment `seg` of the table whose octaves end at 2^top, both parts (Coulomb, LJ): coefficients c[k] of the
// polynomial in tau in [-1, 1] and the energy e0 at the centre.  Planes (kPairSegs entries each):
// {c0 FP64, e0 FP64}, {c1 h, l, c2 h, l}, {c3 h, l, c4 h, l}, {c5, c6, c7, c8}.
__host__ __device__ inline void pair_segment(PairWord* t, int seg, int top, double alpha, double lj_s2, double lj_e24,
                                             double lj_e4)
{
    const double base = ldexp(1.0, top - kPairOctaves + (seg >> kPairSegBits));
    const double h = base * ldexp(1.0, -kPairSegBits - 1);
    const double u = base * (1.0 + (double)(seg & ((1 << kPairSegBits) - 1)) * ldexp(1.0, -kPairSegBits)) + h;
    // x = sqrt(alpha u) and x^2 with their rounding errors put back: erfc and exp amplify them by 2 x^2
    const double r = sqrt(u), iu = 1.0 / u, au = alpha * u, aul = fma(alpha, u, -au), x = sqrt(au);
    const double dx = (fma(-x, x, au) + aul) / (2.0 * x), ga = exp(-au) * (1.0 - aul);
    const double ex = ga / sqrt(kPi * alpha);
    // erfc / r with the rounding errors of the root and the quotient put back too
    const double er = erfc(x), de = -1.12837916709551257390 * ga * dx, q0 = er / r, dr = fma(-r, r, u) / (2.0 * r);
    double c[9], e0 = q0 + ((fma(-q0, r, er) + de) - q0 * dr) / r, B = e0, a2 = 1.0, f = 1.0;
    for (int n = 1; n <= 9; ++n) {
        a2 *= 2.0 * alpha;
        B = ((2 * n - 1) * B + a2 * ex) * iu;
        c[n - 1] = f * B;
        f *= -0.5 * h / (double)n;
    }
    for (int part = 0; part < 2; ++part) {
        if (part == 1) {
            // the sixth power of y = s^2 / u to about 2^-100: a segment's constants serve all its pairs, and their
            // errors do not average out
            const double2 i1 = make_double2(iu, fma(-u, iu, 1.0) * iu), y = pair_dd_mul(i1, make_double2(lj_s2, 0.0));
            const double2 y3 = pair_dd_mul(pair_dd_mul(y, y), y), y6 = pair_dd_mul(y3, y3);
            const double2 a3 = pair_dd_mul(y3, i1), a6 = pair_dd_mul(y6, i1);
            const double hu = h * iu;
            double p7 = 2.0 * lj_e24 * a6.x, p4 = -lj_e24 * a3.x;  // u^-7 and u^-4 terms of f
            e0 = lj_e4 * ((y6.x - y3.x) + (y6.y - y3.y));
            c[0] = lj_e24 * ((2.0 * a6.x - a3.x) + (2.0 * a6.y - a3.y));
            for (int k = 0; k < 9; ++k) {
                if (k > 0) c[k] = p7 + p4;
                p7 *= -hu * (7 + k) / (double)(k + 1);
                p4 *= -hu * (4 + k) / (double)(k + 1);
            }
        }
        PairWord* p = t + (size_t)part * kPairPlanes * kPairSegs + seg;
        auto two = [&](int plane, int j, double x) {
            float fh, fl;
            pair_split(x, fh, fl);
            pair_put(p[(size_t)plane * kPairSegs], j, fh);
            pair_put(p[(size_t)plane * kPairSegs], j + 1, fl);
        };
        pair_put_double(p[0], 0, c[0]);
        pair_put_double(p[0], 2, e0);
        two(1, 0, c[1]);
        two(1, 2, c[2]);
        two(2, 0, c[3]);
        two(2, 2, c[4]);
        for (int k = 5; k < 9; ++k) pair_put(p[3 * (size_t)kPairSegs], k - 5, (float)c[k]);
    }
}

struct FF {
    float h, l;
};

// a b + c.  ANY: any sizes (TwoSum); otherwise |c| is at least |a b| (Fast2Sum): the Coulomb
// polynomial, whose coefficients all have their full size, while those of the LJ part pass through zero.
template <bool ANY>
__host__ __device__ __forceinline__ FF ff_fma(FF a, FF b, FF c)
{
    const float p = RBE_MUL(a.h, b.h);
    float e = RBE_FMA(a.h, b.h, -p);
    e = RBE_FMA(a.h, b.l, e);
    e = RBE_FMA(a.l, b.h, e);
    FF r;
    r.h = RBE_ADD(c.h, p);
    float d;
    if (ANY) {
        const float bb = RBE_ADD(r.h, -c.h);
        d = RBE_ADD(RBE_ADD(c.h, -RBE_ADD(r.h, -bb)), RBE_ADD(p, -bb));
    } else {
        d = RBE_ADD(RBE_ADD(c.h, -r.h), p);
    }
    r.l = RBE_ADD(d, RBE_ADD(e, c.l));
    return r;
}

__host__ __device__ __forceinline__ FF ff_mul(FF a, FF b)
{
    FF r;
    r.h = RBE_MUL(a.h, b.h);
    r.l = RBE_FMA(a.l, b.h, RBE_FMA(a.h, b.l, RBE_FMA(a.h, b.h, -r.h)));
    return r;
}

// s += x (TwoSum of the high parts)
__host__ __device__ __forceinline__ void ff_acc(FF& s, FF x)
{
    const float t = RBE_ADD(s.h, x.h), bb = RBE_ADD(t, -s.h);
    const float e = RBE_ADD(RBE_ADD(s.h, -RBE_ADD(t, -bb)), RBE_ADD(x.h, -bb));
    s.h = t;
    s.l = RBE_ADD(s.l, RBE_ADD(x.l, e));
}

// A double's top 48 bits as a float-float, by its bits; below 2^-103 zero (the low part keeps every bit that is at
// least a float's smallest step), above the float range undefined.
// ANY false: at least 2^-103 by the caller's word.
template <bool ANY = true>
__host__ __device__ __forceinline__ FF ff_of(uint32_t hi, uint32_t lo)
{
    const uint32_t sign = hi & 0x80000000u, e = (hi >> 20) & 0x7ffu;
    const uint32_t m = ((hi & 0xFFFFFu) << 3) | (lo >> 29);  // 23 bits
    FF r;
    r.h = fx_float(sign | ((e - 896u) << 23) | m);
    // the next 24 bits as a fraction, times the unit 2^(e - 1023 - 23) of the high part
    const float rest = RBE_MUL(RBE_MUL(fx_i2f((int)((lo >> 5) & 0xFFFFFFu)), 0x1.0p-24f), fx_float((e - 919u) << 23));
    r.l = fx_float(fx_bits(rest) | sign);
    if (ANY && e < 920u) r.h = r.l = 0.0f;
    return r;
}

// A float's value as a double, by its bits (zero and subnormal give a value below 2^-126).
__host__ __device__ __forceinline__ double float_as_double(float f)
{
    const uint32_t b = fx_bits(f);
    const uint32_t hi = (((b & 0x7fffffffu) >> 3) + 0x38000000u) | (b & 0x80000000u);
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)(b << 29));
#else
    const unsigned long long x = ((unsigned long long)hi << 32) | (b << 29);
    double d;
    __builtin_memcpy(&d, &x, 8);
    return d;
#endif
}

// Separations as integers: coordinates in units of 2^-s, modulo 2^64, with s such that the cutoff is in
// [2^61, 2^62): exact for every coordinate above rc / 512 in size (its last bit is a multiple of the unit),
// and so are the differences, box vectors added, of a pair near the cutoff or below.  r^2 is counted in
// 2^(64 - 2 s): the cutoff's square is in [2^58, 2^60).
constexpr int kPairDrop = 11;  // bits of a separation left out where it becomes a double

struct PairUnit {
    int s;                   // the unit's exponent
    int e;                   // r^2 with z leading zeros has the binary exponent e - z
    int base;                // of the table's segments
    unsigned long long rc2;  // the cutoff's square
};

// The tables' range.  Coulomb: segments up to alpha u = 40 (there a force factor of cutoffs up to 1e4 is above
// 2^-97, where ff_of keeps all of it; half a segment's alpha h is 0.16, for a series good to 2^-42 of itself);
// pairs beyond are evaluated directly, as those below the table are.
inline int pair_segs(double alpha, int top)
{
    const double u = 40.0 / alpha;
    if (!(u < std::ldexp(1.0, top))) return kPairSegs;
    const int e = std::ilogb(u), oct = e - (top - kPairOctaves);
    return oct < 0 ? 0 : (oct << kPairSegBits) + (int)((std::ldexp(u, -e) - 1.0) * (1 << kPairSegBits));
}

// LJ: coefficients below 2^100 at the table's inner end, terms above 2^-97 at its outer end, and above 2^-58 where
// the force passes through zero (a constant term there is a small part of them).
inline bool pair_lj_fits(double s2, double e24, int top)
{
    const double in = std::ldexp(1.0, top - kPairOctaves), out = std::ldexp(1.0, top), yi = s2 / in, yo = s2 / out;
    const double big = 50.0 * std::fabs(e24) * std::pow(yi, 6) / s2, far = std::fabs(e24) * yo * yo * yo / out;
    return std::isfinite(big) && big < 1e30 && big * yi < 1e30 && far > 0x1.0p-97 && std::fabs(e24) / s2 > 0x1.0p-56;
}

inline PairUnit pair_unit(double rc, int top)
{
    PairUnit u;
    u.s = 61 - std::ilogb(rc);
    u.e = 127 - 2 * u.s;
    u.base = ((u.e - top + kPairOctaves) << kPairSegBits) - (1 << kPairSegBits);
    const double m = std::ldexp(rc, u.s - 61);  // rc in [1, 2)
    u.rc2 = (unsigned long long)std::ldexp(m * m, 58);
    return u;
}

// x in units of 2^-s, modulo 2^64, rounded to the nearest (finite x).
__host__ __device__ __forceinline__ unsigned long long pair_fixed(unsigned long long bits, int s)
{
    const int e = (int)(bits >> 52) & 0x7ff;
    const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = e - 1075 + s;
    unsigned long long v = 0;
    if (e != 0 && sh >= 0 && sh < 64) v = m << sh;
    else if (e != 0 && sh < 0 && sh >= -54) v = ((m >> (-sh - 1)) + 1) >> 1;
    return bits >> 63 ? 0ull - v : v;
}

// The square sum of three separations (below 2^63 in size), times 2^-64: from the signed 32-bit halves,
// without the squares of the low ones (a quarter in the mean), rounded down after adding `start` 2^-31.
constexpr unsigned long long kPairHalf = 3ull << 29;  // the mean of what is left out: sums over pairs are unbiased
__host__ __device__ __forceinline__ unsigned long long pair_r2(long long x, long long y, long long z,
                                                               unsigned long long start = 0)
{
    const int xl = (int)x, yl = (int)y, zl = (int)z;
    const int xh = (int)(x >> 32) - (xl >> 31), yh = (int)(y >> 32) - (yl >> 31), zh = (int)(z >> 32) - (zl >> 31);
    const long long mid = (long long)mad_wide(xh, xl, mad_wide(yh, yl, mad_wide(zh, zl, start)));
    return mad_wide(xh, xh, mad_wide(yh, yh, mad_wide(zh, zh, (unsigned long long)(mid >> 31))));
}

// The segment of u = r^2 and its argument tau = h + l (to 2^-46); seg is outside [0, kPairSegs) where u is.
struct PairArg {
    int seg;
    FF tau;
    float half;         // half the segment's half width
    uint32_t hi, lo;    // u normalised, the first bit set
    int e;              // and its binary exponent
};

__host__ __device__ __forceinline__ int pair_clz(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}

__host__ __device__ __forceinline__ PairArg pair_arg(unsigned long long n, int e, int base)
{
    PairArg a;
    const int z = pair_clz((uint32_t)(n >> 32));  // 32 and a segment far below for n < 2^32
    n <<= z;
    a.hi = (uint32_t)(n >> 32);
    a.lo = (uint32_t)n;
    a.e = e - z;
    a.seg = (int)(a.hi >> (31 - kPairSegBits)) - (z << kPairSegBits) + base;
    // the mantissa bits below the segment's: the first 23, and the next 23
    constexpr int k = 31 - kPairSegBits - 23;
    a.tau.h = RBE_FMA(2.0f, fx_float(((a.hi >> k) & 0x7FFFFFu) | 0x3F800000u), -3.0f);
    // (and half of their last, the mean of what is below)
    a.tau.l = RBE_FMA(fx_float((((a.hi << (23 - k)) | (a.lo >> (9 + k))) & 0x7FFFFFu) | 0x3F800000u), 0x1.0p-22f,
                      0x1.0p-46f - 0x1.0p-22f);
    // half width 2^(e - kPairSegBits - 1), halved
    a.half = fx_float((uint32_t)(a.e + 127 - kPairSegBits - 2) << 23);
    return a;
}

// One part (0: Coulomb, 1: LJ) from its table planes: the force factor as c0 + q, the energy as e0 + de, |de| at most
// about 2^-8 of it where it has its full size.
template <int PART>
__host__ __device__ __forceinline__ void pair_eval(const PairWord* t, const PairArg& a, double& c0, FF& q, double& e0,
                                                   FF& de)
{
    const PairWord* p = t + PART * kPairPlanes * kPairSegs + a.seg;
    const PairWord w0 = p[0], w1 = p[kPairSegs], w2 = p[2 * kPairSegs], w3 = p[3 * kPairSegs];
    const FF tau = a.tau;
    const FF c1{fx_float(w1.w[0]), fx_float(w1.w[1])}, c2{fx_float(w1.w[2]), fx_float(w1.w[3])};
    const FF c3{fx_float(w2.w[0]), fx_float(w2.w[1])}, c4{fx_float(w2.w[2]), fx_float(w2.w[3])};
    const float c5 = fx_float(w3.w[0]), c6 = fx_float(w3.w[1]), c7 = fx_float(w3.w[2]), c8 = fx_float(w3.w[3]);
    const float s = RBE_FMA(RBE_FMA(RBE_FMA(c8, tau.h, c7), tau.h, c6), tau.h, c5);
    constexpr bool ANY = PART == 1;
    q = ff_fma<ANY>(FF{s, 0.0f}, tau, c4);
    q = ff_fma<ANY>(q, tau, c3);
    q = ff_fma<ANY>(q, tau, c2);
    q = ff_fma<ANY>(q, tau, c1);
    q = ff_mul(q, tau);
    c0 = pair_get_double(w0, 0);
    e0 = pair_get_double(w0, 2);
    // -half tau (c0 + tau (c1 / 2 + tau (c2 / 3 + tau (c3 / 4 + ...))))
    float si = RBE_FMA(RBE_MUL(c6, 1.0f / 7.0f), tau.h, RBE_MUL(c5, 1.0f / 6.0f));
    si = RBE_FMA(si, tau.h, RBE_MUL(c4.h, 0.2f));
    si = RBE_FMA(si, tau.h, RBE_MUL(c3.h, 0.25f));
    const FF third{(float)(1.0 / 3.0), (float)(1.0 / 3.0 - (double)(float)(1.0 / 3.0))};
    FF in = ff_fma<ANY>(FF{si, 0.0f}, tau, ff_mul(c2, third));
    in = ff_fma<ANY>(in, tau, FF{RBE_MUL(0.5f, c1.h), RBE_MUL(0.5f, c1.l)});
    in = ff_fma<ANY>(in, tau, ff_of<ANY>(w0.w[1], w0.w[0]));  // (pair_segs)
    de = ff_mul(in, FF{RBE_MUL(-a.half, tau.h), RBE_MUL(-a.half, tau.l)});
}

// The same with the energy as one float-float (2^-45 of it).
template <int PART>
__host__ __device__ __forceinline__ void pair_eval(const PairWord* t, const PairArg& a, double& c0, FF& q, FF& energy)
{
    double e0;
    FF de;
    pair_eval<PART>(t, a, c0, q, e0, de);
    pair_split(e0, energy.h, energy.l);
    ff_acc(energy, de);
}

// ---------------------------------------------------------------------------------
// Device side: the table in shared memory and the accumulation of one pair.
#ifdef __CUDACC__

// Warps of an FP64 pair block: one block per SM, its warps share the table.  From a list 16 (an NPT run of four
// steps at N = 2e4: 1147 us; 18 warps 1166, 20 1194, 24 1328: fewer registers and less L1 beside the table); the
// water's cell search, mostly loads and FP32, 24 (3000 molecules: 1710 us with 16, 1717 with 18, 1625 with 20, 1602).
#ifndef RBE_PAIR64_WARPS
#define RBE_PAIR64_WARPS 16
#endif
#ifndef RBE_WATER_PAIR_WARPS
#define RBE_WATER_PAIR_WARPS 24
#endif
constexpr int kPair64Warps = RBE_PAIR64_WARPS, kWaterPairWarps = RBE_WATER_PAIR_WARPS;

// The FP64 pair kernels' constants beside PairConst.
struct Pair64Const {
    const PairWord* tab;  // device table, NULL: direct evaluation (cutoff or LJ sizes outside the table's range)
    unsigned segs;        // its usable segments (pair_segs)
    PairUnit unit;
    double scale;         // 2^(kPairDrop - s), the unit of the separations as doubles
    int lj;
    double alpha, sa, two_sa_pi, qk, s2, e4, e24;
};

// Sums of one lane: the particle's force and over all particles of the warp the virial (its trace, or its
// diagonal), separations in units; and the energies.
template <bool DIAG>
struct Pair64Sums {
    double fx, fy, fz;
    double w[DIAG ? 3 : 1];
    double ecd, eld;  // energies: the table's constant terms, and the pairs evaluated directly
    FF ec, el;        // the polynomials' rest, small beside them
};

__device__ __forceinline__ FF ff_of_double(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    return (hi & 0x7ff00000u) == 0u ? FF{0.0f, 0.0f} : ff_of<false>(hi, lo);  // (charge_fits)
}

// A charge product that float-floats hold to 48 bits: zero, or between 2^-60 and 2^60.
__device__ __forceinline__ bool charge_fits(double q)
{
    const uint32_t e = ((uint32_t)__double2hiint(q) >> 20) & 0x7ffu;
    return e == 0u || (e > 963u && e < 1083u);
}

// d / 2^11 (at most 2^51) rounded to an integer, as a double: one FP64 addition (the conversion of a 64-bit
// integer is two conversions and an FMA on the FP64 pipe).  The rounding is 2^-52 of the cutoff at most, as much
// as FP64 coordinates have at four times the cutoff.
__device__ __forceinline__ double pair_double(long long d)
{
    const long long v = (d + (1 << (kPairDrop - 1))) >> kPairDrop;
    return __dadd_rn(__longlong_as_double(v + 0x4338000000000000ll), -0x1.8p52);
}

// A pair below the table (r under 1/16 of the cutoff at least) or beyond its range: the force factor and
// the energies (Coulomb, LJ).  Not inlined: rare, and its registers are not the evaluation's.
static __device__ __noinline__ double3 pair_direct(double r2, double qq, double sa, double two_sa_pi, double alpha,
                                                   double s2, double e24, double e4)
{
    const double r = sqrt(r2), inv_r = 1.0 / r, inv_r2 = inv_r * inv_r;
    const double coul = qq * inv_r, er = erfc(sa * r);
    const double sr2 = s2 * inv_r2, sr6 = sr2 * sr2 * sr2;
    return make_double3(coul * (er + two_sa_pi * r * exp(-alpha * r2)) * inv_r2 + e24 * (2.0 * sr6 * sr6 - sr6) * inv_r2,
                        coul * er, e4 * (sr6 * sr6 - sr6));
}

// One pair: separation d (from i to the neighbour) and n = r^2 < rc^2 in units, qq the charge product with the
// Coulomb constant.  The table's force factor: qq (c0 + q) + (d0 + p), the two large terms in one FP64 FMA, the
// small ones in float-float first.
template <bool DIAG>
__device__ __forceinline__ void pair64_add(const PairWord* __restrict__ tab, const Pair64Const& pc, bool lj, long long dxi,
                                           long long dyi, long long dzi, unsigned long long n, double qq,
                                           Pair64Sums<DIAG>& s)
{
    const PairArg a = pair_arg(n, pc.unit.e, pc.unit.base);
    double dx = pair_double(dxi), dy = pair_double(dyi), dz = pair_double(dzi);
    double f, r2;
    if (pc.tab && (unsigned)a.seg < pc.segs && charge_fits(qq)) {
        FF q, de;
        double e0;
        pair_eval<0>(tab, a, f, q, e0, de);
        const FF qf = ff_of_double(qq);
        s.ecd = fma(qq, e0, s.ecd);
        ff_acc(s.ec, ff_mul(de, qf));
        q = ff_mul(q, qf);
        double d0 = 0.0;
        if (lj) {
            FF p;
            pair_eval<1>(tab, a, d0, p, e0, de);
            s.eld += e0;
            ff_acc(s.el, de);
            ff_acc(q, p);
        }
        f = (fma(f, qq, d0) + float_as_double(q.h)) + float_as_double(q.l);
        // the mantissa rounded: truncated it made the virial 3e-16 smaller than it is
        const unsigned long long m = ((unsigned long long)a.hi << 32) | a.lo;
        r2 = __longlong_as_double(((long long)(a.e + 1022) << 52) + (long long)((m >> 11) + (m >> 10 & 1)));
    } else {
        // close pairs: the separations to 53 bits of their own size, in the same unit
        dx = (double)dxi * (1.0 / (1 << kPairDrop));
        dy = (double)dyi * (1.0 / (1 << kPairDrop));
        dz = (double)dzi * (1.0 / (1 << kPairDrop));
        const double x = dx * pc.scale, y = dy * pc.scale, z = dz * pc.scale;
        r2 = x * x + y * y + z * z;
        const double3 t = pair_direct(r2, qq, pc.sa, pc.two_sa_pi, pc.alpha, lj ? pc.s2 : 0.0, pc.e24, pc.e4);
        f = t.x;
        s.ecd += t.y;
        if (lj) s.eld += t.z;
    }
    // force on i is -f d
    if (DIAG) {
        const double tx = f * dx, ty = f * dy, tz = f * dz;
        s.fx -= tx;
        s.fy -= ty;
        s.fz -= tz;
        s.w[0] += tx * dx;
        s.w[DIAG ? 1 : 0] += ty * dy;
        s.w[DIAG ? 2 : 0] += tz * dz;
    } else {
        s.fx -= f * dx;
        s.fy -= f * dy;
        s.fz -= f * dz;
        s.w[0] += f * r2;
    }
}

// Box edges in units, and the axes whose image is taken from FP32 separations per pair (mi).  There |d| can be
// half an edge and still within the cutoff only if the edge is hardly above 2 rc: then the image is put right in
// integers (near; the edge is below 2^64 units).
struct PairBox {
    unsigned long long L[3];
    bool near[3];
};

__device__ __forceinline__ PairBox pair_box(const double L[3], double rc, int s)
{
    PairBox b;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        b.L[t] = pair_fixed((unsigned long long)__double_as_longlong(L[t]), s);
        b.near[t] = L[t] < 2.5 * rc;
    }
    return b;
}

// d plus the image of code c: 0: -L, 1: none, 2: +L
__device__ __forceinline__ long long pair_shift(long long d, int c, unsigned long long L)
{
    return (long long)((unsigned long long)d + (c == 1 ? 0ull : (c == 0 ? 0ull - L : L)));
}

// d less the k edges that its FP32 value is nearest to
__device__ __forceinline__ long long pair_nearest(long long d, float d32, float invL, unsigned long long L, bool near)
{
    d = (long long)((unsigned long long)d - (unsigned long long)__float2ll_rn(d32 * invL) * L);
    if (near) {
        const long long half = (long long)(L >> 1);
        if (d > half) d = (long long)((unsigned long long)d - L);
        else if (d < -half) d = (long long)((unsigned long long)d + L);
    }
    return d;
}

// A packed particle: its coordinates in units (as bits) and its charge.
__device__ __forceinline__ double4_32a pair_pack(double x, double y, double z, double q, int s)
{
    double4_32a v;
    v.x = __longlong_as_double((long long)pair_fixed((unsigned long long)__double_as_longlong(x), s));
    v.y = __longlong_as_double((long long)pair_fixed((unsigned long long)__double_as_longlong(y), s));
    v.z = __longlong_as_double((long long)pair_fixed((unsigned long long)__double_as_longlong(z), s));
    v.w = q;
    return v;
}

__device__ __forceinline__ long long pair_diff(double a, double b)
{
    return (long long)((unsigned long long)__double_as_longlong(a) - (unsigned long long)__double_as_longlong(b));
}

// The warp's force sums of one particle: a transposing tree (6 FP64 additions instead of 15) that ends with x,
// y, z in lanes 0, 8, 16; they are written to F[0], F[1], F[2], times the separations' unit.
__device__ __forceinline__ void warp_force_out(double fx, double fy, double fz, double unit, int lane, double* F)
{
    const bool up = lane & 16, mid = lane & 8;
    double k0 = up ? fz : fx, k1 = up ? 0.0 : fy;
    k0 += __shfl_xor_sync(0xffffffffu, up ? fx : fz, 16);
    k1 += __shfl_xor_sync(0xffffffffu, up ? fy : 0.0, 16);
    double k = mid ? k1 : k0;
    k += __shfl_xor_sync(0xffffffffu, mid ? k0 : k1, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) k += __shfl_xor_sync(0xffffffffu, k, off);
    if ((lane & 7) == 0 && lane < 24) F[lane >> 3] = k * unit;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// A block's particles [u0, u1) over its W warps: round `base` gives one to each warp, and the last, partial
// round gives each of its particles to `parts` warps (a power of two), warp wib taking part `part`: at 132
// particles and 16 warps the last round of 4 takes a quarter of the time.  u < 0: none for this warp.
template <int W>
__device__ __forceinline__ int pair_round(int base, int u1, int wib, int& part, int& parts)
{
    const int left = u1 - base;
    parts = 1;
    while (2 * parts * left <= W) parts *= 2;
    part = wib & (parts - 1);
    const int k = wib / parts;
    return k < left ? base + k : -1;
}

// The partial forces of a particle's warps (f[warp]), summed by the first of them in order.  All threads of
// the block.
template <int W>
__device__ __forceinline__ void pair_parts_out(const double (*f)[3], int u, int i, int part, int parts, int wib, int lane,
                                               double* __restrict__ Fr)
{
    __syncthreads();
    if (u >= 0 && part == 0 && lane < 3) {
        double t = f[wib][lane];
        for (int k = 1; k < parts; ++k) t += f[wib + k][lane];
        Fr[3 * (int64_t)i + lane] = t;
    }
}

// Block partials of the sums: half of each (every pair is visited from both ends), virial components from slot
// o, then E_coul and E_lj.  All threads of the block.
template <bool DIAG, int W>
__device__ __forceinline__ void pair64_partials(const Pair64Sums<DIAG>& s, double unit, double (*red)[W],
                                                double* __restrict__ partials, int o)
{
    constexpr int nw = DIAG ? 3 : 1;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < nw + 2; ++k) {
        const double v = k < nw ? (DIAG ? s.w[k < nw ? k : 0] * unit * unit : s.w[0])
                                : (k == nw ? (double)s.ec.h + (double)s.ec.l + s.ecd
                                           : (double)s.el.h + (double)s.el.l + s.eld);
        const double t = warp_sum(v);
        if (lane == 0) red[k][wib] = t;
    }
    __syncthreads();
    if (threadIdx.x < nw + 2) {
        double t = 0.0;
        for (int v = 0; v < W; ++v) t += red[threadIdx.x][v];
        partials[o + threadIdx.x] = 0.5 * t;
    }
}

// The particle's coordinate in the box, in cells.
__device__ __forceinline__ float pair_cell_coord(float x, float invL, int nc)
{
    const float f = x * invL;
    return (f - floorf(f)) * (float)nc;
}

// Lane's segment of the slots of the 27 cells around cell c: row r = lane / 2 of the 3 x 3 rows (dy, dz), part
// lane % 2 (a row that wraps in x has two); [lo, hi) and the image shift (sx, sy, sz), 0 on an axis whose
// image is taken per pair (mi).  An axis with fewer than 3 cells visits each of them once.  Cells that lie
// farther than the search radius from the particle (fractional coordinates f of its image in the box, in cells of
// width w; with the search's margin of 2^-16 edges) are left out: about a quarter of the slots at cells of 1.1 rc.
// False: no segment.
__device__ __forceinline__ bool pair_segment_of(int c, const int nc[3], const float f[3], const float w[3], float pass,
                                                int lane, const bool mi[3],
                                                const int* __restrict__ cnt, const int* __restrict__ start, int& lo,
                                                int& hi, int& sx, int& sy, int& sz)
{
    const int cxy = nc[0] * nc[1];
    const int cz = c / cxy, cy = (c - cz * cxy) / nc[0], cx = c - cz * cxy - cy * nc[0];
    const int r = lane >> 1, part = lane & 1;
    const int dy = r % 3 - 1, dz = r / 3 - 1;
    if (!(r < 9 && dy >= (nc[1] >= 3 ? -1 : 0) && dy <= (nc[1] >= 2 ? 1 : 0) && dz >= (nc[2] >= 3 ? -1 : 0) &&
          dz <= (nc[2] >= 2 ? 1 : 0)))
        return false;
    const int uy = cy + dy, uz = cz + dz;
    const int yy = uy < 0 ? uy + nc[1] : (uy >= nc[1] ? uy - nc[1] : uy);
    const int zz = uz < 0 ? uz + nc[2] : (uz >= nc[2] ? uz - nc[2] : uz);
    // distance to the row, and what it leaves for x
    auto gap = [&](int t, int d, int cell) {
        if (nc[t] < 3 || d == 0) return 0.0f;
        float g = f[t] - (float)cell;  // in [0, 1], but for rounding over the box's edge
        g = g < -0.5f ? g + (float)nc[t] : (g > 1.5f ? g - (float)nc[t] : g);
        return fmaxf(0.0f, ((d < 0 ? g : 1.0f - g) - ((float)nc[t] * 0x1.0p-16f + 1e-4f)) * w[t]);
    };
    const float gy = gap(1, dy, cy), gz = gap(2, dz, cz), left2 = pass - gy * gy - gz * gz;
    if (left2 < 0.0f) return false;
    const float gl = gap(0, -1, cx), gr = gap(0, 1, cx);
    const int nl = gl * gl < left2 ? 1 : 0, nr = gr * gr < left2 ? 1 : 0;
    sx = 0;
    sy = mi[1] ? 0 : (uy < 0 ? -1 : (uy >= nc[1] ? 1 : 0));
    sz = mi[2] ? 0 : (uz < 0 ? -1 : (uz >= nc[2] ? 1 : 0));
    const int row = (zz * nc[1] + yy) * nc[0], nx = nc[0];
    int a = -1, e = -1;  // cells a..e of the row
    if (nx < 3) {
        if (part == 0) a = 0, e = nx - 1;
    } else if (cx == 0) {
        if (part == 0) a = 0, e = nr;
        else if (nl) a = e = nx - 1, sx = -1;
    } else if (cx == nx - 1) {
        if (part == 0) a = nx - 1 - nl, e = nx - 1;
        else if (nr) a = e = 0, sx = 1;
    } else if (part == 0) {
        a = cx - nl, e = cx + nr;
    }
    if (a < 0) return false;
    if (mi[0]) sx = 0;
    lo = start[row + a];
    hi = start[row + e] + cnt[row + e];
    return true;
}

__device__ __forceinline__ void load_pair_table(const PairWord* __restrict__ src, PairWord* dst)
{
    if (!src) return;
    const uint4* a = reinterpret_cast<const uint4*>(src);
    uint4* b = reinterpret_cast<uint4*>(dst);
    for (int i = threadIdx.x; i < (int)(kPairTabBytes / 16); i += blockDim.x) b[i] = a[i];
}

#endif

}  // namespace rbe
