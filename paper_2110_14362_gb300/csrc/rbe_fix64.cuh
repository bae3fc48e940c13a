// Sine and cosine of a 64-bit fixed-point phase to about 2^-53, from 32-bit integer and FP32
// operations: the arithmetic of the FP64 path's pair passes.
//
// Why: GB300 issues an FP64 instruction over about 80 clocks per warp and scheduler (measured:
// 1.6 FMA per clock and SM; FP32 119, 32-bit IMAD 61, IMAD.WIDE 23, random 16-byte table loads
// from shared memory 9.8 clocks per warp and SM), and a pair of the FP64 formulation takes about
// 35 of them per pass.  Here a pair takes none.
//
// Phase.  s = r / l is a 64-bit fraction of a revolution (error about 2^-64, against 2^-53 of a
// double), so m.s mod 1 is exact in wrapping integer arithmetic.  The top 11 bits, rounded, pick
// an entry a of a table of 2048 angles; the rest is x, |x| <= 2 pi 2^-12, a float-float.
//   sin(a + x) = S + sin x (C - S t),  cos(a + x) = C - sin x (S + C t),  t = tan(x / 2)
// (S, C the table's sine and cosine).  The bracket and the product are float-float: their result
// is at most 2^-9.3, so 2^-46 of it is enough.  It is turned into fixed point by two FP32
// additions of a constant (the mantissa bits of c + v hold round(v)) and added to the table's
// 64-bit value.  Result: a 64-bit integer in units of 2^-62.  Errors: the fixed-point rounding of
// the low part (at most 2^-53), the table (2^-61), the float-float product (about 2^-55).
//
// The bracket's float-float sum is Fast2Sum-exact because |C t| < |S| for every table entry with
// S != 0 (the smallest is sin(2 pi / 2048) = 3.1e-3, |t| <= 7.7e-4).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "rbe_device.cuh"

namespace rbe {

constexpr int kTrigN = 2048;                   // table angles per revolution
constexpr int kTrigLen = kTrigN + kTrigN / 4;  // entries: cos(a) = sin(a + 1/4 revolution)

// v: sin(2 pi i / kTrigN) in units of 2^-62, made odd (so that no product of it with a power of
// two is a rounding tie, and sin(a + pi) is the exact negative), plus kMulBias - kTrigBias; h + l: the
// same sine times 2^30 as a float-float.
struct alignas(16) TrigEntry {
    unsigned long long v;
    float h, l;
};

#ifdef __CUDA_ARCH__
#define RBE_FMA(a, b, c) __fmaf_rn(a, b, c)
#define RBE_MUL(a, b) __fmul_rn(a, b)
#define RBE_ADD(a, b) __fadd_rn(a, b)
#else
#define RBE_FMA(a, b, c) fmaf(a, b, c)
#define RBE_MUL(a, b) ((a) * (b))
#define RBE_ADD(a, b) ((a) + (b))
#endif

__host__ __device__ __forceinline__ uint32_t fx_bits(float f)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    uint32_t u;
    __builtin_memcpy(&u, &f, 4);
    return u;
#endif
}

__host__ __device__ __forceinline__ float fx_float(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    __builtin_memcpy(&f, &u, 4);
    return f;
#endif
}

// a * b + c with a 64-bit c, signed 32-bit factors (one IMAD.WIDE)
__host__ __device__ __forceinline__ unsigned long long mad_wide(int a, int b, unsigned long long c)
{
    return c + (unsigned long long)((long long)a * (long long)b);
}

// kHiMagic + v holds round(v) in its mantissa (|v| < 2^22); kLoMagic + v holds v (|v| < 1; here at most
// 0.7: half a unit and the products' rounding errors) on a grid of 2^-22.  kTrigBias removes the
// constants' own bits from the sum.
constexpr float kHiMagic = 12582912.0f;  // 1.5 2^23, bits 0x4B400000
constexpr float kLoMagic = 3.0f;         // bits 0x40000000 + (v + 1) 2^22
constexpr unsigned long long kTrigBias = (0x4B400000ull << 32) + (1ull << 40) + (1ull << 32);
// 2^31 on a 64-bit value makes its low word, read with the top bit flipped, the signed remainder of its
// high word: the form in which 64-bit values enter a product.
constexpr unsigned long long kMulBias = 1ull << 31;

// Entry i: the sine by its Taylor series in 64-bit fixed point (units of 2^-63, errors of a few of
// them) on [0, pi/4] and by symmetry elsewhere.
__host__ __device__ inline TrigEntry trig_entry(int i)
{
    const int j = i % kTrigN, half = j % (kTrigN / 2), quarter = kTrigN / 4;
    const int k = half <= quarter ? half : kTrigN / 2 - half;     // angle pi k / 1024 in [0, pi/2]
    const bool use_cos = k > quarter / 2;
    const unsigned kk = (unsigned)(use_cos ? quarter - k : k);    // argument pi kk / 1024 in [0, pi/4]
    const unsigned __int128 pi61 = 0x6487ED5110B4611Aull;         // floor(pi 2^61)
    const unsigned long long x = (unsigned long long)((pi61 * kk) >> 8);  // the argument in units of 2^-63
    const unsigned long long x2 = (unsigned long long)(((unsigned __int128)x * x) >> 63);
    unsigned long long term = use_cos ? 1ull << 63 : x, sum = term;
    bool minus = true;
    for (int n = use_cos ? 1 : 2; n < 26; n += 2, minus = !minus) {
        term = (unsigned long long)(((unsigned __int128)term * x2) >> 63) / (unsigned)(n * (n + 1));
        sum = minus ? sum - term : sum + term;
    }
    long long v = (long long)((sum >> 1) + (sum & 1));  // units of 2^-62
    if ((v & 1) == 0) v += v == 0 ? 1 : -1;
    const double s = (double)sum * 0x1.0p-33;  // the sine times 2^30
    TrigEntry e;
    e.h = (float)s;
    e.l = (float)(s - (double)e.h);
    if (j >= kTrigN / 2) {
        v = -v;
        e.h = -e.h;
        e.l = -e.l;
    }
    e.v = (unsigned long long)v - kTrigBias + kMulBias;
    return e;
}

// Start value of a phase sum: half a table spacing in the high word (the index is the rounded
// phase) and half of 2^32 in the low word (which is then read as a signed remainder).
constexpr unsigned long long kPhaseStart = (1ull << 52) + (1ull << 31);

// The remainder of a phase: sin x = sh + sl (|sl| at most half a unit of sh), tan(x / 2) = th + tl.
struct PhaseX {
    float sh, sl, th, tl;
};

// hi: high word of the phase sum (with kPhaseStart), lo: low word.
__host__ __device__ __forceinline__ PhaseX phase_x(uint32_t hi, uint32_t lo)
{
    // 2 pi 2^-32 = k1 + k2, and k1 2^-32 for the low word
    const float k1 = 1.46291807926715968e-9f;              // RN(2 pi 2^-32)
    const float k2 = (float)(1.46291807926715968105e-9 - (double)1.46291807926715968e-9f);
    const float k3 = k1 * 2.3283064365386963e-10f;
    const float dh = RBE_ADD(fx_float((hi & 0x1FFFFFu) | 0x4B000000u), -(8388608.0f + 1048576.0f));
#ifdef __CUDA_ARCH__
    const float dl = __int2float_rn((int)(lo ^ 0x80000000u));
#else
    const float dl = (float)(int)(lo ^ 0x80000000u);
#endif
    const float xh = RBE_MUL(dh, k1);
    float xl = RBE_FMA(dh, k1, -xh);
    xl = RBE_FMA(dh, k2, xl);
    xl = RBE_FMA(dl, k3, xl);  // up to 7.3e-10: not below xh's last bit
    // sin x = x - x^3 / 6 + x^5 / 120, tan(x/2) = x/2 + x^3 / 24 (the next term is below 2^-54)
    const float y = RBE_ADD(xh, xl), x2 = RBE_MUL(y, y), x3 = RBE_MUL(x2, y);
    const float sl = RBE_FMA(RBE_FMA(x2, 1.0f / 120.0f, -1.0f / 6.0f), x3, xl);
    PhaseX r;
    r.sh = RBE_ADD(xh, sl);  // Fast2Sum: |xh| >= |sl| or xh = 0
    r.sl = RBE_ADD(sl, -RBE_ADD(r.sh, -xh));
    r.th = RBE_MUL(0.5f, xh);
    r.tl = RBE_FMA(x3, 1.0f / 24.0f, RBE_MUL(0.5f, xl));
    return r;
}

// V + sg sin x (D - sg V' t): with (vh, vl) the float-float of the value whose entry v is given, and
// (dh, dl) that of its derivative: sg = +1 gives sin(a + x) from (S; C), sg = -1 cos(a + x) from
// (C; S).  Result in units of 2^-62, plus kMulBias.
template <int SG>
__host__ __device__ __forceinline__ unsigned long long trig_value(unsigned long long v, float vh, float vl, float dh,
                                                                  float dl, const PhaseX& x)
{
    const float nh = SG > 0 ? -vh : vh, nl = SG > 0 ? -vl : vl;
    const float ah = RBE_FMA(nh, x.th, dh);
    float al = RBE_FMA(nh, x.th, RBE_ADD(dh, -ah));
    al = RBE_FMA(nh, x.tl, al);
    al = RBE_FMA(nl, x.th, al);
    al = RBE_ADD(al, dl);
    const float sx = SG > 0 ? x.sh : -x.sh, sxl = SG > 0 ? x.sl : -x.sl;
    const float p = RBE_MUL(ah, sx);
    float e = RBE_FMA(ah, sx, -p);
    e = RBE_FMA(ah, sxl, e);
    e = RBE_FMA(al, sx, e);
    const float t1 = RBE_ADD(p, kHiMagic);
    const float r = RBE_ADD(p, -RBE_ADD(t1, -kHiMagic));
    const float t3 = RBE_ADD(RBE_ADD(r, e), kLoMagic);
    const unsigned long long w = v + (unsigned long long)fx_bits(t3) * 1024ull;
    return w + ((unsigned long long)fx_bits(t1) << 32);
}

// The signed halves of a value held with kMulBias: v = fx_hi 2^32 + fx_lo.
__host__ __device__ __forceinline__ int fx_hi(unsigned long long v) { return (int)(uint32_t)(v >> 32); }
__host__ __device__ __forceinline__ int fx_lo(unsigned long long v) { return (int)((uint32_t)v ^ 0x80000000u); }

// a b 2^-64 for a (signed) and b (0 <= b < 2^62) given as signed halves, rounded, plus kMulBias: three
// IMAD.WIDE.  The product of the low words (at most a quarter unit, of either sign) is left out.
__host__ __device__ __forceinline__ unsigned long long mul_fix(int a_hi, int a_lo, int b_hi, int b_lo)
{
    unsigned long long c = mad_wide(a_lo, b_hi, (1ull << 63) + (1ull << 31));
    c = mad_wide(a_hi, b_lo, c);
    return mad_wide(a_hi, b_hi, c >> 32);
}

// 1 / l as a 64-bit mantissa (rounded to the last bit) and a power of two, l a positive normal double
// with inv = the double nearest 1 / l: the double's 53 bits corrected by the remainder.
__host__ __device__ inline FixScale fix_scale64(double l, double inv)
{
    unsigned long long lb, ib;
#ifdef __CUDA_ARCH__
    lb = (unsigned long long)__double_as_longlong(l);
    ib = (unsigned long long)__double_as_longlong(inv);
#else
    __builtin_memcpy(&lb, &l, 8);
    __builtin_memcpy(&ib, &inv, 8);
#endif
    const unsigned long long ml = (lb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const unsigned long long mi = ((ib & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 11;  // inv = mi 2^e
    const int el = (int)((lb >> 52) & 0x7ff) - 1075, e = (int)((ib >> 52) & 0x7ff) - 1075 - 11;
    // 1 = ml mi 2^(el + e) (1 + small): the remainder 2^-(el + e) - ml mi, modulo 2^64, is a small signed
    // number (|.| <= 2^52 2^11), and the correction of mi is remainder / ml
    const int n = -(el + e);  // 115 or 116: 2^n is 0 modulo 2^64
    const long long rem = (n < 64 ? (long long)(1ull << n) : 0ll) - (long long)(ml * mi);
    const float corr = (float)rem / (float)ml;  // at most 2^10 in magnitude: FP32 places it to 2^-13
    const int k = (int)(corr < 0.0f ? corr - 0.5f : corr + 0.5f);
    const unsigned long long q = mi + (unsigned long long)(long long)k;
    if (k > 0 && q < mi) return FixScale{0xFFFFFFFFFFFFFFFFull, e};  // 1 / l rounded up to a power of two
    return FixScale{q, e};
}

// round(r / l * 2^64) mod 2^64 for a finite double r (zero and subnormal r give 0): the 117-bit product
// of r's mantissa and the 64-bit 1 / l, shifted and rounded to nearest.
__host__ __device__ inline unsigned long long fixed_frac64(unsigned long long rb, FixScale sc)
{
    const unsigned er = (unsigned)(rb >> 52) & 0x7ffu;
    if (er == 0u || er == 0x7ffu) return 0ull;
    const unsigned long long mr = (rb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = (int)er - 1075 + sc.e + 64;  // r / l * 2^64 = mr q 2^sh
#ifdef __CUDA_ARCH__
    const unsigned long long hi = __umul64hi(mr, sc.q);
#else
    const unsigned long long hi = (unsigned long long)(((unsigned __int128)mr * sc.q) >> 64);
#endif
    const unsigned long long lo = mr * sc.q;
    unsigned long long res;
    if (sh >= 0) {
        res = sh >= 64 ? 0ull : lo << sh;
    } else {
        const int d = -sh;
        unsigned long long lo2 = lo, hi2 = hi;
        if (d <= 64) {
            lo2 = lo + (1ull << (d - 1));
            hi2 = hi + (lo2 < lo ? 1ull : 0ull);
        } else if (d < 128) {
            hi2 = hi + (1ull << (d - 65));
        }
        if (d < 64) res = (lo2 >> d) | (hi2 << (64 - d));
        else if (d < 128) res = hi2 >> (d - 64);
        else res = 0ull;
    }
    return (rb >> 63) ? 0ull - res : res;
}

// |q| as a 59-bit fraction of 2^(E + 1), E = the unbiased exponent field of a number no smaller than
// |q|: floor(|q| 2^(58 - E)).  eb: that exponent field (1 .. 2046).
__host__ __device__ inline unsigned long long fix_magnitude(unsigned long long qb, int eb)
{
    const int e = (int)((qb >> 52) & 0x7ff);
    if (e == 0 || e > eb) return 0ull;  // zero or subnormal (below 2^-1022)
    const unsigned long long m = (qb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = 6 - (eb - e);  // m 2^(e - eb) 2^(58 - 52)
    return sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ull);
}

}  // namespace rbe
