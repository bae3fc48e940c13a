// Sine and cosine of a 64-bit fixed-point phase to about 2^-53, from 32-bit integer and FP32
// operations: the arithmetic of the FP64 path's pair passes.
//
// Why: GB300 issues an FP64 instruction over about 80 clocks per warp and scheduler (measured:
// 1.6 FMA per clock and SM; FP32 119, 32-bit IMAD 61, IMAD.WIDE 23, random 16-byte table loads
// from shared memory 9.8 clocks per warp and SM), and a pair of the FP64 formulation takes about
// 35 of them per pass.  Here a pair takes none.
//
// Phase.  s = r / l is a fraction of a revolution with 64 bits, kept as an integer in units of 2^-32 and
// an FP32 remainder (error at most 2^-58).  m.s is the wrapping integer sum of the m s_hi and the FP32
// sum of the m s_lo: an error of about |m| 2^-57 revolutions (FP64: |m| 2^-54 from s alone).
// The top 11 bits, rounded, pick an entry a of a table of 2048 angles; the rest is x, |x| <= 2 pi 2^-12
// (and a little more: the FP32 sum is at most |m| units), a float-float.
//   sin(a + x) = S + sin x (C - S t),  cos(a + x) = C - sin x (S + C t),  t = tan(x / 2)
// (S, C the table's sine and cosine).  The bracket and the product are float-float: their result
// is at most 2^-9.3, so 2^-46 of it is enough.  Its integer part is taken by an FP32 addition of a
// constant (the mantissa bits of c + v hold round(v)) and added to the table's.  Result: an integer in
// units of 2^-30 and an FP32 remainder.  Errors: the remainder's rounding (2^-54), the table (2^-55),
// the float-float product (about 2^-55).
//
// The bracket's float-float sum is Fast2Sum-exact because |C t| < |S| for every table entry with
// S != 0 (the smallest is sin(2 pi / 2048) = 3.1e-3, |t| <= 7.7e-4).
//
// A 64-bit multiply-add of 32-bit factors is a multiplication and two additions here (23 per clock and SM
// against 61 fused 32-bit ones), so only the products that need 64 bits take it.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "rbe_device.cuh"

namespace rbe {

constexpr int kTrigN = 2048;                   // table angles per revolution

// sin and cos of 2 pi i / kTrigN as a + r 2^-24 in units of 2^-30, a the nearest integer and r an integer
// (TrigEntry); a is the float (float)a plus at most 32, and (that rest) + r 2^-24 as a float is the low part of
// the value as a float-float (kept in a second plane).  Half a revolution on, every part is the exact
// negative.  Random loads cost bank conflicts (17.7 clocks of the SM for 16 bytes per lane, 9.6 for 8):
// with the floats stored whole beside the integers the shared-memory pipe was 80 % busy and bound the
// passes; with everything rebuilt from the integers the conversions did.
struct alignas(16) TrigEntry {
    int sa, sr, ca, cr;
};
struct alignas(8) TrigLow {
    float s, c;
};
// For a sine alone: the sine's integers and the cosine's float-float; the sine's low part in its own plane.
struct alignas(16) TrigSine {
    int sa, sr;
    float ch, cl;
};
// The table (88 KB, a constant of the library's device image: formed by the compiler).
struct TrigTable {
    TrigEntry entry[kTrigN];
    TrigLow low[kTrigN];
    TrigSine sine[kTrigN];
    float sine_low[kTrigN];
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

// kHiMagic + v holds round(v) in its mantissa (|v| < 2^22).
constexpr float kHiMagic = 12582912.0f;  // 1.5 2^23, bits 0x4B400000
// 2^31 on a 64-bit value makes its low word, read with the top bit flipped, the signed remainder of its
// high word: the form in which 64-bit values enter a product.
constexpr unsigned long long kMulBias = 1ull << 31;

// sin(pi k / 1024) for k in [0, 512], in units of 2^-63: Taylor series in 64-bit fixed point (errors of a
// few units) on [0, pi/4] and by symmetry beyond.
constexpr unsigned long long quarter_sine(int k)
{
    const bool use_cos = k > kTrigN / 8;
    const unsigned kk = (unsigned)(use_cos ? kTrigN / 4 - k : k);         // argument pi kk / 1024 in [0, pi/4]
    const unsigned __int128 pi61 = 0x6487ED5110B4611Aull;                 // floor(pi 2^61)
    const unsigned long long x = (unsigned long long)((pi61 * kk) >> 8);  // the argument in units of 2^-63
    const unsigned long long x2 = (unsigned long long)(((unsigned __int128)x * x) >> 63);
    unsigned long long term = use_cos ? 1ull << 63 : x, sum = term;
    bool minus = true;
    for (int n = use_cos ? 1 : 2; n < 26; n += 2, minus = !minus) {
        term = (unsigned long long)(((unsigned __int128)term * x2) >> 63) / (unsigned)(n * (n + 1));
        sum = minus ? sum - term : sum + term;
    }
    return sum;
}

// A sine (u 2^-63, negated if neg) as a table entry's two parts.
constexpr void trig_split(unsigned long long u, bool neg, int& a, int& r)
{
    a = (int)((u + (1ull << 32)) >> 33);
    const long long rest = (long long)(u - ((unsigned long long)a << 33));  // units of 2^-63, up to 2^32
    r = (int)((rest + 256) >> 9);
    if (neg) {
        a = -a;
        r = -r;
    }
}

constexpr TrigEntry trig_entry(int i)
{
    const int q = kTrigN / 4, half = i % (2 * q);
    TrigEntry e{};
    trig_split(quarter_sine(half <= q ? half : 2 * q - half), i >= 2 * q, e.sa, e.sr);
    trig_split(quarter_sine(half <= q ? q - half : half - q), (i >= 2 * q) != (half > q), e.ca, e.cr);
    return e;
}

constexpr TrigLow trig_low(const TrigEntry& e)
{
    TrigLow l{};
    l.s = (float)((double)(e.sa - (int)(float)e.sa) + (double)e.sr * 0x1.0p-24);
    l.c = (float)((double)(e.ca - (int)(float)e.ca) + (double)e.cr * 0x1.0p-24);
    return l;
}

constexpr TrigTable make_trig_table()
{
    TrigTable t{};
    for (int i = 0; i < kTrigN; ++i) {
        const TrigEntry e = trig_entry(i);
        t.entry[i] = e;
        t.low[i] = trig_low(e);
        t.sine[i].sa = e.sa;
        t.sine[i].sr = e.sr;
        t.sine[i].ch = (float)e.ca;
        t.sine[i].cl = t.low[i].c;
        t.sine_low[i] = t.low[i].s;
    }
    return t;
}

// Start value of the integer phase sum: half a table spacing, so that the index is the rounded phase.
constexpr uint32_t kPhaseStart = 1u << 20;

// A 64-bit fraction as its nearest multiple of 2^-32 and the rest in those units.
struct Frac {
    int hi;
    float lo;
};

// The FP32 sum of the low words, m.s_lo, is up to 3/2 of the largest |m| in units of 2^-32.  phase_x and
// trig_value take it up to about 2^17 (the series of the remainder, the integer part below 2^22), with the lengths
// |m| up to kPhaseNarrow as it is.  Beyond, phase_whole moves its whole part into the integer sum first: errors
// then grow as |m| 2^-56 revolutions (FP64 phases: |m| 2^-54) for any 32-bit m.
constexpr uint32_t kPhaseNarrow = 1u << 16;

__host__ __device__ __forceinline__ bool phase_is_wide(int mx, int my, int mz)
{
    constexpr uint32_t n = kPhaseNarrow;
    return (uint32_t)mx + n > 2u * n || (uint32_t)my + n > 2u * n || (uint32_t)mz + n > 2u * n;
}

__host__ __device__ __forceinline__ void phase_whole(uint32_t& hi, float& lo)
{
    const float k = rintf(lo);
    hi += (uint32_t)(unsigned long long)(long long)k;
    lo = RBE_ADD(lo, -k);
}

// The remainder of a phase: sin x = sh + sl, tan(x / 2) = th + tl.
struct PhaseX {
    float sh, sl, th, tl;
};

// hi: integer phase sum (with kPhaseStart), lo: the FP32 sum, in units of 2^-32 revolutions.
__host__ __device__ __forceinline__ PhaseX phase_x(uint32_t hi, float lo)
{
    // 2 pi 2^-32 = k1 + k2
    const float k1 = 1.46291807926715968e-9f;
    const float k2 = (float)(1.46291807926715968105e-9 - (double)1.46291807926715968e-9f);
    const float d = RBE_ADD(fx_float((hi & 0x1FFFFFu) | 0x4B000000u), -(8388608.0f + 1048576.0f));
    // d + lo = dh + dl: exact, since d is an integer (also where |d| < |lo|)
    const float dh = RBE_ADD(d, lo), dl = RBE_ADD(lo, -RBE_ADD(dh, -d));
    PhaseX r;
    r.sh = RBE_MUL(dh, k1);
    float xl = RBE_FMA(dh, k1, -r.sh);
    xl = RBE_FMA(dh, k2, xl);
    xl = RBE_FMA(dl, k1, xl);
    // sin x = x - x^3 / 6 + x^5 / 120, tan(x/2) = x/2 + x^3 / 24 (the next term is below 2^-54)
    const float x2 = RBE_MUL(r.sh, r.sh), x3 = RBE_MUL(x2, r.sh);
    r.sl = RBE_FMA(RBE_FMA(x2, 1.0f / 120.0f, -1.0f / 6.0f), x3, xl);
    r.th = RBE_MUL(0.5f, r.sh);
    r.tl = RBE_FMA(x3, 1.0f / 24.0f, RBE_MUL(0.5f, xl));
    return r;
}

__host__ __device__ __forceinline__ float fx_i2f(int i)
{
#ifdef __CUDA_ARCH__
    return __int2float_rn(i);
#else
    return (float)i;
#endif
}

// V + sg sin x (D - sg V t) for a value V = (a + ...) with the float-float (vh, vl) and its derivative (dh,
// dl): sg = +1 gives sin(a + x) from (sine, cosine), sg = -1 cos(a + x) from (cosine, sine).  Result hi + lo
// plus the table's r 2^-24, in units of 2^-30: an integer and a float, |lo| < 1.3.
template <int SG>
__host__ __device__ __forceinline__ void trig_value(int a, float vh, float vl, float dh, float dl, const PhaseX& x,
                                                    int& hi, float& lo)
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
    const float t = RBE_ADD(p, kHiMagic);
    lo = RBE_ADD(RBE_ADD(p, -RBE_ADD(t, -kHiMagic)), e);
    hi = (int)((uint32_t)a + fx_bits(t) - 0x4B400000u);
}

// lo + r 2^-24 as a float and as an integer in units of 2^-24 (both below 1.8 in magnitude).
__host__ __device__ __forceinline__ float trig_low_f(int r, float lo) { return RBE_FMA(fx_i2f(r), 0x1.0p-24f, lo); }
__host__ __device__ __forceinline__ int trig_low_i(int r, float lo)
{
#ifdef __CUDA_ARCH__
    return r + __float2int_rn(RBE_MUL(lo, 16777216.0f));
#else
    return r + (int)rintf(lo * 16777216.0f);
#endif
}

// The signed halves of a value held with kMulBias: v = fx_hi 2^32 + fx_lo.
__host__ __device__ __forceinline__ int fx_hi(unsigned long long v) { return (int)(uint32_t)(v >> 32); }
__host__ __device__ __forceinline__ int fx_lo(unsigned long long v) { return (int)((uint32_t)v ^ 0x80000000u); }

// v b 2^-60 for v = v_hi + v_lo 2^-24 (units of 2^-30; |v_lo| < 2^25) and b = b_hi 2^30 + b_lo
// (0 <= b < 2^60, b_lo signed), rounded, plus kMulBias: three 64-bit products; that of the low words (below
// two units) is left out.
__host__ __device__ __forceinline__ unsigned long long mul_fix(int v_hi, int v_lo, int b_hi, int b_lo)
{
    // the constant: 2^31 as the bias (c is below 2^31 in magnitude) and one half, both shifted by 30
    unsigned long long c = mad_wide((int)((uint32_t)v_lo << 6), b_hi, (1ull << 61) + (1ull << 29));
    c = mad_wide(v_hi, b_lo, c);
    return mad_wide(v_hi, b_hi, (unsigned long long)(uint32_t)(c >> 30));
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

__host__ __device__ __forceinline__ Frac frac_of(unsigned long long f)
{
    const unsigned long long g = f + kMulBias;
    return Frac{fx_hi(g), fx_i2f(fx_lo(g)) * 0x1.0p-32f};
}

// |q| as a fraction of 2^(E + 1), E = the unbiased exponent of a number no smaller than |q| (eb: its
// exponent field, 1 .. 2046), in units of 2^-55, rounded: exact for charges within a factor of 4 of it.
__host__ __device__ inline unsigned long long fix_magnitude(unsigned long long qb, int eb)
{
    const int e = (int)((qb >> 52) & 0x7ff);
    if (e == 0 || e > eb) return 0ull;  // zero or subnormal (below 2^-1022)
    const unsigned long long m = (qb & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = 2 - (eb - e);  // m 2^(e - eb) 2^(54 - 52)
    return sh >= 0 ? m << sh : (sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0ull);
}

}  // namespace rbe
