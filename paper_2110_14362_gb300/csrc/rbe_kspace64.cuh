// Pair passes of the FP64 path: rho, its reduction and the forces, on the 64-bit fixed-point sine and
// cosine of rbe_fix64.cuh.  No FP64 instruction runs per pair; sums over particles and frequencies are
// integers (exact, in any order), converted to double once per chunk or particle.
//
// What bounds them: a pair is about 90 instructions on the FMA and ALU pipes in either pass, 5 or 6 of them
// 64-bit products, and 25 bytes of random table loads from shared memory; at P = 500 a pair takes 106
// clocks of a scheduler in the rho pass and 124 in the force pass (0.86 and 0.70 instructions per clock;
// the force pass waits for the heavy FMA pipe, which the integer products run on); DRAM moves 32 to 56 B
// per particle.  Against FP64 sincospi per pair (about 35 FP64 instructions per pass, 76 clocks of a
// scheduler each): N = 3e5, P = 200 8330 -> 385 us per evaluation, 1e6 x 500 67.8 -> 2.87 ms, 1e3 x 100
// 386 -> 20.5 us.
#pragma once

#include <type_traits>

#include "rbe_fix64.cuh"
#include "rbe_kspace_tiles.cuh"

namespace rbe {

// Resident blocks the registers are sized for, and the unrolling of the pair loops (slab, N = 3e5, P = 200:
// rho 199 us unrolled by 2, 216 by 1, 205 by 4, 217 at one block of 128 registers; force 186 us by 4, 209
// by 1, 197 by 2, 219 at three blocks of 80 registers, 242 at five of 48).
#ifndef RBE_RHO64_MINB
#define RBE_RHO64_MINB 2
#endif
#ifndef RBE_FORCE64_MINB
#define RBE_FORCE64_MINB 4
#endif
#ifndef RBE_RHO64_UNROLL
#define RBE_RHO64_UNROLL 2
#endif
#ifndef RBE_FORCE64_UNROLL
#define RBE_FORCE64_UNROLL 4
#endif
constexpr int kRho64Unroll = RBE_RHO64_UNROLL, kForce64Unroll = RBE_FORCE64_UNROLL;
constexpr int kRho64Threads = 512;   // threads of a rho block at most
constexpr int kRho64Stage = 512;     // particles staged per tile at most (32 B each)
constexpr int kRho64Group = 32;      // pairs whose products (at most 2^57 each) are summed in 64 bits
constexpr int kForce64Threads = 256;
constexpr int kForce64Stage = 256;   // frequencies staged per tile (48 B each)
constexpr size_t kRho64Trig = (sizeof(TrigEntry) + sizeof(TrigLow)) * kTrigN;  // planes entry and low
constexpr size_t kForce64Trig = (sizeof(TrigSine) + sizeof(float)) * kTrigN;    // planes sine and sine_low
constexpr size_t kRho64Smem = kRho64Trig + 32 * (size_t)kRho64Stage;
constexpr size_t kForce64Smem = kForce64Trig + 48 * (size_t)kForce64Stage;

__device__ const TrigTable g_trig = make_trig_table();

__device__ __forceinline__ void load_trig(const void* __restrict__ src_v, void* dst_v, int bytes)
{
    const uint4* src = reinterpret_cast<const uint4*>(src_v);
    uint4* dst = reinterpret_cast<uint4*>(dst_v);
    for (int i = threadIdx.x; i < bytes / 16; i += blockDim.x) dst[i] = src[i];
}

// A 128-bit integer as the nearest double or next to it (two roundings), times 2^e.
__device__ __forceinline__ double int128_to_double(__int128 s, int e)
{
    const bool neg = s < 0;
    const unsigned __int128 a = neg ? (unsigned __int128)0 - (unsigned __int128)s : (unsigned __int128)s;
    const double d = ldexp((double)(unsigned long long)(a >> 64), 64) + (double)(unsigned long long)a;
    return ldexp(neg ? -d : d, e);
}

// Fixed-order block sums of two doubles per thread; valid in thread 0.
__device__ __forceinline__ void block_sum2(double& a, double& b, double (*scratch)[32])
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (nw == 1) return;
    if (lane == 0) {
        scratch[0][warp] = a;
        scratch[1][warp] = b;
    }
    __syncthreads();
    if (warp == 0) {
        a = lane < nw ? scratch[0][lane] : 0.0;
        b = lane < nw ? scratch[1][lane] : 0.0;
        for (int off = 16; off > 0; off >>= 1) {
            if (off >= nw) continue;  // the same for every lane; the lanes beyond hold zeros
            a += __shfl_xor_sync(0xffffffffu, a, off);
            b += __shfl_xor_sync(0xffffffffu, b, off);
        }
    }
}

// A coordinate that is not finite, or whose r / l is not.  Not inlined: the pair loop keeps its registers (inlined,
// the rho pass took 5 % longer).
static __device__ __noinline__ bool coord_bad(const KState* ks, unsigned long long bx, unsigned long long by,
                                              unsigned long long bz)
{
    const double s = __longlong_as_double((long long)bx) * ks->inv[0], t = __longlong_as_double((long long)by) * ks->inv[1],
                 u = __longlong_as_double((long long)bz) * ks->inv[2];
    return !isfinite(s) || !isfinite(t) || !isfinite(u);
}

// =================================================================================
// rho pass.  Block (kt, c): T frequency lanes (thread j of sub-stream s owns frequency kt T + j) in S
// particle sub-streams over the particles of chunk c, staged kRho64Stage at a time as 64-bit
// fixed-point positions and charges and read as broadcasts.
//
// Charges: |q| is taken as a 55-bit fraction qh 2^-27 + ql 2^-55 of twice the power of two of the chunk's
// largest |q| (exact for charges within a factor of 4 of it, an error of 2^-56 of that power below); the
// sign is half a revolution of the phase.  With the sine (or cosine) as v + w, v an integer in units of
// 2^-30, a product takes two integer multiplications, v qh and v ql, summed in 64 bits over 32 pairs,
// and one FP32 FMA for w qh (2^-57 of the charge at most, so the FP32 sum of 32 of them is good to
// 2^-78); the groups' sums are added in 128 bits.  Where every charge of the staged tile has ql = 0 (27
// significant bits do: integers, equal magnitudes that are a power of two) v ql is left out.
// Partials: (Re, Im) at [l * nchunks + c]; row K holds the chunk's sum of q^2 in FP64.
// CHECK: a list whose |m| the host does not bound (rbe_ctx_s::m_narrow): the warps with a frequency beyond kPhaseNarrow
// move the low phase's whole part into the integer sum.  Kernels of their own, because the second loop beside the
// ordinary one took its registers: N = 3e5, P = 200 391 us per evaluation against 387, 1e6 x 500 2.93 against 2.87 ms
// (a weighted call of the former size: 388.2 us with CHECK, 387.1 without).
template <bool CHECK>
__global__ void __launch_bounds__(kRho64Threads, RBE_RHO64_MINB)
k_rho_f64(const double* __restrict__ pos, const double* __restrict__ q, int64_t N, const KState* __restrict__ ks,
          const int4* __restrict__ m, int K, int64_t chunk_len, int nchunks, double2* __restrict__ partials,
          unsigned* __restrict__ status, int S, int T)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    TrigEntry* st = reinterpret_cast<TrigEntry*>(s_raw);
    int4* sp = reinterpret_cast<int4*>(s_raw + kRho64Trig);
    __shared__ int s_eb, s_bad;
    __shared__ double s_red[2][32];
    const int tid = threadIdx.x, nt = blockDim.x, kt = blockIdx.x, c = blockIdx.y;
    const int64_t start = (int64_t)c * chunk_len, end = min(N, start + chunk_len);
    if (tid == 0) {
        s_eb = 1;
        s_bad = 0;
    }
    __syncthreads();
    load_trig(g_trig.entry, st, (int)kRho64Trig);
    // the largest exponent field of the chunk's charges, and the sum of their squares (inputs only)
    int eb = 1;
    double q2 = 0.0, zero = 0.0;
    for (int64_t i = start + tid; i < end; i += nt) {
        const double qi = q[i];
        const int e = (int)(((unsigned long long)__double_as_longlong(qi) >> 52) & 0x7ffull);
        eb = max(eb, e);
        if (kt == 0) q2 += qi * qi;
    }
    eb = __reduce_max_sync(0xffffffffu, eb);
    if ((tid & 31) == 0) atomicMax(&s_eb, eb);
    if (kt == 0) block_sum2(q2, zero, s_red);
    __syncthreads();
    eb = min(s_eb, 0x7fe);
    const bool bad_q = s_eb == 0x7ff;
    pdl_wait();
    pdl_trigger();
    if (bad_q && tid == 0) {
        atomicOr(status, kStatusNonFinite);
        s_bad = 1;
    }
    const int j = tid % T, ss = tid / T, l = kt * T + j;
    const bool act = ss < S && l < K;
    const int share = kRho64Stage / S, stage = share * S;
    const int4 mv = act ? m[l] : make_int4(0, 0, 0, 0);
    const float mfx = (float)mv.x, mfy = (float)mv.y, mfz = (float)mv.z;
    const FixScale scx = fs(ks->sc64[0]), scy = fs(ks->sc64[1]), scz = fs(ks->sc64[2]);
    // r / l is below 2^(exponent field - 958 + sc.e): finite up to this field
    const int far = min(1982 - max(max(scx.e, scy.e), scz.e), 0x7fe);
    const bool wide = CHECK && __any_sync(0xffffffffu, phase_is_wide(mv.x, mv.y, mv.z));
    const TrigLow* sw = reinterpret_cast<const TrigLow*>(st + kTrigN);
    __int128 re = 0, im = 0;
    for (int64_t base = start; base < end; base += stage) {
        __syncthreads();  // every thread is done with the previous tile
        const int here = (int)min((int64_t)stage, end - base);
        int low = 0;
        for (int u = tid; u < here; u += nt) {
            const int64_t i = base + u;
            const unsigned long long bx = (unsigned long long)__double_as_longlong(pos[3 * i]);
            const unsigned long long by = (unsigned long long)__double_as_longlong(pos[3 * i + 1]);
            const unsigned long long bz = (unsigned long long)__double_as_longlong(pos[3 * i + 2]);
            const unsigned long long bq = (unsigned long long)__double_as_longlong(q[i]);
            const int ex = (int)(bx >> 52) & 0x7ff, ey = (int)(by >> 52) & 0x7ff, ez = (int)(bz >> 52) & 0x7ff;
            if (max(max(ex, ey), ez) > far && coord_bad(ks, bx, by, bz)) {
                atomicOr(status, kStatusNonFinite);
                s_bad = 1;
            }
            const Frac x = frac_of(fixed_frac64(bx, scx)), y = frac_of(fixed_frac64(by, scy)),
                       z = frac_of(fixed_frac64(bz, scz));
            const unsigned long long a = fix_magnitude(bq, eb) + (1ull << 27);
            const int ql = (int)(a & 0xFFFFFFFull) - (1 << 27);
            low |= ql;
            sp[2 * u] = make_int4(x.hi, y.hi, z.hi, (int)((uint32_t)(a >> 28) | ((uint32_t)(bq >> 63) << 31)));
            sp[2 * u + 1] = make_int4(__float_as_int(x.lo), __float_as_int(y.lo), __float_as_int(z.lo), ql);
        }
        const bool has_low = __syncthreads_or(low) != 0;
        if (!act) continue;
        const int p1 = min(here, (ss + 1) * share);
        auto group = [&](auto low_tag, auto wide_tag, int p, int n) {
            constexpr bool LOW = decltype(low_tag)::value, WIDE = decltype(wide_tag)::value;
            unsigned long long ar = 0, ai = 0, br = 0, bi = 0;
            float cr = 0.0f, ci = 0.0f;
#pragma unroll kRho64Unroll
            for (int u = p; u < p + n; ++u) {
                const int4 a = sp[2 * u], b = sp[2 * u + 1];
                uint32_t hi = (uint32_t)mv.x * (uint32_t)a.x + kPhaseStart;
                hi += (uint32_t)mv.y * (uint32_t)a.y;
                hi += (uint32_t)mv.z * (uint32_t)a.z;
                hi ^= (uint32_t)a.w & 0x80000000u;
                float lo = fmaf(mfx, __int_as_float(b.x), fmaf(mfy, __int_as_float(b.y), mfz * __int_as_float(b.z)));
                if (WIDE) phase_whole(hi, lo);
                const TrigEntry e = st[hi >> 21];
                const TrigLow w = sw[hi >> 21];
                const PhaseX x = phase_x(hi, lo);
                const float sf = fx_i2f(e.sa), cf = fx_i2f(e.ca);
                int sh, ch;
                float sl, cl;
                trig_value<1>(e.sa, sf, w.s, cf, w.c, x, sh, sl);
                trig_value<-1>(e.ca, cf, w.c, sf, w.s, x, ch, cl);
                const int qh = a.w & 0x7fffffff;
                const float qf = fx_i2f(qh);
                ar = mad_wide(ch, qh, ar);
                ai = mad_wide(sh, qh, ai);
                if (LOW) {
                    br = mad_wide(ch, b.w, br);
                    bi = mad_wide(sh, b.w, bi);
                }
                cr = fmaf(trig_low_f(e.cr, cl), qf, cr);
                ci = fmaf(trig_low_f(e.sr, sl), qf, ci);
            }
            re += ((__int128)(long long)ar << 28) + (long long)br + __float2ll_rn(cr * 0x1.0p28f);
            im += ((__int128)(long long)ai << 28) + (long long)bi + __float2ll_rn(ci * 0x1.0p28f);
        };
        for (int p = ss * share; p < p1; p += kRho64Group) {
            const int n = min(kRho64Group, p1 - p);
            if constexpr (CHECK) {
                if (wide) {
                    group(std::true_type{}, std::true_type{}, p, n);
                    continue;
                }
            }
            if (has_low) group(std::true_type{}, std::false_type{}, p, n);
            else group(std::false_type{}, std::false_type{}, p, n);
        }
    }
    __syncthreads();
    // the sub-streams' sums (integers: any order gives the same)
    __int128* sum = reinterpret_cast<__int128*>(sp);
    if (S > 1) {
        if (act) {
            sum[2 * (ss * T + j)] = re;
            sum[2 * (ss * T + j) + 1] = im;
        }
        __syncthreads();
        if (act && ss == 0)
            for (int s = 1; s < S; ++s) {
                re += sum[2 * (s * T + j)];
                im += sum[2 * (s * T + j) + 1];
            }
    }
    if (act && ss == 0) {
        const int e = eb - 1023 + 1 - 85;  // units of 2^-30 2^-55 of 2^(eb - 1023 + 1)
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        // an input that is not finite shows in every output, beside the latched status
        partials[(size_t)l * nchunks + c] =
            s_bad ? make_double2(nan, nan) : make_double2(int128_to_double(re, e), int128_to_double(im, e));
    }
    if (kt == 0 && tid == 0) partials[(size_t)K * nchunks + c] = make_double2(q2, 0.0);
}

// =================================================================================
// Reduction: block l (of K + 1) sums its row over the chunks in a fixed order; thread 0 forms the
// frequency's energy and virial terms (as on the FP32-phase path, freq_pre before the wait), the force
// amplitude R = c[7] |rho| and arg rho as a 64-bit fixed-point phase.
//
// arg rho without an FP64 arctangent (a chain of about 60 FP64 instructions of one warp, 4 us here): the
// FP32 arctangent, rounded to 2^-30 revolutions, as a first angle; its exact sine and cosine from the
// table; and the remaining angle (below 2^-22) from Im(rho e^{-i phi}) / |rho|.
__global__ void __launch_bounds__(kReduceThreads)
k_reduce_f64(const double2* __restrict__ partials, int nchunks, int K, const int4* __restrict__ m,
             const double* __restrict__ w, const KState* __restrict__ ks,
             double2* __restrict__ rho, double* __restrict__ terms, double2* __restrict__ coef,
             unsigned* __restrict__ status)
{
    __shared__ double red[2][32];
    const int l = blockIdx.x;
    // the sampler completed before the rho pass passed its wait, and the rho pass lets this
    // launch start only after that wait: m, w and ks are final here
    double c[8];
    if (threadIdx.x == 0 && l < K) freq_pre(m[l], w[l], ks, c);
    pdl_wait();
    pdl_trigger();
    double re = 0.0, im = 0.0;
    const double2* row = partials + (size_t)l * nchunks;
    for (int j = threadIdx.x; j < nchunks; j += blockDim.x) {
        const double2 v = row[j];
        re += v.x;
        im += v.y;
    }
    block_sum2(re, im, red);
    if (threadIdx.x != 0) return;
    double* t = terms + (size_t)l * 8;
    if (l == K) {
        t[0] = re;  // sum of q^2
        return;
    }
    const double rho2 = re * re + im * im;
    const double e = c[0] * rho2;
    t[0] = e;
#pragma unroll
    for (int a = 1; a < 7; ++a) t[a] = e * c[a];
    t[7] = 0.0;
    rho[l] = make_double2(re, im);
    unsigned long long phi = 0ull;
    double R = 0.0, h2 = rho2;
    if (((uint32_t)__double2hiint(rho2) >> 20) - 93u > 1860u) {
        // a square below 2^-930, above 2^930 or not finite: the forces are linear in rho, whose size is within FP64's
        const double big = fmax(fabs(re), fabs(im));
        if (!isfinite(re) || !isfinite(im)) {
            atomicOr(status, kStatusNonFinite);
            c[7] = re - re + (im - im);  // NaN
            h2 = 0.0;
        } else if (big > 0.0) {
            const int e = ilogb(big);
            re = ldexp(re, -e);
            im = ldexp(im, -e);
            c[7] = ldexp(c[7], e);
            h2 = re * re + im * im;
        }
    }
    if (h2 > 0.0) {
        const double inv = rsqrt(h2);
        R = fabs(c[7]) * (h2 * inv);
        const double cr = re * inv, ci = im * inv;  // (cos, sin) of arg rho
        const float rev = atan2f((float)ci, (float)cr) * 0.159154943f;
        phi = (unsigned long long)(long long)__float2int_rn(rev * 1073741824.0f) << 34;
        const uint32_t ph = (uint32_t)(phi >> 32) + kPhaseStart;
        const PhaseX x = phase_x(ph, 0.0f);
        const TrigEntry te = g_trig.entry[ph >> 21];
        const TrigLow tw = g_trig.low[ph >> 21];
        const float sf = fx_i2f(te.sa), cf = fx_i2f(te.ca);
        int sh, ch;
        float sl, cl;
        trig_value<1>(te.sa, sf, tw.s, cf, tw.c, x, sh, sl);
        trig_value<-1>(te.ca, cf, tw.c, sf, tw.s, x, ch, cl);
        const double s = (double)sh + (double)trig_low_f(te.sr, sl), co = (double)ch + (double)trig_low_f(te.cr, cl);
        // ci co - cr s = sin(arg rho - phi) in units of 2^-30; revolutions in units of 2^-64: 2^34 / 2 pi
        const double d = fma(ci, co, -(cr * s)) * 2734261102.3059327;
        phi += (unsigned long long)__double2ll_rn(d);
        if (c[7] < 0.0) phi += 1ull << 63;  // a negative weight is half a revolution: R enters the force pass as a magnitude
    } else {
        R = c[7] * 0.0;  // NaN for a rho, a weight or a 1 / |k|^2 that is not finite
    }
    coef[l] = make_double2(__longlong_as_double((long long)(0ull - phi)), R);
}

// =================================================================================
// Force pass: F_i,theta = q_i (2 pi / l_theta) sum_l R_l m_l,theta sin(theta_il - arg rho_l).
// A block takes rounds of kForce64Threads / SL particles (lanes) with the frequencies of a staged tile split
// over SL slices, whose integer sums are added at the end of the round: SL > 1 spreads small systems
// over the GPU.  Per staged tile the amplitudes R_l become integers: scaled so that sum_l |m_l| R_l
// (an FP32 bound, rounded up) is below 2^60, each product R sin is rounded to 2^-60 of that sum.
// The launch carries one extra block that computes the energy and virial sums (final_sums) meanwhile.
// CHECK: as in k_rho_f64, by the staged tile.
template <int SL, bool CHECK>
__global__ void __launch_bounds__(kForce64Threads, RBE_FORCE64_MINB)
k_force_f64(const double* __restrict__ pos, const double* __restrict__ q, int64_t N, int64_t per_block,
            const KState* __restrict__ ks, const int4* __restrict__ mk, const double2* __restrict__ coef, int K,
            double* __restrict__ F, unsigned* __restrict__ status,
            const double* __restrict__ terms, double* __restrict__ W_out, double* __restrict__ E_out)
{
    if (blockIdx.x == gridDim.x - 1) {
        pdl_wait();
        final_sums(terms, K, ks, W_out, E_out, status);
        return;
    }
    constexpr int PB = kForce64Threads / SL;
    extern __shared__ __align__(16) unsigned char s_raw[];
    TrigSine* st = reinterpret_cast<TrigSine*>(s_raw);
    const float* sw = reinterpret_cast<const float*>(st + kTrigN);
    // per frequency: (mx, my, mz, phase high), the same m as floats and the phase low, (R high, R low)
    int4* sk = reinterpret_cast<int4*>(s_raw + kForce64Trig);
    __shared__ unsigned long long s_sum[SL > 1 ? 3 : 1][SL > 1 ? kForce64Threads : 1];
    __shared__ int s_e;
    __shared__ float s_b[3][kForce64Threads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int pl = tid % PB, sl = tid / PB;
    load_trig(g_trig.sine, st, (int)kForce64Trig);
    pdl_wait();  // (ks: see k_rho_f64)
    const FixScale scx = fs(ks->sc64[0]), scy = fs(ks->sc64[1]), scz = fs(ks->sc64[2]);
    const double cx = 2.0 * kPi * ks->inv[0], cy = 2.0 * kPi * ks->inv[1], cz = 2.0 * kPi * ks->inv[2];
    const int64_t b0 = (int64_t)blockIdx.x * per_block, b1 = min(N, b0 + per_block);
    const bool one_tile = K <= kForce64Stage;
    int sh = 0;  // R as an integer is R 2^sh
    [[maybe_unused]] int wide = 0;  // the staged tile has frequencies beyond kPhaseNarrow
    for (int64_t base = b0; base < b1; base += PB) {
        const int64_t i = base + pl;
        Frac x{0, 0.0f}, y{0, 0.0f}, z{0, 0.0f};
        if (i < b1) {
            x = frac_of(fixed_frac64((unsigned long long)__double_as_longlong(pos[3 * i]), scx));
            y = frac_of(fixed_frac64((unsigned long long)__double_as_longlong(pos[3 * i + 1]), scy));
            z = frac_of(fixed_frac64((unsigned long long)__double_as_longlong(pos[3 * i + 2]), scz));
        }
        double fx = 0.0, fy = 0.0, fz = 0.0;
        for (int k0 = 0; k0 < K; k0 += kForce64Stage) {
            const int nk = min(kForce64Stage, K - k0);
            if (!one_tile || base == b0) {
                // one frequency per thread: exponent of the largest R, then sum |m| R in its units
                __syncthreads();
                int4 mm = make_int4(0, 0, 0, 0);
                double2 co = make_double2(0.0, 0.0);
                if (tid < nk) {
                    mm = mk[k0 + tid];
                    co = coef[k0 + tid];
                }
                if (tid == 0) s_e = 1;
                __syncthreads();
                const unsigned long long rb = (unsigned long long)__double_as_longlong(co.y);
                const int e = (int)((rb >> 52) & 0x7ffull);
                const int emax = __reduce_max_sync(0xffffffffu, e);
                if (lane == 0) atomicMax(&s_e, emax);
                __syncthreads();
                const int er = min(s_e, 0x7fe);
                // R 2^(1023 - er) below 2, as FP32 (23 mantissa bits, truncated)
                const float rf = e > 0 && e <= er && er - e < 64
                                     ? __uint_as_float(((uint32_t)(127 + e - er) << 23) | (uint32_t)((rb >> 29) & 0x7fffffu))
                                     : 0.0f;
                float bx = rf * fabsf((float)mm.x), by = rf * fabsf((float)mm.y), bz = rf * fabsf((float)mm.z);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    bx += __shfl_xor_sync(0xffffffffu, bx, off);
                    by += __shfl_xor_sync(0xffffffffu, by, off);
                    bz += __shfl_xor_sync(0xffffffffu, bz, off);
                }
                if (lane == 0) {
                    s_b[0][warp] = bx;
                    s_b[1][warp] = by;
                    s_b[2][warp] = bz;
                }
                __syncthreads();
                bx = by = bz = 0.0f;
#pragma unroll
                for (int v = 0; v < kForce64Threads / 32; ++v) {
                    bx += s_b[0][v];
                    by += s_b[1][v];
                    bz += s_b[2][v];
                }
                // the bound, at least 2 (the largest R itself), rounded up well above the FP32 sums' error
                const float bound = fmaxf(2.0f, fmaxf(bx, fmaxf(by, bz)) * 1.0001f);
                const int lg = (int)((__float_as_uint(bound) >> 23) & 0xffu) - 127 + 1;  // bound < 2^lg
                sh = 60 - lg + 1023 - er;  // sum |m| R 2^sh < 2^60
                if (tid < nk) {
                    // R 2^sh = mantissa 2^(e - 1075 + sh)
                    const unsigned long long mant = e > 0 ? (rb & 0xFFFFFFFFFFFFFull) | (1ull << 52) : 0ull;
                    const int k = e - 1075 + sh;
                    const unsigned long long A =
                        (k >= 0 ? mant << min(k, 63) : (k > -64 ? mant >> -k : 0ull)) + (1ull << 29);
                    const Frac off = frac_of((unsigned long long)__double_as_longlong(co.x));
                    sk[3 * tid] = make_int4(mm.x, mm.y, mm.z, (int)((uint32_t)off.hi + kPhaseStart));
                    sk[3 * tid + 1] = make_int4(__float_as_int((float)mm.x), __float_as_int((float)mm.y),
                                                __float_as_int((float)mm.z), __float_as_int(off.lo));
                    sk[3 * tid + 2] = make_int4((int)(A >> 30), (int)(A & 0x3FFFFFFFull) - (1 << 29), 0, 0);
                }
                if (CHECK) wide = __syncthreads_or(phase_is_wide(mm.x, mm.y, mm.z));
                else __syncthreads();
            }
            unsigned long long ax = 0, ay = 0, az = 0;
            uint32_t hx = 0, hy = 0, hz = 0;
            const int per = SL > 1 ? (nk + SL - 1) / SL : nk;
            const int l1 = SL > 1 ? min(nk, (sl + 1) * per) : nk;
            // the pair loop, and with CHECK before it a copy that moves the low phase's whole part: one of them runs
#pragma unroll
            for (int mode = CHECK ? 1 : 0; mode >= 0; --mode) {
                if (CHECK && (mode == 1) != (wide != 0)) continue;
#pragma unroll kForce64Unroll
                for (int l = SL > 1 ? sl * per : 0; l < l1; ++l) {
                    const int4 a = sk[3 * l], b = sk[3 * l + 1];
                    const int2 r = *reinterpret_cast<const int2*>(sk + 3 * l + 2);
                    uint32_t hi = (uint32_t)a.x * (uint32_t)x.hi + (uint32_t)a.w;
                    hi += (uint32_t)a.y * (uint32_t)y.hi;
                    hi += (uint32_t)a.z * (uint32_t)z.hi;
                    float lo = fmaf(__int_as_float(b.x), x.lo,
                                    fmaf(__int_as_float(b.y), y.lo, fmaf(__int_as_float(b.z), z.lo, __int_as_float(b.w))));
                    if (mode == 1) phase_whole(hi, lo);
                    const TrigSine e = st[hi >> 21];
                    const float vl0 = sw[hi >> 21];
                    const PhaseX p = phase_x(hi, lo);
                    int vh;
                    float vl;
                    trig_value<1>(e.sa, fx_i2f(e.sa), vl0, e.ch, e.cl, p, vh, vl);
                    const unsigned long long h = mul_fix(vh, trig_low_i(e.sr, vl), r.x, r.y);
                    const int hh = fx_hi(h), hl = fx_lo(h);
                    ax = mad_wide(a.x, hl, ax);
                    ay = mad_wide(a.y, hl, ay);
                    az = mad_wide(a.z, hl, az);
                    hx += (uint32_t)a.x * (uint32_t)hh;
                    hy += (uint32_t)a.y * (uint32_t)hh;
                    hz += (uint32_t)a.z * (uint32_t)hh;
                }
            }
            ax += (unsigned long long)hx << 32;
            ay += (unsigned long long)hy << 32;
            az += (unsigned long long)hz << 32;
            if (SL > 1) {
                __syncthreads();  // the previous round's sums have been read
                s_sum[0][tid] = ax;
                s_sum[1][tid] = ay;
                s_sum[2][tid] = az;
                __syncthreads();
                if (sl == 0)
#pragma unroll
                    for (int s = 1; s < SL; ++s) {
                        ax += s_sum[0][s * PB + pl];
                        ay += s_sum[1][s * PB + pl];
                        az += s_sum[2][s * PB + pl];
                    }
            }
            // units of 2^-30 (sine) times 2^30 (mul_fix's) over 2^sh
            if (sl == 0 && i < b1) {
                // (an R that is not finite: no force is)
                const double u = s_e == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(1.0, -sh);
                fx += u * (double)(long long)ax;
                fy += u * (double)(long long)ay;
                fz += u * (double)(long long)az;
            }
        }
        if (sl == 0 && i < b1) {
            const double qi = q[i];
            F[3 * i] = qi * cx * fx;
            F[3 * i + 1] = qi * cy * fy;
            F[3 * i + 2] = qi * cz * fz;
        }
    }
}

}  // namespace rbe
