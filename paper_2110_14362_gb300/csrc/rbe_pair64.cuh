// Pair terms of the FP64 real space from tables: force factor and energy of the erfc Coulomb and of the
// Lennard-Jones 12-6 potential as functions of u = r^2, to about 2^-52 (force) and 2^-45 (energy) per pair.
//
// Why: GB300 issues an FP64 instruction over about 76 clocks of a warp and scheduler, and sqrt, the
// division, exp and erfc of a pair are about 90 of them (the pair kernels kept the FP64 pipe 85 % busy).
//
// Each octave of u below the cutoff (eight of them) has 128 segments; in a segment the force factor is its
// Taylor polynomial of degree 8 about the centre (half a segment is at most 2^-8 of u, so each further
// term is about 2^-7 smaller, and the first one left out below 2^-58), the constant term in FP64 and the
// rest, at most 2^-5 of it, in float-float with FP32 for the small terms: two FP64 additions.  The
// segment and the argument come from the bits of u.  With dU/du = -f/2 the energy is the integral
// of the same polynomial from the segment's centre, in float-float throughout.
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

__host__ __device__ inline void pair_put_double(PairWord& p, double x)
{
    unsigned long long b;
#ifdef __CUDA_ARCH__
    b = (unsigned long long)__double_as_longlong(x);
#else
    __builtin_memcpy(&b, &x, 8);
#endif
    p.w[0] = (uint32_t)b;
    p.w[1] = (uint32_t)(b >> 32);
}

// Segment `seg` of the table whose octaves end at 2^top, both parts (Coulomb, LJ): coefficients c[k] of the
// polynomial in tau in [-1, 1] and the energy e0 at the centre.  Planes (kPairSegs entries each):
// {c0 FP64, e0 h, l}, {c1 h, l, c2 h, l}, {c3 h, l, c4 h, l}, {c5, c6, c7, c8}.
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
    double c[9], e0 = (erfc(x) - 1.12837916709551257390 * ga * dx) / r, B = e0, a2 = 1.0, f = 1.0;
    for (int n = 1; n <= 9; ++n) {
        a2 *= 2.0 * alpha;
        B = ((2 * n - 1) * B + a2 * ex) * iu;
        c[n - 1] = f * B;
        f *= -0.5 * h / (double)n;
    }
    for (int part = 0; part < 2; ++part) {
        if (part == 1) {
            const double y = lj_s2 * iu, y3 = y * y * y, hu = h * iu;
            double p7 = 2.0 * lj_e24 * y3 * y3 * iu, p4 = -lj_e24 * y3 * iu;  // u^-7 and u^-4 terms of f
            e0 = lj_e4 * (y3 * y3 - y3);
            for (int k = 0; k < 9; ++k) {
                c[k] = p7 + p4;
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
        pair_put_double(p[0], c[0]);
        two(0, 2, e0);
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

// A double's top 48 bits as a float-float, by its bits (normal and within the float range).
__host__ __device__ __forceinline__ FF ff_of(uint32_t hi, uint32_t lo)
{
    const uint32_t sign = hi & 0x80000000u, e = (hi >> 20) & 0x7ffu;
    const uint32_t m = ((hi & 0xFFFFFu) << 3) | (lo >> 29);  // 23 bits
    FF r;
    r.h = fx_float(sign | ((e - 896u) << 23) | m);
    // the next 24 bits times the unit 2^(e - 1023 - 47)
    const float rest = RBE_MUL(fx_i2f((int)((lo >> 5) & 0xFFFFFFu)), fx_float((e - 896u - 47u) << 23));
    r.l = fx_float(fx_bits(rest) | sign);
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

// The segment of u and its argument tau (exact, tau = h + l); seg is outside [0, kPairSegs) where u is.
struct PairArg {
    int seg;
    FF tau;
    float half;  // half the segment's half width
};

// base: (1023 + top - kPairOctaves) << kPairSegBits
__host__ __device__ __forceinline__ PairArg pair_arg(uint32_t hi, uint32_t lo, int base)
{
    PairArg a;
    a.seg = (int)(hi >> (20 - kPairSegBits)) - base;
    // the mantissa bits below the segment's: the first 23, and the others
    constexpr int k = kPairSegBits + 3;
    a.tau.h = RBE_FMA(2.0f, fx_float((((hi << k) | (lo >> (32 - k))) & 0x7FFFFFu) | 0x3F800000u), -3.0f);
    a.tau.l = RBE_FMA(fx_float(((lo << (k - 9)) & 0x7FFFFFu) | 0x3F800000u), 0x1.0p-22f, -0x1.0p-22f);
    // half width 2^(e - kPairSegBits - 1), halved
    a.half = fx_float((((hi >> 20) - 896u) - (uint32_t)(kPairSegBits + 2)) << 23);
    return a;
}

// Force factor (FP64) and energy (float-float) of one part (0: Coulomb, 1: LJ) from its table planes.
template <int PART>
__host__ __device__ __forceinline__ void pair_eval(const PairWord* t, const PairArg& a, double& f, FF& energy)
{
    const PairWord* p = t + PART * kPairPlanes * kPairSegs + a.seg;
    const PairWord w0 = p[0], w1 = p[kPairSegs], w2 = p[2 * kPairSegs], w3 = p[3 * kPairSegs];
    const FF tau = a.tau;
    const FF c1{fx_float(w1.w[0]), fx_float(w1.w[1])}, c2{fx_float(w1.w[2]), fx_float(w1.w[3])};
    const FF c3{fx_float(w2.w[0]), fx_float(w2.w[1])}, c4{fx_float(w2.w[2]), fx_float(w2.w[3])};
    const float c5 = fx_float(w3.w[0]), c6 = fx_float(w3.w[1]), c7 = fx_float(w3.w[2]), c8 = fx_float(w3.w[3]);
    const float s = RBE_FMA(RBE_FMA(RBE_FMA(c8, tau.h, c7), tau.h, c6), tau.h, c5);
    constexpr bool ANY = PART == 1;
    FF q = ff_fma<ANY>(FF{s, 0.0f}, tau, c4);
    q = ff_fma<ANY>(q, tau, c3);
    q = ff_fma<ANY>(q, tau, c2);
    q = ff_fma<ANY>(q, tau, c1);
    q = ff_mul(q, tau);
#ifdef __CUDA_ARCH__
    f = __dadd_rn(__dadd_rn(__hiloint2double((int)w0.w[1], (int)w0.w[0]), float_as_double(q.h)), float_as_double(q.l));
#else
    double d0;
    const unsigned long long b = ((unsigned long long)w0.w[1] << 32) | w0.w[0];
    __builtin_memcpy(&d0, &b, 8);
    f = (d0 + float_as_double(q.h)) + float_as_double(q.l);
#endif
    // energy e0 - half tau (c0 + tau (c1 / 2 + tau (c2 / 3 + tau (c3 / 4 + ...))))
    float si = RBE_FMA(RBE_MUL(c6, 1.0f / 7.0f), tau.h, RBE_MUL(c5, 1.0f / 6.0f));
    si = RBE_FMA(si, tau.h, RBE_MUL(c4.h, 0.2f));
    si = RBE_FMA(si, tau.h, RBE_MUL(c3.h, 0.25f));
    const FF third{(float)(1.0 / 3.0), (float)(1.0 / 3.0 - (double)(float)(1.0 / 3.0))};
    FF in = ff_fma<ANY>(FF{si, 0.0f}, tau, ff_mul(c2, third));
    in = ff_fma<ANY>(in, tau, FF{RBE_MUL(0.5f, c1.h), RBE_MUL(0.5f, c1.l)});
    in = ff_fma<ANY>(in, tau, ff_of(w0.w[1], w0.w[0]));
    energy = ff_fma<ANY>(in, FF{RBE_MUL(-a.half, tau.h), RBE_MUL(-a.half, tau.l)}, FF{fx_float(w0.w[2]), fx_float(w0.w[3])});
}

// ---------------------------------------------------------------------------------
// Device side: the table in shared memory and the accumulation of one pair.
#ifdef __CUDACC__

constexpr int kPair64Warps = 16;  // warps of an FP64 pair block: one block per SM, its warps share the table

// The FP64 pair kernels' constants beside PairConst.
struct Pair64Const {
    const PairWord* tab;  // device table, NULL: direct evaluation (cutoff or LJ sizes beyond the float range)
    int base;             // (1023 + top - kPairOctaves) << kPairSegBits
    int lj;
    double alpha, sa, two_sa_pi, qk, s2, e4, e24;
    unsigned long long rc2;  // bits of rc^2
};

// Sums of one lane: the particle's force, and over all particles of the warp the virial (its trace, or its
// diagonal), and the energies: Coulomb without the Coulomb constant.
template <bool DIAG>
struct Pair64Sums {
    double fx, fy, fz;
    double w[DIAG ? 3 : 1];
    FF ecp, ec, el;   // ecp: sum_j q_j E of the current particle
    double ecd, eld;  // energies of the pairs evaluated directly
};

__device__ __forceinline__ FF ff_of_double(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    return (hi & 0x7ff00000u) == 0u ? FF{0.0f, 0.0f} : ff_of(hi, lo);
}

// A charge that float-floats hold to 48 bits: zero, or between 2^-60 and 2^60.
__device__ __forceinline__ bool charge_fits(double q)
{
    const uint32_t e = ((uint32_t)__double2hiint(q) >> 20) & 0x7ffu;
    return e == 0u || (e > 963u && e < 1083u);
}

// One pair: separation d (from i to the neighbour), r2 = |d|^2 < rc^2, charges qi, qj.
template <bool DIAG>
__device__ __forceinline__ void pair64_add(const PairWord* __restrict__ tab, const Pair64Const& pc, bool lj, double dx,
                                           double dy, double dz, double r2, double qi, double qj, double qki,
                                           Pair64Sums<DIAG>& s)
{
    const PairArg a = pair_arg((uint32_t)__double2hiint(r2), (uint32_t)__double2loint(r2), pc.base);
    double f;
    if (pc.tab && (unsigned)a.seg < (unsigned)kPairSegs && charge_fits(qj) && charge_fits(qi)) {
        FF e;
        pair_eval<0>(tab, a, f, e);
        f *= qki * qj;
        ff_acc(s.ecp, ff_mul(e, ff_of_double(qj)));
        if (lj) {
            double fl;
            pair_eval<1>(tab, a, fl, e);
            f += fl;
            ff_acc(s.el, e);
        }
    } else {
        // below the table (r under 1/16 of the cutoff at least) or outside the float range
        const double r = sqrt(r2), inv_r = 1.0 / r, inv_r2 = inv_r * inv_r;
        const double coul = qki * qj * inv_r, er = erfc(pc.sa * r);
        s.ecd += coul * er;
        f = coul * (er + pc.two_sa_pi * r * exp(-pc.alpha * r2)) * inv_r2;
        if (lj) {
            const double sr2 = pc.s2 * inv_r2, sr6 = sr2 * sr2 * sr2;
            s.eld += pc.e4 * (sr6 * sr6 - sr6);
            f += pc.e24 * (2.0 * sr6 * sr6 - sr6) * inv_r2;
        }
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

// The warp's force sums of one particle: a transposing tree (6 FP64 additions instead of 15) that ends with x,
// y, z in lanes 0, 8, 16; they are written to F[3 i], F[3 i + 1], F[3 i + 2].
__device__ __forceinline__ void warp_force_out(double fx, double fy, double fz, int lane, double* __restrict__ F)
{
    const bool up = lane & 16, mid = lane & 8;
    double k0 = up ? fz : fx, k1 = up ? 0.0 : fy;
    k0 += __shfl_xor_sync(0xffffffffu, up ? fx : fz, 16);
    k1 += __shfl_xor_sync(0xffffffffu, up ? fy : 0.0, 16);
    double k = mid ? k1 : k0;
    k += __shfl_xor_sync(0xffffffffu, mid ? k0 : k1, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) k += __shfl_xor_sync(0xffffffffu, k, off);
    if ((lane & 7) == 0 && lane < 24) F[lane >> 3] = k;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Block partials of the sums: half of each (every pair is visited from both ends), virial components from slot
// o, then E_coul (times the Coulomb constant) and E_lj.  All threads of the block.
template <bool DIAG>
__device__ __forceinline__ void pair64_partials(const Pair64Sums<DIAG>& s, double qk, double (*red)[kPair64Warps],
                                                double* __restrict__ partials, int o)
{
    constexpr int nw = DIAG ? 3 : 1;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < nw + 2; ++k) {
        const double v = k < nw ? s.w[k < nw ? k : 0]
                                : (k == nw ? qk * ((double)s.ec.h + (double)s.ec.l) + s.ecd
                                           : (double)s.el.h + (double)s.el.l + s.eld);
        const double t = warp_sum(v);
        if (lane == 0) red[k][wib] = t;
    }
    __syncthreads();
    if (threadIdx.x < nw + 2) {
        double t = 0.0;
        for (int v = 0; v < kPair64Warps; ++v) t += red[threadIdx.x][v];
        partials[o + threadIdx.x] = 0.5 * t;
    }
}

// Lane's segment of the slots of the 27 cells around cell c: row r = lane / 2 of the 3 x 3 rows (dy, dz), part
// lane % 2 (a row that wraps in x has two); [lo, hi) and the image shift (sx, sy, sz), 0 on an axis whose
// image is taken per pair (mi).  An axis with fewer than 3 cells visits each of them once.  False: no
// segment.
__device__ __forceinline__ bool pair_segment_of(int c, const int nc[3], int lane, const bool mi[3],
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
    sx = 0;
    sy = mi[1] ? 0 : (uy < 0 ? -1 : (uy >= nc[1] ? 1 : 0));
    sz = mi[2] ? 0 : (uz < 0 ? -1 : (uz >= nc[2] ? 1 : 0));
    const int row = (zz * nc[1] + yy) * nc[0], nx = nc[0];
    int a = -1, e = -1;  // cells a..e of the row
    if (nx < 3) {
        if (part == 0) a = 0, e = nx - 1;
    } else if (cx == 0) {
        if (part == 0) a = 0, e = 1;
        else a = e = nx - 1, sx = -1;
    } else if (cx == nx - 1) {
        if (part == 0) a = nx - 2, e = nx - 1;
        else a = e = 0, sx = 1;
    } else if (part == 0) {
        a = cx - 1, e = cx + 1;
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
