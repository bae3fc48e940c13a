// Langevin NPT step of rigid 3-site water on the device (the paper's water runs keep molecules
// rigid, Sec. 5.1; the equations of Sec. 3.2 act on the molecular centres, SHAKE and RATTLE hold
// the internal geometry).  Sites are stored O, H, H per molecule; molecules stay whole in storage
// (after each step a molecule moves by the lattice vector that brings its oxygen into the box).
//
// One step is a fixed sequence of launches on the context's stream:
//   k_npt_cell_a    the isotropic cell part (rbe_npt.cu): V^p/2 with the molecular pressure, the
//                   sub-step coefficients, V/2, O^p, V/2, the cell-list constants
//   k_water_drift   one thread per molecule: R^p/2, R/2, O, R/2 of the centre (exact flows) and of
//                   the internal motion (kick, free move, SHAKE, momentum correction, projection)
//   k-space         tables of the device box, sampler, rho, force pass over all sites (on a side stream beside
//                   the drift and the real space, KspaceFork in rbe_npt.cu)
//   cell list       count, scan, fill, sort (rbe_npt.cu)
//   k_water_pair    one warp per site: erfc Coulomb with sites of other molecules, LJ between
//                   oxygens, nearest image per pair
//   k_water_finish  one thread per molecule: total forces with the intramolecular exclusion,
//                   R^p/2, the centres' 2K and the molecular virial; last block: P_ins, V^p/2
// FP64 state and sums; the pair terms as in rbe_pair64.cuh, the constraints' 3x3 solves in FP32 on FP64 residuals
// (w_shake); the k-space follows the context's precision.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "rbe_context.h"
#include "rbe_device.cuh"
#include "rbe_npt_common.cuh"
#include "rbe_pair64.cuh"

namespace rbe {

// Molecules per block of the per-molecule kernels (k_water_whole, k_water_drift, k_water_finish):
// one warp's, so that their FP64 constraint and virial arithmetic spreads over as many SMs'
// FP64 pipes as there are warps of molecules (3000 molecules: 94 SMs, against 24 with blocks of
// 128, where the drift took 97 us bound by the FP64 pipe of those 24 SMs).  The drift and the
// finishing kernel give a block three more warps, on the SM's other three schedulers, for what does not
// depend on the chain of constraints: the normals of one site, the exclusion of one site pair.
constexpr int kWaterThreads = 32;
constexpr int kWaterWarps = 4;
constexpr int kCellExcl = 25;       // cell block: the exclusion energy
constexpr int kWaterHitCap = 64;    // buffered candidates per warp (< 32 buffered + 32 new)

// the sites of constraint c: (0,1), (0,2), (1,2)
__host__ __device__ constexpr int wpa(int c) { return c == 2 ? 1 : 0; }
__host__ __device__ constexpr int wpb(int c) { return c == 0 ? 1 : 2; }

// The molecule starting at site 3I made whole from its oxygen by the nearest image.
__device__ __forceinline__ void w_whole(const double* __restrict__ pos, int64_t I, const double L[3],
                                        const double inv[3], double x[3][3])
{
    #pragma unroll
    for (int t = 0; t < 3; ++t) x[0][t] = pos[9 * I + t];
    for (int s = 1; s < 3; ++s)
        #pragma unroll
        for (int t = 0; t < 3; ++t) {
            const double d = pos[9 * I + 3 * s + t] - x[0][t];
            x[s][t] = x[0][t] + (d - L[t] * rint(d * inv[t]));
        }
}

__device__ __forceinline__ double det3(const double A[3][3])
{
    return A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) - A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
           A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
}

// x = A^{-1} b by Cramer's rule with one reciprocal of det A.
__device__ __forceinline__ void solve3(const double A[3][3], const double b[3], double x[3])
{
    const double id = 1.0 / det3(A);
    #pragma unroll
    for (int k = 0; k < 3; ++k) {
        double B[3][3];
        #pragma unroll
        for (int c = 0; c < 3; ++c)
            #pragma unroll
            for (int d = 0; d < 3; ++d) B[c][d] = d == k ? b[c] : A[c][d];
        x[k] = det3(B) * id;
    }
}

// x / y with r = 1 / y: the product and its residual's correction (Markstein 1990: correctly rounded but for
// rare last bits), three instructions for the division's ten.
__device__ __forceinline__ double w_div(double x, double y, double r)
{
    const double q = x * r;
    return fma(fma(-q, y, x), r, q);
}

// A double as a float: its leading bits (0 below the float range, infinity above it).
__device__ __forceinline__ float w_float(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7ffu;
    if (e > 1150u) return __int_as_float(0x7f800000);
    return e < 897u ? 0.0f : __uint_as_float((hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
}

// The change of (x_a - x_b) of constraint c per unit multiplier of constraint d, in units of
// s_d: ((a_c == a_d) - (a_c == b_d))/m_{a_c} - ((b_c == a_d) - (b_c == b_d))/m_{b_c}.
__device__ __forceinline__ double coupling(int c, int d, const double im[3])
{
    const int a = wpa(c), b = wpb(c);
    return ((a == wpa(d)) - (a == wpb(d))) * im[a] - ((b == wpa(d)) - (b == wpb(d))) * im[b];
}

// The position constraints of one molecule after an unconstrained move from the constrained xo:
// x_i <- x_i + sum_d lambda_d s_old,d (e_{i,a_d} - e_{i,b_d}) / m_i with lambda making every
// |x_a - x_b|^2 = d^2, the equations SHAKE solves (corrections along the old separations).  Here by
// Newton's method on lambda (quadratic convergence from lambda = 0): it stops once every
// |r^2 - d^2| <= tol d^2, at the root SHAKE's sweeps converge to.  Returns false when max_iter iterations did
// not get there.  The residuals and the moves are FP64; the 3x3 solves are FP32, which leaves about 2^-20 of a
// residual beside the quadratic term (the same two or three iterations, for 42 FP64 instructions each instead
// of 127), and FP64 in the last four iterations allowed.
__device__ bool w_shake(double x[3][3], const double xo[3][3], const double im[3], const rbe_water_params& wp)
{
    const double dd[3] = {wp.d_OH * wp.d_OH, wp.d_OH * wp.d_OH, wp.d_HH * wp.d_HH};
    double so[3][3];
    float sof[3][3], K2[3][3];
    #pragma unroll
    for (int c = 0; c < 3; ++c) {
        #pragma unroll
        for (int t = 0; t < 3; ++t) {
            so[c][t] = xo[wpa(c)][t] - xo[wpb(c)][t];
            sof[c][t] = (float)so[c][t];
        }
        #pragma unroll
        for (int d = 0; d < 3; ++d) K2[c][d] = (float)(2.0 * coupling(c, d, im));
    }
    for (int it = 0; it < wp.shake_max_iter; ++it) {
        double s[3][3], g[3], dl[3];
        bool done = true;
        #pragma unroll
        for (int c = 0; c < 3; ++c) {
            g[c] = -dd[c];
            #pragma unroll
            for (int t = 0; t < 3; ++t) {
                s[c][t] = x[wpa(c)][t] - x[wpb(c)][t];
                g[c] = fma(s[c][t], s[c][t], g[c]);
            }
            if (fabs(g[c]) > wp.shake_tol * dd[c]) done = false;
        }
        if (done) return true;
        float det = 0.0f;
        if (it + 4 < wp.shake_max_iter) {
            float sf[3][3], J[3][3], cof[3][3];
            #pragma unroll
            for (int c = 0; c < 3; ++c)
                #pragma unroll
                for (int t = 0; t < 3; ++t) sf[c][t] = w_float(s[c][t]);
            #pragma unroll
            for (int c = 0; c < 3; ++c)
                #pragma unroll
                for (int d = 0; d < 3; ++d)
                    J[c][d] = K2[c][d] * (sf[c][0] * sof[d][0] + sf[c][1] * sof[d][1] + sf[c][2] * sof[d][2]);
            #pragma unroll
            for (int c = 0; c < 3; ++c)
                #pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const int c1 = (c + 1) % 3, c2 = (c + 2) % 3, d1 = (d + 1) % 3, d2 = (d + 2) % 3;
                    cof[c][d] = J[c1][d1] * J[c2][d2] - J[c1][d2] * J[c2][d1];
                }
            det = J[0][0] * cof[0][0] + J[0][1] * cof[0][1] + J[0][2] * cof[0][2];
            const float id = -1.0f / det, r0 = id * (float)g[0], r1 = id * (float)g[1], r2 = id * (float)g[2];
            #pragma unroll
            for (int d = 0; d < 3; ++d) dl[d] = (double)(cof[0][d] * r0 + cof[1][d] * r1 + cof[2][d] * r2);
        }
        if (!(fabsf(det) > 1e-24f && fabsf(det) < 1e24f)) {  // the last iterations, or far from a molecule's sizes
            double J[3][3];
            #pragma unroll
            for (int c = 0; c < 3; ++c) {
                g[c] = -g[c];
                #pragma unroll
                for (int d = 0; d < 3; ++d)
                    J[c][d] = 2.0 * coupling(c, d, im) * (s[c][0] * so[d][0] + s[c][1] * so[d][1] + s[c][2] * so[d][2]);
            }
            solve3(J, g, dl);
        }
        #pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double la = dl[d] * im[wpa(d)], lb = dl[d] * im[wpb(d)];
            #pragma unroll
            for (int t = 0; t < 3; ++t) {
                x[wpa(d)][t] += la * so[d][t];
                x[wpb(d)][t] -= lb * so[d][t];
            }
        }
    }
    return false;
}

// RATTLE's velocity stage: p_i += sum_c mu_c s_c (e_{i,a_c} - e_{i,b_c}), s_c = x_{a_c} - x_{b_c},
// mu solving the 3x3 system that makes every (v_a - v_b) . s_c vanish (Cramer's rule).
__device__ void w_project(double p[3][3], const double x[3][3], const double im[3])
{
    double s[3][3];
    #pragma unroll
    for (int c = 0; c < 3; ++c)
        #pragma unroll
        for (int t = 0; t < 3; ++t) s[c][t] = x[wpa(c)][t] - x[wpb(c)][t];
    double A[3][3], b[3], mu[3];
    #pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int a = wpa(c), bb = wpb(c);
        double dv = 0.0;
        #pragma unroll
        for (int t = 0; t < 3; ++t) dv += (p[a][t] * im[a] - p[bb][t] * im[bb]) * s[c][t];
        b[c] = -dv;
        #pragma unroll
        for (int d = 0; d < 3; ++d)
            A[c][d] = coupling(c, d, im) * (s[c][0] * s[d][0] + s[c][1] * s[d][1] + s[c][2] * s[d][2]);
    }
    solve3(A, b, mu);
    #pragma unroll
    for (int c = 0; c < 3; ++c)
        #pragma unroll
        for (int t = 0; t < 3; ++t) {
            p[wpa(c)][t] += mu[c] * s[c][t];
            p[wpb(c)][t] -= mu[c] * s[c][t];
        }
}

// R^p/2 of one molecule: the centre's exact flow P <- P a + 100 F b, the internal momenta kicked by
// 100 h (F_i - m_i F / M), then the projection.
__device__ void w_kick(double p[3][3], const double F[3][3], const double x[3][3], const double m3[3],
                       const double im[3], double a, double b, double h)
{
    const double M = m3[0] + m3[1] + m3[2], rM = 1.0 / M;
    double P[3] = {0.0, 0.0, 0.0}, Ft[3] = {0.0, 0.0, 0.0};
    #pragma unroll
    for (int k = 0; k < 3; ++k)
        #pragma unroll
        for (int t = 0; t < 3; ++t) {
            P[t] += p[k][t];
            Ft[t] += F[k][t];
        }
    double dP[3];
    #pragma unroll
    for (int t = 0; t < 3; ++t) dP[t] = P[t] * a + kFConv * Ft[t] * b - P[t];
    #pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double mM = w_div(m3[k], M, rM);
        #pragma unroll
        for (int t = 0; t < 3; ++t) p[k][t] += kFConv * h * (F[k][t] - mM * Ft[t]) + mM * dP[t];
    }
    w_project(p, x, im);
}

// R/2 of one molecule: the centre R <- R + R (a - 1) + cap((P/M) b), the offsets moved by h (p/m
// - P/M) and SHAKEn, the SHAKE displacement added to the momenta as m dd / h, then the projection
// at the new positions.  Returns false when SHAKE did not converge.
__device__ bool w_drift(double x[3][3], double p[3][3], const double m3[3], const double im[3], double am1, double b,
                        double h, double cap, const rbe_water_params& wp)
{
    const double M = m3[0] + m3[1] + m3[2], rM = 1.0 / M, rh = 1.0 / h;
    double R[3], P[3] = {0.0, 0.0, 0.0}, d[3][3], dn[3][3], ds[3][3];
    #pragma unroll
    for (int t = 0; t < 3; ++t) R[t] = w_div(m3[0] * x[0][t] + m3[1] * x[1][t] + m3[2] * x[2][t], M, rM);
    #pragma unroll
    for (int k = 0; k < 3; ++k)
        #pragma unroll
        for (int t = 0; t < 3; ++t) {
            P[t] += p[k][t];
            d[k][t] = x[k][t] - R[t];
        }
    double D[3], V[3];
    #pragma unroll
    for (int t = 0; t < 3; ++t) {
        V[t] = w_div(P[t], M, rM);
        D[t] = V[t] * b;
    }
    if (cap > 0.0) {
        const double len = sqrt(D[0] * D[0] + D[1] * D[1] + D[2] * D[2]);
        if (len > cap)
            #pragma unroll
            for (int t = 0; t < 3; ++t) D[t] *= cap / len;
    }
    double Rn[3];
    #pragma unroll
    for (int t = 0; t < 3; ++t) Rn[t] = R[t] + R[t] * am1 + D[t];
    #pragma unroll
    for (int k = 0; k < 3; ++k)
        #pragma unroll
        for (int t = 0; t < 3; ++t) {
            dn[k][t] = d[k][t] + h * (p[k][t] * im[k] - V[t]);
            ds[k][t] = dn[k][t];
        }
    const bool ok = w_shake(ds, d, im, wp);
    #pragma unroll
    for (int k = 0; k < 3; ++k)
        #pragma unroll
        for (int t = 0; t < 3; ++t) {
            p[k][t] += w_div(m3[k] * (ds[k][t] - dn[k][t]), h, rh);
            x[k][t] = Rn[t] + ds[k][t];
        }
    w_project(p, x, im);
    return ok;
}

// The molecules made whole from their oxygen and moved by the lattice vector that brings the
// oxygen into [0, L) (rbe_water_init: the caller's sites may be wrapped one by one).
__global__ void __launch_bounds__(kWaterThreads)
k_water_whole(int64_t Nmol, double* __restrict__ pos, const double* __restrict__ cell)
{
    const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= Nmol) return;
    const double L[3] = {cell[0], cell[1], cell[2]};
    const double inv[3] = {1.0 / L[0], 1.0 / L[1], 1.0 / L[2]};
    double x[3][3];
    w_whole(pos, I, L, inv, x);
    #pragma unroll
    for (int t = 0; t < 3; ++t) {
        const double sh = L[t] * floor(x[0][t] * inv[t]);
        #pragma unroll
        for (int k = 0; k < 3; ++k) pos[9 * I + 3 * k + t] = x[k][t] - sh;
    }
}

// Particles before the forces, one thread of warp 0 per molecule: R^p/2, R/2, O, R/2, the wrap by molecule; warp
// 1 + k forms site k's noise meanwhile.  Bound by the serial FP64 chain of warp 0, about 76 clocks an
// instruction: 3000 molecules 85 -> 55 us with the noise on other warps, quotients by reciprocals and the FP32
// constraint solves.
__global__ void __launch_bounds__(kWaterThreads * kWaterWarps)
k_water_drift(int64_t Nmol, double* __restrict__ pos, double* __restrict__ mom, const double* __restrict__ force,
              const double* __restrict__ mass, const NptCoef* __restrict__ cfp, uint64_t seed,
              const double* __restrict__ cell, const rbe_water_params wp, double dt, unsigned* __restrict__ status)
{
    __shared__ double sz[3][3][kWaterThreads];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t I = (int64_t)blockIdx.x * kWaterThreads + lane;
    const bool on = I < Nmol;
    const NptCoef& c = *cfp;
    const double h = 0.5 * dt;
    double x[3][3], p[3][3], m3[3], im[3];
    bool ok = true;
    if (on && warp > 0) {
        const int k = warp - 1;
        double z[4] = {0.0, 0.0, 0.0, 0.0};
        if (c.noise) npt_normals(seed, 1u, cell_step(cell), (uint32_t)(3 * I + k), z);
        const double s = c.sog * sqrt(mass[3 * I + k]);
        #pragma unroll
        for (int t = 0; t < 3; ++t) sz[k][t][lane] = s * z[t];
    } else if (on) {
        double F[3][3];
        w_whole(pos, I, c.L, c.invL, x);
        #pragma unroll
        for (int k = 0; k < 3; ++k) {
            m3[k] = mass[3 * I + k];
            im[k] = 1.0 / m3[k];
            #pragma unroll
            for (int t = 0; t < 3; ++t) {
                p[k][t] = mom[9 * I + 3 * k + t];
                F[k][t] = force[9 * I + 3 * k + t];
            }
        }
        w_kick(p, F, x, m3, im, c.a1[0], c.b1[0], h);
        ok = w_drift(x, p, m3, im, c.a2m1[0], c.b2[0], h, c.half_cap, wp);
    }
    __syncthreads();  // the one barrier of every thread of the block
    if (warp > 0 || !on) return;
    #pragma unroll
    for (int k = 0; k < 3; ++k)
        #pragma unroll
        for (int t = 0; t < 3; ++t) p[k][t] = p[k][t] * c.g + sz[k][t][lane];
    w_project(p, x, im);
    ok = w_drift(x, p, m3, im, c.a3m1[0], c.b3[0], h, c.half_cap, wp) && ok;
    if (!ok) atomicOr(status, kStatusShake);
    #pragma unroll
    for (int t = 0; t < 3; ++t) {
        const double sh = c.L[t] * floor(x[0][t] * c.invL[t]);
        #pragma unroll
        for (int k = 0; k < 3; ++k) {
            pos[9 * I + 3 * k + t] = x[k][t] - sh;
            mom[9 * I + 3 * k + t] = p[k][t];
        }
    }
}

// ---------------------------------------------------------------------------------
// Real space between sites of different molecules (Sec. 4.1 Eqs. (U2), (force)) on the cell list
// of the current box: one warp per site in cell order; the lanes set up the 18 row segments of
// the neighbouring cells (an axis with fewer than 3 cells visits each of its cells once) and
// stride over their slots; the separation is the nearest image per pair (sites may sit up to a
// bond outside the box).  The search runs on the FP32 packed positions with rc plus a margin above
// their rounding; the hits (slot, image code) go to a per-warp buffer in ballot order and are evaluated 32
// at a time, one per lane, from the fixed-point positions with the exact cutoff; the pair terms come
// from the tables of rbe_pair64.cuh, the sums are FP64 (k_pair64 says more; in a box with an edge shorter than
// 2 rc + 0.1 %, or than `few`, five bonds, where sites on opposite sides can be 1.5 edges apart, the image is taken
// per pair).  Half of it is the search: cells out of reach are left out
// (195 -> 164 us at 9000 sites), 24 warps a block (164 -> 150 us; 146 with energies in FP64).  A hit of the
// same molecule (site index / 3) is skipped; LJ acts between oxygens (site index divisible by 3).
// Each pair is
// visited from both ends: energies and the virial take half.  Per-block partials {W_r, E_coul,
// E_lj} at slots 1..3 (the isotropic layout).  A box beyond the cell arrays leaves F_r = 0.
__global__ void __launch_bounds__(kWaterPairWarps * 32, 1)
k_water_pair(int64_t N, const CellConsts* __restrict__ cc, const Pair64Const pc, double rc, double few,
             const int* __restrict__ cid, const int* __restrict__ cnt, const int* __restrict__ start, const int* __restrict__ sorted,
             const float4* __restrict__ spos32, const double4_32a* __restrict__ spos64, double* __restrict__ Fr,
             double* __restrict__ partials)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    PairWord* tab = reinterpret_cast<PairWord*>(s_raw);
    __shared__ int2 hits[kWaterPairWarps][kWaterHitCap];  // candidates within the FP32 search radius
    __shared__ double red[3][kWaterPairWarps];
    __shared__ double pforce[kWaterPairWarps][3];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    load_pair_table(pc.tab, tab);  // before the wait, as in k_pair64
    pdl_wait();
    Pair64Sums<false> s{};
    __syncthreads();
    if (cc->ncell < 0) {
        for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < 3 * N; j += (int64_t)gridDim.x * blockDim.x)
            Fr[j] = 0.0;
    } else {
        const int nc[3] = {cc->nc[0], cc->nc[1], cc->nc[2]};
        const double L[3] = {cc->L[0], cc->L[1], cc->L[2]};
        const float Lf[3] = {cc->Lf[0], cc->Lf[1], cc->Lf[2]}, invf[3] = {cc->invLf[0], cc->invLf[1], cc->invLf[2]};
        const PairBox box = pair_box(L, rc, pc.unit.s);
        const double lmin = fmin(L[0], fmin(L[1], L[2]));
        const bool exact = 2.0 * rc > 0.999 * lmin || lmin < few;
        const bool mi[3] = {true, true, true};  // the segments carry no image: it is taken per pair
        const float pass = cc->pass64;
        const int64_t per = (N + gridDim.x - 1) / gridDim.x;
        const int u1 = (int)min(N, (blockIdx.x + 1) * per);
        const float wid[3] = {Lf[0] / nc[0], Lf[1] / nc[1], Lf[2] / nc[2]};
        for (int base = (int)(blockIdx.x * per); base < u1; base += kWaterPairWarps) {
            int part, parts, i = 0;
            const int u = pair_round<kWaterPairWarps>(base, u1, wib, part, parts);
            s.fx = s.fy = s.fz = 0.0;
            if (u >= 0) {
                i = sorted[u];
                const double4_32a me = spos64[u];
                const float4 me32 = spos32[u];
                const int mol_i = i / 3;
                const bool oxy_i = i % 3 == 0 && pc.lj;
                const double qki = pc.qk * me.w;
                int lo = 0, hi = 0, sx, sy, sz, nh = 0;
                const float frac[3] = {pair_cell_coord(me32.x, invf[0], nc[0]), pair_cell_coord(me32.y, invf[1], nc[1]),
                                       pair_cell_coord(me32.z, invf[2], nc[2])};
                pair_segment_of(cid[i], nc, frac, wid, pass, lane, mi, cnt, start, lo, hi, sx, sy, sz);
                auto evaluate = [&](int count) {
                    const bool on = lane < count;
                    const int2 h = on ? hits[wib][lane] : make_int2(u, 1 | (1 << 2) | (1 << 4));
                    const int j = sorted[h.x];
                    const double4_32a o = spos64[h.x];
                    long long dx = pair_diff(o.x, me.x), dy = pair_diff(o.y, me.y), dz = pair_diff(o.z, me.z);
                    if (exact) {
                        const float4 o32 = spos32[h.x];
                        dx = pair_nearest(dx, o32.x - me32.x, invf[0], box.L[0], box.near[0]);
                        dy = pair_nearest(dy, o32.y - me32.y, invf[1], box.L[1], box.near[1]);
                        dz = pair_nearest(dz, o32.z - me32.z, invf[2], box.L[2], box.near[2]);
                    } else if (__any_sync(0xffffffffu, h.y != (1 | (1 << 2) | (1 << 4)))) {
                        dx = pair_shift(dx, h.y & 3, box.L[0]);
                        dy = pair_shift(dy, (h.y >> 2) & 3, box.L[1]);
                        dz = pair_shift(dz, (h.y >> 4) & 3, box.L[2]);
                    }
                    const unsigned long long n = pair_r2(dx, dy, dz, kPairHalf);
                    // another molecule (the site itself excluded with its own) and r2 < rc^2
                    if (on && j / 3 != mol_i && n < pc.unit.rc2)
                        pair64_add<false>(tab, pc, oxy_i && j % 3 == 0, dx, dy, dz, n, qki * o.w, s);
                    __syncwarp();
                };
                for (int g = 0; g < 18; ++g) {
                    const int glo = __shfl_sync(0xffffffffu, lo, g), ghi = __shfl_sync(0xffffffffu, hi, g);
                    for (int s0 = glo + 32 * part; s0 < ghi; s0 += 32 * parts) {  // the same trip count on every lane
                        const int sl = s0 + lane;
                        const float4 o = spos32[sl < ghi ? sl : glo];
                        float dx = o.x - me32.x, dy = o.y - me32.y, dz = o.z - me32.z;
                        // sites lie within a bond of [0, l): in boxes of more than a few bonds the image is -1, 0 or 1
                        // (rounded by adding 1.5 2^23: rintf runs on a quarter-rate pipe)
                        const float kx = (dx * invf[0] + 12582912.f) - 12582912.f, ky = (dy * invf[1] + 12582912.f) - 12582912.f,
                                    kz = (dz * invf[2] + 12582912.f) - 12582912.f;
                        dx -= Lf[0] * kx;
                        dy -= Lf[1] * ky;
                        dz -= Lf[2] * kz;
                        const bool hit = sl < ghi && sl != u && dx * dx + dy * dy + dz * dz < pass;
                        const unsigned m = __ballot_sync(0xffffffffu, hit);
                        if (hit) {
                            const int code = (1 - (int)kx) | ((1 - (int)ky) << 2) | ((1 - (int)kz) << 4);
                            hits[wib][nh + __popc(m & ((1u << lane) - 1u))] = make_int2(sl, code);
                        }
                        nh += __popc(m);
                        if (nh >= 32) {
                            __syncwarp();
                            evaluate(32);
                            __syncwarp();
                            if (lane < nh - 32) hits[wib][lane] = hits[wib][32 + lane];
                            __syncwarp();
                            nh -= 32;
                        }
                    }
                }
                __syncwarp();
                if (nh > 0) evaluate(nh);
                __syncwarp();
                warp_force_out(s.fx, s.fy, s.fz, pc.scale, lane, parts == 1 ? Fr + 3 * (int64_t)i : pforce[wib]);
            }
            if (parts > 1) pair_parts_out<kWaterPairWarps>(pforce, u, i, part, parts, wib, lane, Fr);  // the last round
        }
    }
    pair64_partials<false>(s, pc.scale, red, partials + kPartStride * (size_t)blockIdx.x, 1);
}

// ---------------------------------------------------------------------------------
// One thread per molecule: F_i = qqr2e F_k,i + F_r,i plus the intramolecular exclusion
// -qqr2e q_a q_b erf(sqrt(alpha) r)/r of its three site pairs (with real space on); with do_kick,
// R^p/2; the centres' 2K, the exclusion's virial plus the molecular correction -sum_i F_i . d_i,
// and the exclusion energy as block partials {0: 2K, 4: W, 5: E_excl}.  The last block sums the
// partials in a fixed order, forms W_mol = qqr2e tr(W_k) + W_r + W, P_ins = (2K + W_mol)/(3V) and,
// with do_kick, V^p/2 and the step index.  Warp 0 has the molecules' chains, warp 1 + c their exclusions of site
// pair c (3000 molecules: 40 -> 29 us).
__global__ void __launch_bounds__(kWaterThreads * kWaterWarps)
k_water_finish(int64_t Nmol, double* __restrict__ mom, double* __restrict__ force, const double* __restrict__ pos,
               const double* __restrict__ q, const double* __restrict__ mass, const double* __restrict__ Fk,
               const double* __restrict__ Fr, const double* __restrict__ WEk, const NptCoef* __restrict__ cfp,
               double* __restrict__ partials, int nblocks_pair, unsigned* __restrict__ counter,
               double* __restrict__ cell, rbe_npt_params prm, double alpha, int do_kick, unsigned* __restrict__ status)
{
    // of each site pair's exclusion: the force factor, energy and virial
    __shared__ double s_ex[3][3][kWaterThreads];
    __shared__ bool is_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t I = (int64_t)blockIdx.x * kWaterThreads + lane;
    const bool on = I < Nmol;
    double k2 = 0.0, wc = 0.0, ex = 0.0;
    double x[3][3], F[3][3], p[3][3];
    if (on) {
        const double L[3] = {cell[0], cell[1], cell[2]};
        const double inv[3] = {1.0 / L[0], 1.0 / L[1], 1.0 / L[2]};
        w_whole(pos, I, L, inv, x);
    }
    if (on && warp > 0 && prm.real) {
        const double sa = sqrt(alpha), tsp = 2.0 * sqrt(alpha / kPi);
        #pragma unroll
        for (int cp = 0; cp < 3; ++cp) {
            if (cp != warp - 1) continue;
            const int a = wpa(cp), b = wpb(cp);
            double d[3];
            #pragma unroll
            for (int t = 0; t < 3; ++t) d[t] = x[b][t] - x[a][t];
            const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2], r = sqrt(r2);
            const double qq = prm.qqr2e * q[3 * I + a] * q[3 * I + b], ef = erf(sa * r);
            const double f = qq * (tsp * exp(-alpha * r2) / r - ef / r2) / r;
            s_ex[cp][0][lane] = f;
            s_ex[cp][1][lane] = qq * ef / r;
            s_ex[cp][2][lane] = f * r2;
        }
    }
    if (on && warp == 0) {
        #pragma unroll
        for (int k = 0; k < 3; ++k)
            #pragma unroll
            for (int t = 0; t < 3; ++t) {
                const int64_t j = 9 * I + 3 * k + t;
                F[k][t] = (prm.kspace ? prm.qqr2e * Fk[j] : 0.0) + (prm.real ? Fr[j] : 0.0);
                p[k][t] = mom[j];
            }
    }
    __syncthreads();
    if (on && warp == 0) {
        const NptCoef& c = *cfp;
        const double m3[3] = {mass[3 * I], mass[3 * I + 1], mass[3 * I + 2]};
        if (prm.real) {
            #pragma unroll
            for (int cp = 0; cp < 3; ++cp) {
                const int a = wpa(cp), b = wpb(cp);
                const double f = s_ex[cp][0][lane];
                ex -= s_ex[cp][1][lane];
                #pragma unroll
                for (int t = 0; t < 3; ++t) {
                    const double d = x[b][t] - x[a][t];
                    F[b][t] += f * d;
                    F[a][t] -= f * d;
                }
                wc += s_ex[cp][2][lane];
            }
        }
        const double M = m3[0] + m3[1] + m3[2], rM = 1.0 / M;
        double R[3];
        #pragma unroll
        for (int t = 0; t < 3; ++t) R[t] = w_div(m3[0] * x[0][t] + m3[1] * x[1][t] + m3[2] * x[2][t], M, rM);
        #pragma unroll
        for (int k = 0; k < 3; ++k)
            #pragma unroll
            for (int t = 0; t < 3; ++t) {
                wc -= F[k][t] * (x[k][t] - R[t]);
                force[9 * I + 3 * k + t] = F[k][t];
            }
        if (do_kick) {
            const double im[3] = {1.0 / m3[0], 1.0 / m3[1], 1.0 / m3[2]};
            w_kick(p, F, x, m3, im, c.a4[0], c.b4[0], 0.5 * prm.dt);
            #pragma unroll
            for (int k = 0; k < 3; ++k)
                #pragma unroll
                for (int t = 0; t < 3; ++t) mom[9 * I + 3 * k + t] = p[k][t];
        }
        double P[3] = {0.0, 0.0, 0.0};
        #pragma unroll
        for (int k = 0; k < 3; ++k)
            #pragma unroll
            for (int t = 0; t < 3; ++t) P[t] += p[k][t];
        k2 = (P[0] * P[0] + P[1] * P[1] + P[2] * P[2]) / M * (1.0 / kFConv);
    }
    if (warp == 0) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            k2 += __shfl_xor_sync(0xffffffffu, k2, off);
            wc += __shfl_xor_sync(0xffffffffu, wc, off);
            ex += __shfl_xor_sync(0xffffffffu, ex, off);
        }
        if (lane == 0) {
            double* row = partials + kPartStride * (size_t)(nblocks_pair + blockIdx.x);
            row[0] = k2;
            row[4] = wc;
            row[5] = ex;
            __threadfence();
        }
    }
    if (threadIdx.x == 0) is_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // fin: 0 2K, 1 W_r, 2 E_coul, 3 E_lj, 4 W (exclusion + correction), 5 E_excl
    __shared__ double fin[6][kWaterThreads * kWaterWarps];
    {
        double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int b = threadIdx.x; b < (int)gridDim.x; b += kWaterThreads * kWaterWarps) {
            const double* pb = partials + kPartStride * (size_t)(nblocks_pair + b);
            v[0] += __ldcg(pb);
            v[4] += __ldcg(pb + 4);
            v[5] += __ldcg(pb + 5);
        }
        if (prm.real)
            for (int b = threadIdx.x; b < nblocks_pair; b += kWaterThreads * kWaterWarps)
                for (int a = 1; a <= 3; ++a) v[a] += __ldcg(partials + kPartStride * (size_t)b + a);
        for (int a = 0; a < 6; ++a) fin[a][threadIdx.x] = v[a];
    }
    __syncthreads();
    for (int half = kWaterThreads * kWaterWarps / 2; half > 0; half >>= 1) {
        if (threadIdx.x < half)
            for (int a = 0; a < 6; ++a) fin[a][threadIdx.x] += fin[a][threadIdx.x + half];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    double Wk = 0.0, Ek = 0.0;
    if (prm.kspace) {
        Wk = prm.qqr2e * (__ldcg(WEk + 0) + __ldcg(WEk + 4) + __ldcg(WEk + 8));
        Ek = prm.qqr2e * (__ldcg(WEk + 9) + __ldcg(WEk + 10));
    }
    const double K2 = fin[0][0], W = Wk + fin[1][0] + fin[4][0];
    const double V = cell[0] * cell[1] * cell[2];
    const double Pins = (K2 + W) / (3.0 * V);
    double pV = prm.barostat ? cell[3] : 0.0;
    if (do_kick && prm.barostat) pV += 0.5 * prm.dt * (Pins - prm.P_ext);
    cell[3] = pV;
    cell[4] = W;
    cell[5] = K2;
    cell[6] = Pins;
    cell[7] = Ek;
    cell[8] = fin[2][0];
    cell[9] = fin[3][0];
    cell[10] = V;
    cell[kCellExcl] = fin[5][0];
    if (do_kick) cell[kCellStep] = __longlong_as_double((long long)(cell_step(cell) + 1));
    if (!isfinite(Pins) || !isfinite(pV)) atomicOr(status, kStatusNonFinite);
    *counter = 0u;
}

// ---------------------------------------------------------------------------------
// Host side.

static rbe_status water_check(rbe_ctx ctx, const char* what)
{
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? RBE_OK : cuda_fail(ctx, e, what);
}

static rbe_status water_validate(rbe_ctx ctx, const rbe_system* sys, const rbe_water_params* wp)
{
    rbe_status st = npt_validate(ctx, sys);
    if (st != RBE_OK) return st;
    if (!wp) return fail(ctx, RBE_EINVAL, "water parameters are NULL");
    if (sys->N % 3 != 0) return fail(ctx, RBE_EINVAL, "N must count whole molecules (3 sites each)");
    if (sys->params.barostat > 1) return fail(ctx, RBE_EINVAL, "rigid water runs with barostat 0 or 1");
    if (sys->params.skin > 0.0) return fail(ctx, RBE_EINVAL, "rigid water runs without a neighbour list (skin 0)");
    if (!(wp->d_OH > 0.0) || !(wp->d_HH > 0.0) || !std::isfinite(wp->d_OH) || !std::isfinite(wp->d_HH) ||
        !(wp->d_HH < 2.0 * wp->d_OH) || !(wp->shake_tol > 0.0) || !(wp->shake_tol < 1e-3) || wp->shake_max_iter < 1)
        return fail(ctx, RBE_EINVAL, "invalid water parameters");
    return RBE_OK;
}

// Forces, molecular virial and energies at the current state (batch = the device step index; the k-space
// tables have been launched on `fork`), then the finishing kernel.
static rbe_status water_forces(rbe_ctx ctx, rbe_system* sys, const rbe_water_params& wp, KspaceFork& fork, int do_kick)
{
    NptBuffers& b = ctx->npt;
    const rbe_npt_params& prm = sys->params;
    cudaStream_t s = ctx->stream;
    const int64_t N = sys->N, Nmol = N / 3;
    const int nbp = pair_blocks64(ctx, N);
    rbe_status st = fork.passes(sys);
    if (st != RBE_OK) return st;
    if (prm.real) {
        if (b.n64 < N) return fail(ctx, RBE_ESTATE, "the FP64 packed positions are missing: call rbe_water_init again");
        if ((st = launch_cell_list(ctx, N, sys->pos, sys->charge, nullptr, true, pair_unit(prm.rc, 0).s, false)) != RBE_OK)
            return st;
        Pair64Const pc;
        bool built;
        if ((st = pair64_const(ctx, prm, &pc, &built)) != RBE_OK) return st;
        cudaError_t e = smem_opt_in(ctx, kSmemWaterPair, k_water_pair, kPairTabBytes);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "shared memory of k_water_pair");
        e = launch_ordered(!built && ctx->early, k_water_pair, dim3(nbp), dim3(kWaterPairWarps * 32), kPairTabBytes, s, N,
                           static_cast<const CellConsts*>(b.cellc), pc, prm.rc, 5.0 * wp.d_OH, b.cid, b.cnt, b.start,
                           b.sorted, b.spos32, b.spos64, b.Fr, b.partials);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "k_water_pair");
    }
    if ((st = fork.join()) != RBE_OK) return st;
    const int nbm = (int)std::max<int64_t>(1, (Nmol + kWaterThreads - 1) / kWaterThreads);
    k_water_finish<<<nbm, kWaterThreads * kWaterWarps, 0, s>>>(Nmol, sys->mom, sys->force, sys->pos, sys->charge, sys->mass, b.Fk,
                                                 b.Fr, b.WEk, reinterpret_cast<const NptCoef*>(b.coef), b.partials, nbp,
                                                 b.counter, sys->cell, prm, ctx->alpha, do_kick, ctx->d.status);
    return water_check(ctx, "k_water_finish");
}

rbe_status water_init(rbe_ctx ctx, rbe_system* sys, const rbe_water_params* wp, uint64_t batch)
{
    rbe_status st = water_validate(ctx, sys, wp);
    if (st != RBE_OK) return st;
    // the pair kernel reads FP64 packed positions whatever the context's precision
    const int prec = ctx->precision;
    ctx->precision = RBE_FP64;
    st = npt_prepare(ctx, sys, batch);
    ctx->precision = prec;
    if (st != RBE_OK) return st;
    ctx->npt_ready_N = -1;  // the shared scratch now holds a water system
    ctx->flex_ready_N = -1;
    const int64_t Nmol = sys->N / 3;
    // block partials: the pair pass's blocks, then one slot row per finishing block
    NptBuffers& b = ctx->npt;
    const int need = pair_blocks64(ctx, sys->N) + (int)std::max<int64_t>(1, (Nmol + kWaterThreads - 1) / kWaterThreads);
    if (need > b.partcap) {
        ctx_free(ctx, b.partials);
        b.partials = nullptr;
        b.partcap = 0;
        cudaError_t e = ctx_alloc(ctx, &b.partials, sizeof(double) * kPartStride * (size_t)need);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaMalloc(water partials)");
        b.partcap = need;
    }
    k_water_whole<<<(unsigned)((Nmol + kWaterThreads - 1) / kWaterThreads), kWaterThreads, 0, ctx->stream>>>(
        Nmol, sys->pos, sys->cell);
    if ((st = water_check(ctx, "k_water_whole")) != RBE_OK) return st;
    KspaceFork fork(ctx, sys);
    if ((st = fork.tables(sys)) != RBE_OK || (st = water_forces(ctx, sys, *wp, fork, 0)) != RBE_OK) return st;
    ctx->water_ready_N = sys->N;
    return launch_npt_set_step(ctx, sys->cell, sys->step);
}

rbe_status water_run(rbe_ctx ctx, rbe_system* sys, const rbe_water_params* wp, int32_t nsteps)
{
    if (nsteps < 1) return fail(ctx, RBE_EINVAL, "nsteps must be >= 1");
    rbe_status st = water_validate(ctx, sys, wp);
    if (st != RBE_OK) return st;
    if (ctx->water_ready_N != sys->N) return fail(ctx, RBE_ESTATE, "call rbe_water_init for this system first");
    const int64_t Nmol = sys->N / 3;
    const unsigned nbm = (unsigned)((Nmol + kWaterThreads - 1) / kWaterThreads);
    for (int32_t k = 0; k < nsteps; ++k) {
        KspaceFork fork(ctx, sys);
        if ((st = launch_npt_cell_iso(ctx, sys)) != RBE_OK || (st = fork.tables(sys)) != RBE_OK) return st;
        k_water_drift<<<nbm, kWaterThreads * kWaterWarps, 0, ctx->stream>>>(Nmol, sys->pos, sys->mom, sys->force, sys->mass,
                                                              reinterpret_cast<const NptCoef*>(ctx->npt.coef),
                                                              ctx->seed, sys->cell, *wp, sys->params.dt, ctx->d.status);
        if ((st = water_check(ctx, "k_water_drift")) != RBE_OK) return st;
        if ((st = water_forces(ctx, sys, *wp, fork, 1)) != RBE_OK) return st;
        sys->step += 1;
    }
    return RBE_OK;
}

}  // namespace rbe
