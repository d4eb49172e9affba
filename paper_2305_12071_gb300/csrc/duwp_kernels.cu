// duwp_kernels.cu -- the per-step kernels of the DUWP method (arXiv 2305.12071, Sec. 3.4) on sm_103a.
//
//   k_collide     (persistent, one warp per listed cell): NTC/VHS collisions (Appendix A) of the
//                 cells that have candidates, and absorption with probability P (Eq. p) plus
//                 re-sampling of (1-P) of the wave (Eq. maxsample) in the cells where P > 0.
//   k_stream      (one warp per cell): read the cell's stable list (far movers, R(g-1), S(g),
//                 L(g+1), or the staged list), sample the re-sampled particles of cells without
//                 collisions, free transport with boundaries (Step 3), write the L/S/R runs of the
//                 cell's output block, exact sums of the moments that left or entered (Eq. fp).
//   k_stream_block (2, 4 or 8 warps per cell, small pools): the same.
//   k_absorb      (QMC pools, one warp per cell): survivor masks and re-sampled particles of the cells that
//                 absorb, ahead of the collision kernel.
//   k_far_sort    stable order of the rare particles that moved two or more cells.
//   k_cells       (per cell): conservative update Eq. (r1), time average, primitive state, P, the
//                 slot bound and the plan (counts, class) of the next step.
//   k_offsets     (per cell): output block offsets of the next step (scan of the slot bounds), the
//                 work lists of the collision kernels.
//   k_flux        (per interface): the wave flux from the cell kernel's states, at the start of the
//                 step that applies it, beside that step's particle kernels.
#include <algorithm>
#include <type_traits>
#include <cstdio>

#include "duwp_dsmath.cuh"
#include "duwp_launch.h"

namespace duwp {

// cos and sin of 2 pi k / kTurnTable as double-single pairs (scattering and sampling of
// single-precision records), and the log table of the sampling (1/F and log F at F = 1 + (j - kLogCenter)/1024)
__device__ float4 g_turn[kTurnTable];
__device__ float4 g_logt[kLogTable];

__device__ __forceinline__ float2 ds_split(double x)
{
    const float h = __double2float_rn(x);
    return make_float2(h, __double2float_rn(x - static_cast<double>(h)));
}

__global__ void k_init_turn()
{
    const int k = threadIdx.x;
    if (k < kTurnTable) {
        double s, c;
        sincospi(static_cast<double>(k) / (0.5 * kTurnTable), &s, &c);
        const float2 cc = ds_split(c), ss = ds_split(s);
        g_turn[k] = make_float4(cc.x, cc.y, ss.x, ss.y);
    }
    if (k < kLogTable) {
        const double F = static_cast<double>(1024 + k - kLogCenter) * 0x1p-10;
        const float2 inv = ds_split(1.0 / F), lg = ds_split(log(F));
        g_logt[k] = make_float4(inv.x, inv.y, lg.x, lg.y);
    }
}

// Programmatic dependent launch: the step's kernels are launched with programmatic stream
// serialization, so that a kernel's blocks are scheduled while its predecessor's last blocks finish;
// every step kernel first waits here until the predecessor grid has completed and its memory is
// visible (a no-op where the launch had no programmatic dependency).
__device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void set_err(int32_t *err, int code) { atomicCAS(err, 0, code); }

// ------------------------------------------------------------------------------------------
// Record access (FP32 records are one 16-byte vector; FP64 records two).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ RecF ld_rec(const RecF *p)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return RecF{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ RecD ld_rec(const RecD *p)
{
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p));
    const double2 b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    return RecD{a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void st_rec(RecF *p, const RecF &r)
{
    *reinterpret_cast<float4 *>(p) = make_float4(r.xl, r.u, r.v, r.w);
}
__device__ __forceinline__ void st_rec(RecD *p, const RecD &r)
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(r.xl, r.u);
    reinterpret_cast<double2 *>(p)[1] = make_double2(r.v, r.w);
}

// Storage rounding of a value computed in FP64.
__device__ __forceinline__ float store_val(double x, float) { return __double2float_rn(x); }
__device__ __forceinline__ double store_val(double x, double) { return x; }

// ------------------------------------------------------------------------------------------
// Free transport in cell units with the boundary conditions (Step 3).  The position update
// x + xi dt/dx is one fused multiply-add in the record precision; the new cell is its floor.
// Returns the new local cell or -1 (the particle left the domain).
// ------------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ int64_t apply_walls(const InstDev &I, int64_t dest, T &x, T &u, bool &refl)
{
    const int64_t C = I.C;
    for (int it = 0; it < 64; ++it) {
        if ((dest < 0 && I.bc_left == kBcPhantom) || (dest >= C && I.bc_right == kBcPhantom))
            return dest;     // into another part of the domain (phantom side): kept, exported
        if (dest < 0) {
            if (I.bc_left == 1) {
                dest = -dest - 1;
                x = T(1) - x;
                if (x >= T(1)) { x = T(0); dest += 1; }
                u = -u;
                refl = !refl;
                continue;
            }
            if (I.bc_left == 2) { dest = ((dest % C) + C) % C; continue; }
            return kGone;
        }
        if (dest >= C) {
            if (I.bc_right == 1) {
                dest = 2 * C - dest - 1;
                x = T(1) - x;
                if (x >= T(1)) { x = T(0); dest += 1; }
                u = -u;
                refl = !refl;
                continue;
            }
            if (I.bc_right == 2) { dest = dest % C; continue; }
            return kGone;
        }
        return dest;
    }
    return kGone;   // more than 64 wall reflections within one step: removed
}

__device__ __forceinline__ int64_t transport(const InstDev &I, int64_t cell, double &xl, double &u, bool &refl)
{
    const double s = __fma_rn(u, I.dtdx, xl);
    if (!(fabs(s) < 1e15)) return kGone;
    const double fk = floor(s);
    double x = __dsub_rn(s, fk);
    int64_t k = static_cast<int64_t>(fk);
    if (x >= 1.0) { x = 0.0; k += 1; }
    xl = x;
    return apply_walls<double>(I, cell + k, xl, u, refl);
}

// ------------------------------------------------------------------------------------------
// Maxwellian sample at the primitive state q (Eq. maxsample) by Box-Muller pairs: radius
// sqrt(2RT) sqrt(-ln r2), r2 in (0,1], angle 2 pi r1 -> x (cosine) and y (sine); z from its own pair
// (r3, r4) and its cosine; position uniform in the cell.  Particle j of a cell uses counters
// (id, 4j..4j+2, step, SAMPLE): uniforms 0 -> position, 1 -> r1, 2 -> r2, 3 -> r3, 4 -> r4.
// ------------------------------------------------------------------------------------------
// Per-cell part of the sample: the state and sqrt(2RT), also as double-single values.
struct MaxwellCell {
    double q[5];
    double sq;
    ds U[3];
    ds s;
    const double *qp;       // the cell's primitive state (rho, U, V, W, T) in device memory
};

// Chapman-Enskog factor of a cell's samples under the NS-corrected option (below).
struct CeCell {
    double A, sxx, syy, sxy, sxz, qx, prt, RT;
};

__device__ inline MaxwellCell maxwell_cell(const InstDev &I, const double *q)
{
    MaxwellCell m;
    m.qp = q;
    for (int k = 0; k < 5; ++k) m.q[k] = q[k];
    m.sq = sqrt(2.0 * I.R * q[4]);
    for (int d = 0; d < 3; ++d) {
        const float h = __double2float_rn(q[1 + d]);
        m.U[d] = {h, __double2float_rn(q[1 + d] - static_cast<double>(h))};
    }
    const float h = __double2float_rn(m.sq);
    m.s = {h, __double2float_rn(m.sq - static_cast<double>(h))};
    return m;
}

// The sampling state of a cell for single-precision records drawn without the NS correction: only
// the double-single U and s, formed by integer and single-precision operations (the double-precision
// units are few on this GPU and a chunk of draws is short); q and sq are not set, and a draw that
// takes the double-precision path reads the state from qp.  Double-precision records (and values
// outside the integer conversion's range) take the full state.
template <typename Rec>
__device__ inline MaxwellCell maxwell_cell_for(const InstDev &I, const double *q)
{
    if constexpr (sizeof(Rec) == sizeof(RecF)) {
        MaxwellCell m;
        m.qp = q;
        if (ds_maxwell_params(I.R, q, m.U, m.s)) return m;
    }
    return maxwell_cell(I, q);
}

// Velocities in double precision from the 8 draw words after the position's (w), by the Box-Muller
// transform: the angle 2 pi r1 and the radius sqrt(2RT) sqrt(-ln r2) give the x component (cosine)
// and the y component (sine); z takes its own angle r3 and radius r4 (cosine).
__device__ __forceinline__ void maxwell_xi(const MaxwellCell &mc, const uint32_t *w, double out[3])
{
    const double r1 = u53(w[0], w[1]);
    const double r2 = 1.0 - u53(w[2], w[3]);
    const double r3 = u53(w[4], w[5]);
    const double r4 = 1.0 - u53(w[6], w[7]);
    const double rad = sqrt(-log(r2));
    out[0] = mc.q[1] + (mc.sq * cos(kTwoPi * r1)) * rad;
    out[1] = mc.q[2] + (mc.sq * sin(kTwoPi * r1)) * rad;
    out[2] = mc.q[3] + (mc.sq * cos(kTwoPi * r3)) * sqrt(-log(r4));
}

template <typename T>
__device__ __noinline__ void maxwell_fp64(const MaxwellCell &mc, const uint32_t *w, T out[3])
{
    double xi[3];
    maxwell_xi(mc, w, xi);
#pragma unroll
    for (int d = 0; d < 3; ++d) out[d] = store_val(xi[d], T());
}

// The same double-precision evaluation for a single-precision record from the cell's state in memory
// (words w[2..9] of the draw by value, so that the caller keeps them in registers); returns the
// record's velocities in y, z, w.
__device__ __noinline__ float4 maxwell_fp64_from(double R, const double *q, uint4 wa, uint4 wb)
{
    const double sq = sqrt(2.0 * R * q[4]);
    const double r1 = u53(wa.x, wa.y);
    const double r2 = 1.0 - u53(wa.z, wa.w);
    const double r3 = u53(wb.x, wb.y);
    const double r4 = 1.0 - u53(wb.z, wb.w);
    const double rad = sqrt(-log(r2));
    return make_float4(0.0f, __double2float_rn(q[1] + (sq * cos(kTwoPi * r1)) * rad),
                       __double2float_rn(q[2] + (sq * sin(kTwoPi * r1)) * rad),
                       __double2float_rn(q[3] + (sq * cos(kTwoPi * r3)) * sqrt(-log(r4))));
}

// NS-corrected sampling (resample_mode CE; the first-order Chapman-Enskog form of the equilibrium,
// Eq. ce2): the density f_M (1 + sigma_ij c_i c_j / (2 p R T) + (q . c / (p R T)) (c^2 / (5 R T) - 1)),
// c = xi - U, with the 1D NS stress and heat flux of the wave at the viscosity eps mu of its flux
// (Eq. vp1, Sec. 3.3):
//   sigma_xx = -(4/3) mu_e dU/dx, sigma_yy = sigma_zz = (2/3) mu_e dU/dx, sigma_xy = -mu_e dV/dx,
//   sigma_xz = -mu_e dW/dx, q_x = -kappa_e dT/dx, kappa_e = (5/2) R mu_e / Pr,
// the gradients by central differences of the neighbouring states (the periodic partner or the
// reservoir/mirror state beyond an end; an unusable neighbour counts as the cell's own state).
// Drawn by acceptance-rejection against A = 1 + 30 B, B the largest of |sigma_ij| / p and
// 2 |q_x| / (p sqrt(2RT)) (Garcia and Alder, J. Comput. Phys. 140, 1998); for B > 1/4 the expansion
// is out of range and the plain Maxwellian is drawn.  Every expression keeps the order of
// operations of the double-precision checker, so decisions agree to the last bit of the inputs.
constexpr int kCeAttempts = 64;

// Returns false where the plain Maxwellian is drawn.
__device__ __noinline__ bool ce_coefs(const InstDev &I, const double *prim, const int32_t *valid, int g, int i,
                                      CeCell &m)
{
    if (!valid[g]) return false;
    const double *W0 = prim + 5 * g;
    double wm[5], wp[5];
    bool okm, okp;
    const bool periodic = (I.bc_left == 2);
    if (i > 0 || I.bc_left == kBcPhantom) { for (int k = 0; k < 5; ++k) wm[k] = W0[k - 5]; okm = valid[g - 1] != 0; }
    else if (periodic) { for (int k = 0; k < 5; ++k) wm[k] = prim[5 * (g + I.C - 1) + k]; okm = valid[g + I.C - 1] != 0; }
    else okm = ghost_prim(I, 0, W0, true, wm);
    if (i < I.C - 1 || I.bc_right == kBcPhantom) { for (int k = 0; k < 5; ++k) wp[k] = W0[k + 5]; okp = valid[g + 1] != 0; }
    else if (periodic) { for (int k = 0; k < 5; ++k) wp[k] = prim[5 * (g - I.C + 1) + k]; okp = valid[g - I.C + 1] != 0; }
    else okp = ghost_prim(I, 1, W0, true, wp);
    const double *a = okm ? wm : W0, *b = okp ? wp : W0;
    const double inv = 1.0 / (2.0 * I.dx);
    const double dU = (b[1] - a[1]) * inv, dV = (b[2] - a[2]) * inv, dW = (b[3] - a[3]) * inv;
    const double dT = (b[4] - a[4]) * inv;
    const double RT = I.R * W0[4];
    const double p0 = W0[0] * RT;
    const double mu = viscosity(I, W0[4]);
    const double mue = eps_factor(I.eps_mode, I.dt / (mu / p0)) * mu;
    const double kap = 2.5 * I.R * mue / I.Pr;
    m.sxx = -(4.0 / 3.0) * mue * dU;
    m.syy = (2.0 / 3.0) * mue * dU;
    m.sxy = -mue * dV;
    m.sxz = -mue * dW;
    m.qx = -kap * dT;
    double B = fmax(fmax(fabs(m.sxx), fabs(m.syy)), fmax(fabs(m.sxy), fabs(m.sxz))) / p0;
    B = fmax(B, 2.0 * fabs(m.qx) / (p0 * sqrt(2.0 * RT)));
    if (!(B <= 0.25)) return false;
    m.RT = RT;
    m.prt = p0 * RT;
    m.A = 1.0 + 30.0 * B;
    return true;
}

__device__ __forceinline__ double ce_gamma(const MaxwellCell &mc, const CeCell &m, const double xi[3])
{
    const double cx = xi[0] - mc.q[1], cy = xi[1] - mc.q[2], cz = xi[2] - mc.q[3];
    const double c2 = cx * cx + cy * cy + cz * cz;
    const double s = m.sxx * cx * cx + m.syy * (cy * cy + cz * cz) + 2.0 * (m.sxy * cx * cy + m.sxz * cx * cz);
    return 1.0 + s / (2.0 * m.prt) + (m.qx * cx / m.prt) * (c2 / (5.0 * m.RT) - 1.0);
}

// Velocities of an NS-corrected sample: attempt 0 uses the sample's own words w0 (velocities from
// w0[2..9], acceptance from w0[10..11]); attempt a > 0 draws the counters (id, 4j..4j+2, step,
// SAMPLE + 8a).  After kCeAttempts rejections the attempt-0 Maxwellian is kept.
__device__ __noinline__ void ce_xi(const InstDev &I, uint32_t id, uint32_t j, uint32_t step, const MaxwellCell &mc,
                                   const CeCell &ce, const uint32_t *w0, double xi[3])
{
    maxwell_xi(mc, w0 + 2, xi);
    if (u53(w0[10], w0[11]) * ce.A < ce_gamma(mc, ce, xi)) return;
    uint32_t w[12];
    double t[3];
    for (int a = 1; a < kCeAttempts; ++a) {
#pragma unroll
        for (uint32_t k = 0; k < 3; ++k) draw(I, id, 4u * j + k, step, kSample + 8u * static_cast<uint32_t>(a), w + 4 * k);
        maxwell_xi(mc, w + 2, t);
        if (u53(w[10], w[11]) * ce.A < ce_gamma(mc, ce, t)) {
            xi[0] = t[0]; xi[1] = t[1]; xi[2] = t[2];
            return;
        }
    }
}

// Single-precision rounding of the 53-bit uniform u53(a, b) (exact integer conversion, then a power
// of two): the same value as rounding the double u53(a, b).
__device__ __forceinline__ float u53_float(uint32_t a, uint32_t b)
{
    const unsigned long long m = (static_cast<unsigned long long>(a) << 21) | static_cast<unsigned long long>(b >> 11);
    return __ull2float_rn(m) * 0x1p-53f;
}

template <typename Rec, bool kRolled = true>
__device__ __forceinline__ Rec sample_particle(const InstDev &I, uint32_t id, uint32_t j, uint32_t step, const MaxwellCell &mc,
                                           const CeCell *ce)
{
    uint32_t w[12];
#pragma unroll
    for (uint32_t t = 0; t < 3; ++t) draw(I, id, 4u * j + t, step, kSample, w + 4 * t);
    Rec r;
    using T = decltype(r.xl);
    T x, xi[3];
    if (ce) {
        // NS-corrected option: the acceptance test needs the double-precision velocities
        x = (sizeof(T) == 4) ? static_cast<T>(u53_float(w[0], w[1])) : static_cast<T>(u53(w[0], w[1]));
        double xd[3];
        ce_xi(I, id, j, step, mc, *ce, w, xd);
#pragma unroll
        for (int d = 0; d < 3; ++d) xi[d] = store_val(xd[d], T());
    } else if constexpr (sizeof(T) == 4) {
        // single-precision records: double-single evaluation, double precision only where the
        // rounding of a component cannot be guaranteed
        x = u53_float(w[0], w[1]);
        if (!ds_maxwell<kRolled>(g_turn, g_logt, mc.U, mc.s, w + 2, xi)) {
            const float4 f = maxwell_fp64_from(I.R, mc.qp, make_uint4(w[2], w[3], w[4], w[5]),
                                               make_uint4(w[6], w[7], w[8], w[9]));
            xi[0] = f.y;
            xi[1] = f.z;
            xi[2] = f.w;
        }
    } else {
        x = u53(w[0], w[1]);
        maxwell_fp64<T>(mc, w + 2, xi);
    }
    if (x >= T(1)) x = sizeof(T) == 4 ? T(0x1.fffffep-1f) : x;
    r.xl = x;
    r.u = xi[0];
    r.v = xi[1];
    r.w = xi[2];
    return r;
}

// Samples j0..j1-1 of interior cell g (local index i) under the NS-corrected option, one per lane,
// into dst[j]: the per-cell factor once, then the samples (Maxwellian where the factor is off).
template <typename Rec>
__device__ __noinline__ void sample_run_ce(const InstDev &I, const double *prim, const int32_t *valid, int g, int i,
                                           uint32_t step, Rec *dst, int j0, int j1, int lane)
{
    const MaxwellCell mc = maxwell_cell(I, prim + 5 * g);
    CeCell ce;
    const bool on = ce_coefs(I, prim, valid, g, i, ce);
    for (int j = j0 + lane; j < j1; j += 32)
        st_rec(dst + j, sample_particle<Rec>(I, cell_id(I, i), static_cast<uint32_t>(j), step, mc, on ? &ce : nullptr));
}

// Lower bound of `key` in the far list ordered by (dest, src, q): first index with (dest, src) >= key.
template <typename Rec>
__device__ int far_lower(const FarItem<Rec> *f, int n, int dest, int src)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const bool less = (f[mid].dest < dest) || (f[mid].dest == dest && f[mid].src < src);
        if (less) lo = mid + 1; else hi = mid;
    }
    return lo;
}


// Majorant factor (c_max/c_ref)^{-2 upsilon} of the NTC count; kept per cell and recomputed only when
// c_max is raised.
__device__ __noinline__ double majorant_factor(const InstDev &I, double cmax)   // rare: when c_max rises
{
    return (I.upsilon == 0.0) ? 1.0 : pow(cmax / I.c_ref, -2.0 * I.upsilon);
}

// NTC candidate count of a cell with N particles (Appendix A, nondimensional form), rounded with the
// cell's ROUND draw 1; -1 when the count is absurd (over 1e8).  The density ratio uses the
// precomputed m_p/(dx rho_ref) and the majorant factor comes from the per-cell cache, so the product
// may differ from the plain left-to-right evaluation by a few ulps; the rounded count differs only
// when N_sel + u lies within those ulps of an integer.
__device__ inline int64_t ntc_candidates(const InstDev &I, int N, double rho_t, double cmax, double fmaj, double u)
{
    if (N < 2) return 0;
    // N and N - 1 converted by integer operations (exact)
    const double rr = (I.ntc_rate == 1) ? rho_t * I.inv_rho_ref : fixed_to_double(N, 0) * I.ntc_rr;
    const double nsel = I.ntc_A * rr * fixed_to_double(N - 1, 0) * fmaj * cmax;
    if (!dbl_lt(nsel, 1e8)) return -1;
    const double y = nsel + u;
    return dbl_bits(y) >= 0 ? floor_pos(y) : static_cast<int64_t>(floor(y));
}

__device__ inline int64_t ntc_candidates(const InstDev &I, uint32_t id, uint32_t step, int N, double rho_t, double cmax,
                                         double fmaj)
{
    if (N < 2) return 0;
    return ntc_candidates(I, N, rho_t, cmax, fmaj, round_draw(I, id, 1u, step));
}

// The relative speed of a pair: c_r^2 in single precision (relative error below 4e-7), and what the exact
// c_r = sqrt(c_r^2) is formed from (double-precision records: c_r^2 itself).
struct RelF {
    float q;
};
struct RelD {
    float q;
    double qd;
};
__device__ __forceinline__ RelF rel_of(const RecF &A, const RecF &B)
{
    const float d0 = A.u - B.u, d1 = A.v - B.v, d2 = A.w - B.w;
    return {fmaf(d2, d2, fmaf(d1, d1, d0 * d0))};
}
__device__ __forceinline__ RelD rel_of(const RecD &A, const RecD &B)
{
    const double d0 = A.u - B.u, d1 = A.v - B.v, d2 = A.w - B.w;
    const double q = d0 * d0 + d1 * d1 + d2 * d2;
    return {f32_of_double(q), q};
}
__device__ __forceinline__ double rel_exact(RelF, const RecF &A, const RecF &B)
{
    const double d0 = static_cast<double>(A.u) - static_cast<double>(B.u);
    const double d1 = static_cast<double>(A.v) - static_cast<double>(B.v);
    const double d2 = static_cast<double>(A.w) - static_cast<double>(B.w);
    return sqrt(d0 * d0 + d1 * d1 + d2 * d2);
}
__device__ __forceinline__ double rel_exact(RelD r, const RecD &, const RecD &) { return sqrt(r.qd); }

// ------------------------------------------------------------------------------------------
// NTC collisions (Appendix A).  A candidate's pair, the bounds of its acceptance test and its scattering
// angles depend only on counters, so they are formed ahead for all candidates of a batch at once; what
// is left for the dependent part (a particle must see its collisions in candidate order) is the
// comparison of c_r^2 with the bounds and the scattering of the accepted pairs.
// ------------------------------------------------------------------------------------------

// The acceptance test turned around: u < (c_r/c_max)^e is (c_r/c_max)^2 > u^(2/e), so a candidate's draw
// gives, before its collision partners' velocities are known, bounds lo < u^(2/e) < hi; then
// c_r^2 > hi c_max^2 accepts and c_r^2 < lo c_max^2 rejects (both outside the single-precision error of
// c_r^2, 4e-7, and far from underflow), and the rest, about 1e-5 of the candidates, is decided in
// double precision.  u is known to 2^-32 from its first word: its logarithm has an error below
// 1.443 (2^-32/u + 2^-23) + 2^-22 max(1, |log2 u|) (the approximation instruction's), times 2/e in the
// exponent; the margin is twice the resulting relative error.  e = 0 (Maxwell molecules): lo = hi = 0.
__device__ __forceinline__ float2 accept_bounds(uint32_t w2, float inv_expo)
{
    const float u = __uint2float_rn(w2) * 0x1p-32f;
    if (!(inv_expo < 1e30f)) return make_float2(0.0f, 0.0f);
    if (w2 < 4096u) return make_float2(0.0f, 3e38f);
    float l, p;
    asm("lg2.approx.f32 %0, %1;" : "=f"(l) : "f"(u));
    asm("ex2.approx.f32 %0, %1;" : "=f"(p) : "f"(2.0f * inv_expo * l));
    const float el = 1.443f * (__fdividef(0x1p-32f, u) + 0x1p-23f) + 0x1p-22f * fmaxf(1.0f, -l);
    // relative error of p: ln 2 times that of the exponent (its rounding included), of the exponential,
    // and of c_r^2 and c_max^2
    const float e = 2.0f * (1.4f * inv_expo * (el + 0x1p-21f * -l) + 2e-6f);
    if (!(e < 0.25f)) return make_float2(0.0f, 3e38f);
    return make_float2(p * (1.0f - e), p * (1.0f + e));
}
// The rest of the acceptance tests, in double precision: out of line, as it is rare.
__device__ __noinline__ bool accept_exact(const InstDev &I, uint32_t id, uint32_t k, uint32_t step, double cr, double cm)
{
    uint32_t w[4];
    draw(I, id, 2u * k, step, kCollide, w);
    const double x = cr / cm;
    return u53(w[2], w[3]) < (dbl_is_zero(I.upsilon) ? x : pow(x, I.vhs_expo));
}

// c_max^2 as the tests take it, and the square above which c_r may exceed c_max.
struct Majorant {
    double cm;
    float cm2, near;
};
__device__ __forceinline__ Majorant majorant(double cm)
{
    const float c = f32_of_double(cm);
    return {cm, c * c, c * c * 0.99999f};
}

// Whether candidate k (records A, B; bounds bd) is accepted, and whether it raises c_max (its exact c_r
// exceeds it: Appendix A raises c_max before the test, so it is accepted).  cr / exact: the exact
// relative speed when it was needed.
template <typename Rec, typename Rel>
__device__ __forceinline__ bool accept_pair(const InstDev &I, uint32_t id, uint32_t k, uint32_t step, const Rec &A,
                                            const Rec &B, Rel rel, float2 bd, const Majorant &M, double &cr, bool &exact,
                                            bool &raises)
{
    const float lo = bd.x * M.cm2, hi = bd.y * M.cm2;
    bool a = rel.q > hi && rel.q > 1e-30f;
    const bool rejected = rel.q < lo && lo > 1e-30f;
    raises = false;
    exact = false;
    if (rel.q > M.near || !(a || rejected)) {
        cr = rel_exact(rel, A, B);
        exact = true;
        if (dbl_bits(cr) > dbl_bits(M.cm)) {       // (both positive)
            raises = true;
            a = true;
        } else if (!a) {
            a = accept_exact(I, id, k, step, cr, M.cm);
        }
    }
    return a;
}

// Isotropic VHS scattering of an accepted pair (Appendix A) in double precision: the relative
// velocity keeps its magnitude c_r and takes the direction (theta, phi) with cos(theta) = 2 u1 - 1,
// phi = 2 pi u2 (u1 = u53(v0, v1), u2 = u53(v2, v3)).  Out of line, records by value.
template <typename Rec>
struct RecPair {
    Rec a, b;
};
template <typename Rec>
__device__ __noinline__ RecPair<Rec> scatter_fp64(uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3, Rec A, Rec B,
                                                  double cr)
{
    using T = decltype(A.xl);
    const double ct = 2.0 * u53(v0, v1) - 1.0;
    const double st = sqrt(1.0 - ct * ct);
    double sp, cp;
    sincos(kTwoPi * u53(v2, v3), &sp, &cp);
    const double c0 = (cr * st) * cp, c1 = (cr * st) * sp, c2 = cr * ct;
    const double au = A.u, av = A.v, aw = A.w, bu = B.u, bv = B.v, bw = B.w;
    const double m0 = (au + bu) * 0.5, m1 = (av + bv) * 0.5, m2 = (aw + bw) * 0.5;
    A.u = store_val(m0 + c0 * 0.5, T());
    A.v = store_val(m1 + c1 * 0.5, T());
    A.w = store_val(m2 + c2 * 0.5, T());
    B.u = store_val(m0 - c0 * 0.5, T());
    B.v = store_val(m1 - c1 * 0.5, T());
    B.w = store_val(m2 - c2 * 0.5, T());
    return RecPair<Rec>{A, B};
}

// x / 2 (exact), without the double-precision unit but for zeros, subnormals, infinities and NaN.
__device__ __forceinline__ double dbl_half(double x)
{
    const unsigned e = (static_cast<unsigned>(__double2hiint(x)) >> 20) & 0x7ffu;
    if (e - 2u < 0x7fdu) return __hiloint2double(__double2hiint(x) - 0x100000, __double2loint(x));
    return 0.5 * x;
}

// The scattering angles of candidate k, 32 bytes: cos(theta), sin(theta), cos(phi), sin(phi) as double-single
// pairs (single-precision records; returns whether they are usable) or doubles (the operations of
// scatter_fp64).
__device__ __forceinline__ bool pair_angles(const RecF *, const InstDev &I, uint32_t id, uint32_t k, uint32_t step,
                                            float4 *out)
{
    uint32_t w[4];
    draw(I, id, 2u * k + 1u, step, kCollide, w);
    DsAngles g;
    const bool ok = ds_scatter_angles(g_turn, w[0], w[1], w[2], w[3], g);
    out[0] = make_float4(g.ct.hi, g.ct.lo, g.st.hi, g.st.lo);
    out[1] = make_float4(g.cp.hi, g.cp.lo, g.sp.hi, g.sp.lo);
    return ok;
}
__device__ __forceinline__ bool pair_angles(const RecD *, const InstDev &I, uint32_t id, uint32_t k, uint32_t step,
                                            float4 *out)
{
    uint32_t w[4];
    draw(I, id, 2u * k + 1u, step, kCollide, w);
    // cos(theta) = 2 u1 - 1 (exact)
    const uint64_t m = (static_cast<uint64_t>(w[0]) << 21) | static_cast<uint64_t>(w[1] >> 11);
    const double ct = fixed_to_double(static_cast<int64_t>(m) - (1ll << 52), 52);
    double sp, cp;
    sincos(kTwoPi * u53(w[2], w[3]), &sp, &cp);
    double2 *o = reinterpret_cast<double2 *>(out);
    o[0] = make_double2(ct, sqrt(1.0 - ct * ct));
    o[1] = make_double2(cp, sp);
    return true;
}

// The accepted pair A, B of candidate k scattered with its angles.  cr / exact: the double-precision
// relative speed when the caller already has it.  Single-precision records are scattered in
// double-single arithmetic, which yields the single-precision rounding of the same values as the
// double-precision evaluation; the few pairs where that cannot be guaranteed take the
// double-precision path.
__device__ __forceinline__ void scatter_pair(const InstDev &I, uint32_t id, uint32_t k, uint32_t step, RecF &A, RecF &B,
                                             RelF rel, const float4 *ang, bool angok, double cr, bool exact)
{
    const float4 g0 = ang[0], g1 = ang[1];
    const DsAngles g{{g0.x, g0.y}, {g0.z, g0.w}, {g1.x, g1.y}, {g1.z, g1.w}};
    float o[6];
    if (ds_scatter_apply(A.u, A.v, A.w, B.u, B.v, B.w, g, o) && angok) {
        A.u = o[0]; A.v = o[1]; A.w = o[2];
        B.u = o[3]; B.v = o[4]; B.w = o[5];
    } else {
        uint32_t v[4];
        draw(I, id, 2u * k + 1u, step, kCollide, v);
        const RecPair<RecF> r = scatter_fp64<RecF>(v[0], v[1], v[2], v[3], A, B, exact ? cr : rel_exact(rel, A, B));
        A = r.a;
        B = r.b;
    }
}
__device__ __forceinline__ void scatter_pair(const InstDev &, uint32_t, uint32_t, uint32_t, RecD &A, RecD &B, RelD rel,
                                             const float4 *ang, bool, double cr, bool exact)
{
    const double2 *o = reinterpret_cast<const double2 *>(ang);
    const double2 th = o[0], ph = o[1];
    if (!exact) cr = rel_exact(rel, A, B);
    const double cs = cr * th.y;
    const double c[3] = {dbl_half(cs * ph.x), dbl_half(cs * ph.y), dbl_half(cr * th.x)};
    const double m[3] = {dbl_half(A.u + B.u), dbl_half(A.v + B.v), dbl_half(A.w + B.w)};
    A.u = m[0] + c[0]; A.v = m[1] + c[1]; A.w = m[2] + c[2];
    B.u = m[0] - c[0]; B.v = m[1] - c[1]; B.w = m[2] - c[2];
}

// The same out of line for the collision kernel's warps, whose 64 registers do not hold a candidate's state
// beside the scattering's (records by value: one whose address reached a call would live in local
// memory on every path), with the draw and the angles formed here, for the accepted pairs only: single-
// precision records whose batches seldom need many rounds (forming and keeping the angles of every
// candidate of a batch, as double-precision records and the block kernel do, took 2% more of a shock
// batch's step).
__device__ __noinline__ RecPair<RecF> scatter_warp_drawn(const InstDev &I, uint32_t id, uint32_t k, uint32_t step, RecF A,
                                                         RecF B)
{
    float4 ang[2];
    const bool angok = pair_angles(&A, I, id, k, step, ang);
    scatter_pair(I, id, k, step, A, B, rel_of(A, B), ang, angok, 0.0, false);
    return RecPair<RecF>{A, B};
}

// A cell's particle list as collide_list sees it: position x -> record address.
template <typename Rec>
struct StagedList {
    Rec *p;
    __device__ __forceinline__ Rec *at(int x) const { return p + x; }
};

constexpr int kSelect = 64;            // entries of a masked list's survivor index
constexpr int kHash = 128;             // slots of a warp's touched-particle table (at most 2 x kMaxDirect keys)

// Slot of list position x in the slots [base, base + size) of the touched-particle table (inserted
// if absent; `fresh`: by this call).  At most size/2 keys share those slots, so a free slot or the
// key itself is always found within the probe limit.
__device__ __forceinline__ int seg_insert(int *key, int base, int size, int x, bool &fresh, int32_t *err)
{
    int h = base + static_cast<int>(__umulhi(static_cast<uint32_t>(x) * 2654435761u, static_cast<uint32_t>(size)));
    for (int it = 0; it < size; ++it) {
        const int old = atomicCAS(&key[h], -1, x);
        if (old == -1 || old == x) {
            fresh = (old == -1);
            return h;
        }
        h = (h + 1 == base + size) ? base : h + 1;
    }
    set_err(err, kErrOverflow);
    fresh = false;
    return base;
}

template <typename Rec>
struct CollideShared {
    int key[kHash];     // list position of the particle held in the slot, -1 = empty
    int own[kHash];     // lowest candidate of the current batch that touches the slot (32 = none)
    int mod[kHash];     // changed by an accepted collision
    Rec rec[kHash];
    int pre[kSelect];   // masked lists: survivors before every (stride)-th word of the mask
    float4 ang[sizeof(Rec) == sizeof(RecD) ? 32 : 1][2];  // FP64 records: scattering angles of each lane's candidate
};

// The warp's tables (by their own address, not passed on, so that they are addressed as shared memory in
// functions that are not inlined).
template <typename Rec>
__device__ __forceinline__ CollideShared<Rec> &collide_shared()
{
    extern __shared__ __align__(16) unsigned char smraw[];
    return reinterpret_cast<CollideShared<Rec> *>(smraw)[threadIdx.x >> 5];
}

// The nc NTC candidates of a cell's list of N records in candidate order (one warp): batches of up to 32,
// candidate k0 + lane on its lane, its pair and acceptance bounds (double-precision records: its angles
// too) formed for the whole batch at once.  The batch's particles are held in a shared-memory table (a hash of their list positions:
// key; the lowest remaining candidate touching each: own) and the candidates run in dependency rounds:
// a candidate runs once it is the lowest remaining candidate of the batch on both of its particles, so
// every particle sees its collisions in candidate order -- the sequential order of the NTC loop -- while
// independent candidates run together.  The changed records are written back after the batch.  Every
// candidate of a batch tests against the batch's c_max; where one raises it (Appendix A: c_max is raised to
// the pair's c_r before its test), the table is reloaded from memory and the batch rerun up to that
// candidate, and the next batch starts after it with the raised c_max.
template <typename Rec, typename List>
__device__ __noinline__ void collide_list(const InstDev &I, uint32_t id, uint32_t step, List list, int N, int64_t nc,
                                          double &cmax, int &nacc, int32_t *err)
{
    CollideShared<Rec> &S = collide_shared<Rec>();
    const int lane = threadIdx.x & 31;
    nacc = 0;
    if (N < 2 || nc <= 0) return;
    const float inv_expo = __fdividef(1.0f, I.vhs_expo_f);
    int acc = 0;
    Majorant M = majorant(cmax);
    for (int t = lane; t < kHash; t += 32) {
        S.key[t] = -1;
        S.own[t] = 32;
        S.mod[t] = 0;
    }
    __syncwarp();
    for (int64_t k0 = 0; k0 < nc;) {
        const int nb = static_cast<int>(min(static_cast<int64_t>(32), nc - k0));
        const uint32_t k = static_cast<uint32_t>(k0 + lane);
        const bool act = lane < nb;
        int a = 0, b = 0, ha = 0, hb = 0;
        bool fa = false, fb = false;
        float2 bd = make_float2(0.0f, 0.0f);
        if (act) {
            uint32_t w[4];
            draw(I, id, 2u * k, step, kCollide, w);
            a = static_cast<int>(idx32(w[0], static_cast<uint32_t>(N)));
            b = static_cast<int>(idx32(w[1], static_cast<uint32_t>(N - 1)));
            if (b >= a) ++b;
            ha = seg_insert(S.key, 0, kHash, a, fa, err);
            hb = seg_insert(S.key, 0, kHash, b, fb, err);
            if (fa) S.rec[ha] = ld_rec_rw(list.at(a));
            if (fb) S.rec[hb] = ld_rec_rw(list.at(b));
            bd = accept_bounds(w[2], inv_expo);
            if constexpr (sizeof(Rec) == sizeof(RecD)) pair_angles(S.rec, I, id, k, step, S.ang[lane]);
        }
        __syncwarp();
        // the rounds of candidates [0, limit) of the batch on the table; returns the accepted ones and
        // the lowest candidate that raised c_max (32: none) with its c_r
        int na = 0, rmin = 32;
        double cr_r = 0.0;
        for (int limit = nb;;) {
            bool undone = lane < limit;
            na = 0;
            rmin = 32;
            while (__any_sync(0xffffffffu, undone)) {
                if (undone) {
                    atomicMin(&S.own[ha], lane);
                    atomicMin(&S.own[hb], lane);
                }
                __syncwarp();
                const bool run = undone && S.own[ha] == lane && S.own[hb] == lane;
                __syncwarp();
                if (undone) {
                    S.own[ha] = 32;
                    S.own[hb] = 32;
                }
                bool accd = false, raises = false, exact = false;
                double cr = 0.0;
                if (run) {
                    Rec A = S.rec[ha], B = S.rec[hb];
                    const auto rel = rel_of(A, B);
                    accd = accept_pair(I, id, k, step, A, B, rel, bd, M, cr, exact, raises);
                    if (accd) {
                        if constexpr (sizeof(A.u) == 4) {
                            const RecPair<Rec> r = scatter_warp_drawn(I, id, k, step, A, B);
                            S.rec[ha] = r.a;
                            S.rec[hb] = r.b;
                        } else {
                            scatter_pair(I, id, k, step, A, B, rel, S.ang[lane], true, cr, exact);
                            S.rec[ha] = A;
                            S.rec[hb] = B;
                        }
                        S.mod[ha] = 1;
                        S.mod[hb] = 1;
                    }
                    undone = false;
                }
                const unsigned rm = __ballot_sync(0xffffffffu, raises);
                if (rm) {
                    const int r0 = __ffs(rm) - 1;
                    const double c0 = __shfl_sync(0xffffffffu, cr, r0);
                    if (r0 < rmin) {
                        rmin = r0;
                        cr_r = c0;
                    }
                }
                na += __popc(__ballot_sync(0xffffffffu, accd));
                __syncwarp();
            }
            if (rmin >= limit - 1) break;                // (no raise, or the last candidate that ran raised it)
            // candidates after the first raise saw the old c_max: the table as it was, again up to it
            limit = rmin + 1;
            if (fa) { S.rec[ha] = ld_rec_rw(list.at(a)); S.mod[ha] = 0; }
            if (fb) { S.rec[hb] = ld_rec_rw(list.at(b)); S.mod[hb] = 0; }
            __syncwarp();
        }
        __syncwarp();
        if (fa) { if (S.mod[ha]) st_rec(list.at(a), S.rec[ha]); S.mod[ha] = 0; S.key[ha] = -1; }
        if (fb) { if (S.mod[hb]) st_rec(list.at(b), S.rec[hb]); S.mod[hb] = 0; S.key[hb] = -1; }
        __syncwarp();
        acc += na;
        if (rmin < 32) {
            M = majorant(cr_r);
            k0 += rmin + 1;
        } else {
            k0 += nb;
        }
    }
    cmax = M.cm;
    nacc = acc;
}

// ------------------------------------------------------------------------------------------
// Exact fixed-point sums of particle moments: velocities at 2^-40, |xi|^2/2 at 2^-32.  Integer
// sums do not depend on the order of accumulation, so the per-cell flux sums are identical for
// every launch shape, and the global particle-flux ledger telescopes exactly.
// ------------------------------------------------------------------------------------------
// x * 2^S rounded to the nearest integer (ties to even): the product by the power of two is exact,
// then one conversion; |x| must stay below 2^(62-S) (guarded by the caller's range check).
template <int S>
__device__ __forceinline__ long long fx_bits(float x)
{
    return __float2ll_rn(__fmul_rn(x, static_cast<float>(1ull << S)));
}
__device__ __forceinline__ long long fx_vel(float x) { return fx_bits<40>(x); }
__device__ __forceinline__ long long fx_vel(double x) { return dbl_to_fixed<40>(x); }
// largest velocity component accepted in the exact sums (2^14; |xi|^2 then stays below 2^30):
// faster particles are reported as overflow
__device__ __forceinline__ bool fx_in_range(float x) { return fabsf(x) < 16384.0f; }
__device__ __forceinline__ bool fx_in_range(double x) { return (__double2hiint(x) & 0x7fffffff) < 0x40d00000; }

// |xi|^2/2 * 2^32: squares split exactly into float pairs (TwoProd by fma), summed error-free.
__device__ __forceinline__ long long fx_energy(float u, float v, float w)
{
    const float pu = u * u, pv = v * v, pw = w * w;
    const float qu = __fmaf_rn(u, u, -pu), qv = __fmaf_rn(v, v, -pv), qw = __fmaf_rn(w, w, -pw);
    float s = pu + pv;
    float bb = s - pu;
    float e = (pu - (s - bb)) + (pv - bb);
    const float s2 = s + pw;
    bb = s2 - s;
    e += (s - (s2 - bb)) + (pw - bb);
    const float lo = ((qu + qv) + qw) + e;
    return fx_bits<31>(s2) + fx_bits<31>(lo);
}
__device__ __forceinline__ long long fx_energy(double u, double v, double w)
{
    return dbl_to_fixed<31>(u * u + v * v + w * w);
}

// Prefetch of the 128-byte line holding p into L1 (a hint: no register, no fault on any address).
__device__ __forceinline__ void prefetch_l1(const void *p)
{
    asm volatile("prefetch.global.L1 [%0];" :: "l"(p));
}

// Plain (coherent) loads for records written earlier in the same kernel.
__device__ __forceinline__ RecF ld_rec_rw(const RecF *p)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return RecF{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ RecD ld_rec_rw(const RecD *p)
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0];
    const double2 b = reinterpret_cast<const double2 *>(p)[1];
    return RecD{a.x, a.y, b.x, b.y};
}

// Loads through L2 only (records read once, or overwritten by this block).
__device__ __forceinline__ RecF ld_rec_l2(const RecF *p)
{
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(p));
    return RecF{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ RecD ld_rec_l2(const RecD *p)
{
    const double2 a = __ldcg(reinterpret_cast<const double2 *>(p)), b = __ldcg(reinterpret_cast<const double2 *>(p) + 1);
    return RecD{a.x, a.y, b.x, b.y};
}

// Address of position x of a cell's arrived (sorted) list: far movers from the left, the left
// neighbour's R run (stored backwards), the cell's S run, the right neighbour's L run, far movers
// from the right.
template <typename Rec, typename FR>
__device__ __forceinline__ Rec *arrived_ptr(int x, const CellHdr &h, Rec *in, FR *fs)
{
    int r = x;
    if (r < h.nfb) return &fs[h.fb + r].rec;
    r -= h.nfb;
    if (r < h.Rn) return in + (h.Rend - 1 - r);
    r -= h.Rn;
    if (r < h.Sn) return in + (h.Sa + r);
    r -= h.Sn;
    if (r < h.Ln) return in + (h.La + r);
    r -= h.Ln;
    return &fs[h.fb + h.nfb + r].rec;
}

// Record x of a direct cell's list after re-sampling: the arrived positions, then the re-sampled
// particles after them in the cell's output block blk.
template <typename Rec, typename FR>
__device__ __forceinline__ Rec *list_rec(int x, const CellHdr &h, Rec *in, FR *fs, Rec *blk)
{
    return x < h.n_in ? arrived_ptr<Rec>(x, h, in, fs) : blk + x;
}

// Whether a direct cell's re-sampled particles (if any) are in place before the collision kernels
// run: none, or all drawn ahead by k_sample (kPreSampleMin or more of them).
__device__ __forceinline__ bool light_resampling(const CellHdr &h)
{
    return h.n_new == 0 || h.n_new >= kPreSampleMin;
}

// ------------------------------------------------------------------------------------------
// Collision kernel.  Runs before the streaming kernel on the cells of class kClsDirect and
// kClsStaged (work list built by k_offsets_flux):
//   direct: the candidate pairs depend only on counters, so up to 32 of them are drawn at once;
//           the touched particles (at most 64) are loaded into a shared-memory table keyed by list
//           position, collided there in candidate order, and the changed ones written back in
//           place, into the arrived runs or the far-mover list, where the streaming kernel reads
//           them; cells with more candidates or with re-sampled particles still to draw (drawn first,
//           after the arrived positions) run the candidates in dependency rounds on that list in place;
//   staged: the survivors of the absorption draw (Eq. p) and the re-sampled particles (Eq.
//           maxsample) are written to the first half of the cell's output block and collided there;
//           the streaming kernel reads this list instead of the arrived runs;
//   masked: the staged cells of a pool with the QMC split, absorbed and re-sampled by k_absorb: collided
//           where they arrived.
// ------------------------------------------------------------------------------------------
constexpr int kCollideThreads = 128;

// Position of the n-th (from 0) set bit of m (m has more than n set bits).
__device__ __forceinline__ int nth_set_bit(unsigned m, int n)
{
    int pos = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const int c = __popc(m & ((1u << w) - 1u));
        if (n >= c) {
            n -= c;
            m >>= w;
            pos += w;
        }
    }
    return pos;
}

// Light direct cells (P = 0, 1..kMaxDirect candidates, nothing re-sampled or every re-sampled particle
// drawn ahead by k_sample, as in a first step), packed: the warp holds
// the cells of list positions t0..n_items-1 (at most 32; one round of pack_rounds) and runs them in
// rounds.  A round takes the next cells whose candidates fit in the 32 lanes together:
// cell c on lanes [b_c, b_c + nc_c), lane b_c + k its candidate k, with the table slots
// [4 b_c, 4 (b_c + nc_c)) to itself.  Each ballot is masked
// to the cell's lanes, so every cell follows exactly the batches of a cell alone: its candidates
// drawn at once (the pairs depend only on counters), a batch cut before the first candidate that
// shares a particle with an earlier one of the batch and after the first whose c_r raises c_max.
// The touched particles are loaded into the table by the lane that inserted them, collided there
// in candidate order and the changed ones written back in place (into the arrived runs, the
// far-mover list or the re-sampled positions of the output block, where the streaming kernel reads
// them).
template <typename Rec>
__device__ __forceinline__ void collide_packed(const EngineDev &E, const int32_t *list, int t0, int n_items, Rec *in,
                                               Rec *out, FarItem<Rec> *fs)
{
    CollideShared<Rec> &S = collide_shared<Rec>();
    const int lane = threadIdx.x & 31;
    const unsigned upto = 0xffffffffu >> (31 - lane);          // lanes 0..lane
    int cg = -1, cn = 0;                                        // the chunk's cell at this lane
    if (t0 + lane < n_items) {
        cg = list[t0 + lane];
        const CellHdr *hp = E.hdr + cg;
        const int nc = hp->nc;
        if (hp->cls == kClsDirect && light_resampling(*hp) && nc >= 1 && nc <= kMaxDirect) cn = nc;
    }
    int done = 0;                                               // chunk cells collided so far
    while (__any_sync(0xffffffffu, lane >= done && cn > 0)) {
        int x = (lane >= done) ? cn : 0;                        // inclusive candidate count
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const bool inr = lane >= done && x <= 32;
        const unsigned rm = __ballot_sync(0xffffffffu, inr);
        const unsigned cells = __ballot_sync(0xffffffffu, inr && cn > 0);
        const unsigned starts = __reduce_or_sync(0xffffffffu, (inr && cn > 0) ? (1u << (x - cn)) : 0u);
        const int last = 31 - __clz(rm);
        const int total = __shfl_sync(0xffffffffu, x, last);
        done = last + 1;
        // this lane's cell and candidate
        const bool act = lane < total;
        const int sb = act ? 31 - __clz(starts & upto) : 0;
        const int src = act ? nth_set_bit(cells, __popc(starts & upto) - 1) : 0;
        const int g = __shfl_sync(0xffffffffu, cg, src);
        const int cn_src = __shfl_sync(0xffffffffu, cn, src);
        const int nc = act ? cn_src : 0;
        const int kc = lane - sb;
        if (act && !(kc >= 0 && kc < nc && sb + nc <= 32)) set_err(E.err, kErrOverflow);   // (cannot happen)
        const unsigned segmask = act ? ((0xffffffffu >> (32 - nc)) << sb) : 0u;
        for (int t = lane; t < 4 * total; t += 32) {
            S.key[t] = -1;
            S.own[t] = 32;
            S.mod[t] = 0;
        }
        __syncwarp();
        const CellHdr *hp = E.hdr + (act ? g : 0);
        const InstDev &I = E.inst[act ? hp->b : 0];
        int sa = 0, sc = 0;
        bool fa = false, fb = false;
        float2 bd = make_float2(0.0f, 0.0f);
        Rec *blk = nullptr;
        const uint32_t id = act ? cell_id(I, hp->i) : 0u, step = I.step;
        if (act) {
            const int N = hp->n_in + hp->n_new;
            blk = out + hp->off;
            uint32_t w[4];
            draw(I, id, 2u * static_cast<uint32_t>(kc), step, kCollide, w);
            const int pa = static_cast<int>(idx32(w[0], static_cast<uint32_t>(N)));
            int pb = static_cast<int>(idx32(w[1], static_cast<uint32_t>(N - 1)));
            if (pb >= pa) ++pb;
            sa = seg_insert(S.key, 4 * sb, 4 * nc, pa, fa, E.err);
            sc = seg_insert(S.key, 4 * sb, 4 * nc, pb, fb, E.err);
            if (fa) S.rec[sa] = ld_rec_rw(list_rec<Rec>(pa, *hp, in, fs, blk));
            if (fb) S.rec[sc] = ld_rec_rw(list_rec<Rec>(pb, *hp, in, fs, blk));
            bd = accept_bounds(w[2], __fdividef(1.0f, I.vhs_expo_f));
            if constexpr (sizeof(Rec) == sizeof(RecD)) pair_angles(S.rec, I, id, static_cast<uint32_t>(kc), step, S.ang[lane]);
        }
        __syncwarp();
        Majorant M = majorant(act ? E.cmax[g] : 0.0);
        int acc = 0, k0 = 0;
        bool raised = false;
        while (__any_sync(0xffffffffu, k0 < nc)) {
            const bool live = act && kc >= k0;
            if (live) { atomicMin(&S.own[sa], kc); atomicMin(&S.own[sc], kc); }
            __syncwarp();
            const bool conf = live && (S.own[sa] < kc || S.own[sc] < kc);
            const unsigned cmask = (__ballot_sync(0xffffffffu, conf) & segmask) >> sb;
            const int end1 = cmask ? __ffs(cmask) - 1 : nc;     // first candidate that shares a particle
            const bool inb = live && kc < end1;
            bool accd = false, raises = false, exact = false;
            double cr = 0.0;
            Rec A, B;
            decltype(rel_of(A, B)) rel{};
            if (inb) {
                A = S.rec[sa];
                B = S.rec[sc];
                rel = rel_of(A, B);
                accd = accept_pair(I, id, static_cast<uint32_t>(kc), step, A, B, rel, bd, M, cr, exact, raises);
            }
            const unsigned rmask = (__ballot_sync(0xffffffffu, raises) & segmask) >> sb;
            const int fr = rmask ? __ffs(rmask) - 1 : 32;
            const int end = min(end1, fr + 1);
            const double cr_r = __shfl_sync(0xffffffffu, cr, sb + (fr < 32 ? fr : 0));
            accd = accd && kc < end;
            if (accd) {
                if constexpr (sizeof(A.u) == 4) {
                    const RecPair<Rec> r = scatter_warp_drawn(I, id, static_cast<uint32_t>(kc), step, A, B);
                    S.rec[sa] = r.a;
                    S.rec[sc] = r.b;
                } else {
                    scatter_pair(I, id, static_cast<uint32_t>(kc), step, A, B, rel, S.ang[lane], true, cr, exact);
                    S.rec[sa] = A;
                    S.rec[sc] = B;
                }
                S.mod[sa] = 1;
                S.mod[sc] = 1;
            }
            acc += __popc(__ballot_sync(0xffffffffu, accd) & segmask);
            if (fr < end) {
                M = majorant(cr_r);
                raised = true;
            }
            __syncwarp();
            if (live) { S.own[sa] = 32; S.own[sc] = 32; }
            __syncwarp();
            if (k0 < nc) k0 = end;
        }
        if (act) {
            if (fa && S.mod[sa]) st_rec(list_rec<Rec>(S.key[sa], *hp, in, fs, blk), S.rec[sa]);
            if (fb && S.mod[sc]) st_rec(list_rec<Rec>(S.key[sc], *hp, in, fs, blk), S.rec[sc]);
            if (kc == 0) {
                E.ncand[g] = nc;
                E.nacc[g] = acc;
                if (raised) {
                    E.cmax[g] = M.cm;
                    E.fmaj[g] = majorant_factor(I, M.cm);
                }
            }
        }
        __syncwarp();
    }
}

// The list of a direct cell, read and updated in place: the arrived positions, then the re-sampled
// particles after them in the cell's output block.
template <typename Rec>
struct ArrivedList {
    const CellHdr *h;
    Rec *in;
    FarItem<Rec> *fs;
    Rec *blk;
    __device__ __forceinline__ Rec *at(int x) const { return x < h->n_in ? arrived_ptr<Rec>(x, *h, in, fs) : blk + x; }
};

// Direct cells with more than kMaxDirect candidates or with re-sampled particles, one per warp: the
// re-sampled particles first (sampling precedes the collisions), written after the arrived positions
// in the output block; then the candidates in dependency rounds (collide_list), the records read and
// written in place, where the streaming kernel reads them.
template <typename Rec>
__device__ __noinline__ void collide_big(const EngineDev &E, int g, Rec *in, Rec *out, FarItem<Rec> *fs)
{
    const int lane = threadIdx.x & 31;
    const CellHdr *hp = E.hdr + g;
    const InstDev &I = E.inst[hp->b];
    const int nc = hp->nc, n_in = hp->n_in, nn = hp->n_new, i = hp->i;
    const uint32_t id = cell_id(I, i), step = I.step;
    Rec *blk = out + hp->off;
    if (nn > 0 && !(hp->edges & kEdgePresampled)) {       // (otherwise drawn ahead by k_sample)
        if (I.resample_mode == 1) {
            sample_run_ce<Rec>(I, E.prim, E.valid, g, i, step, blk + n_in, 0, nn, lane);
        } else {
            const MaxwellCell mc = maxwell_cell_for<Rec>(I, E.prim + 5 * g);
            for (int j = lane; j < nn; j += 32)
                st_rec(blk + n_in + j, sample_particle<Rec>(I, id, static_cast<uint32_t>(j), step, mc, nullptr));
        }
        __syncwarp();
    }
    const double cm0 = E.cmax[g];
    double cmax = cm0;
    int na = 0;
    collide_list<Rec>(I, id, step, ArrivedList<Rec>{hp, in, fs, blk}, n_in + nn, nc, cmax, na, E.err);
    if (lane == 0) {
        E.ncand[g] = nc;
        E.nacc[g] = na;
        if (dbl_bits(cmax) != dbl_bits(cm0)) {
            E.cmax[g] = cmax;
            E.fmaj[g] = majorant_factor(I, cmax);
        }
    }
}

// Absorption draw u53(w0, w1) < P decided on the first word: with T = floor(P 2^32), w0 < T means
// u < P and w0 > T means u >= P; only w0 = T needs the 53-bit value.
__device__ __forceinline__ bool absorbed(uint32_t w0, uint32_t w1, double P, uint32_t T, bool all)
{
    if (all) return true;
    if (w0 != T) return w0 < T;
    return u53(w0, w1) < P;
}

template <typename Rec>
__device__ __noinline__ void collide_staged(const EngineDev &E, const InstDev &I, const CellHdr &h, int g, Rec *in, Rec *out,
                                            FarItem<Rec> *fs)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t id = cell_id(I, h.i), step = I.step;
    const double P = E.P[g];
    const bool all = !dbl_lt(P, 1.0), none = !dbl_gt(P, 0.0);   // u53 < 1 always
    const uint32_t T = (all || none) ? 0u : frac32(P);
    Rec *stage = out + h.off;
    int run = 0;
    for (int base = 0; base < h.n_in; base += 32) {
        const int k = base + lane;
        Rec v;
        bool keep = false;
        if (k < h.n_in) {
            v = ld_rec_rw(arrived_ptr<Rec>(k, h, in, fs));
            keep = true;
            if (!none) {
                uint32_t w[4];
                draw(I, id, static_cast<uint32_t>(k), step, kAbsorb, w);
                keep = !absorbed(w[0], w[1], P, T, all);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (keep) st_rec(stage + run + __popc(m & lt), v);
        run += __popc(m);
    }
    const double rho_t = E.psi[5 * g];
    const double rho_w = rho_t - fixed_to_double(run, 0) * I.mp_over_dx;
    const int64_t nn = E.valid[g] ? resample_count(I, id, step, P, rho_w) : 0;
    const int64_t n_tot = run + nn;
    if (n_tot > h.slots) {
        if (lane == 0) {
            set_err(E.err, kErrOverflow);
            E.hdr[g].cls = kClsSkip;
        }
        return;
    }
    if (nn > 0) {
        if (I.resample_mode == 1) {
            sample_run_ce<Rec>(I, E.prim, E.valid, g, h.i, step, stage + run, 0, static_cast<int>(nn), lane);
        } else {
            const MaxwellCell mc = maxwell_cell_for<Rec>(I, E.prim + 5 * g);
            for (int j = lane; j < nn; j += 32)
                st_rec(stage + run + j, sample_particle<Rec>(I, id, static_cast<uint32_t>(j), step, mc, nullptr));
        }
    }
    __syncwarp();
    const double cm0 = E.cmax[g];
    double cmax = cm0;
    int64_t nc = ntc_candidates(I, id, step, static_cast<int>(n_tot), rho_t, cmax, E.fmaj[g]);
    if (nc < 0) {
        if (lane == 0) set_err(E.err, kErrOverflow);
        nc = 0;
    }
    int na = 0;
    collide_list<Rec>(I, id, step, StagedList<Rec>{stage}, static_cast<int>(n_tot), nc, cmax, na, E.err);
    if (lane == 0) {
        E.ncand[g] = static_cast<int32_t>(nc);
        E.nacc[g] = na;
        E.nabs[g] = h.n_in - run;
        E.nnew[g] = static_cast<int32_t>(nn);
        if (dbl_bits(cmax) != dbl_bits(cm0)) {
            E.cmax[g] = cmax;
            E.fmaj[g] = majorant_factor(I, cmax);
        }
    }
}

// The list of a masked cell: the survivors among the arrived positions in their order, then the re-sampled
// particles in the output block.  Survivor x is found in the mask through the index S.pre (survivors
// before every stride-th word).
template <typename Rec>
struct MaskedList {
    const CellHdr *h;
    Rec *in;
    FarItem<Rec> *fs;
    Rec *blk;
    const uint32_t *mask;
    int run, words, stride;
    __device__ __forceinline__ Rec *at(int x) const
    {
        if (x >= run) return blk + x;
        const CollideShared<Rec> &S = collide_shared<Rec>();
        int lo = 0, hi = (words + stride - 1) / stride;         // pre[lo] <= x < pre[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (S.pre[mid] <= x) lo = mid;
            else hi = mid;
        }
        int r = x - S.pre[lo], w = lo * stride;
        uint32_t m = mask[w];
        for (int it = 1; it < stride && r >= __popc(m); ++it) {
            r -= __popc(m);
            m = mask[++w];
        }
        return arrived_ptr<Rec>(32 * w + nth_set_bit(m, r), *h, in, fs);
    }
};

// The candidates of a masked cell (absorbed and re-sampled by k_absorb), one warp, in place.
template <typename Rec>
__device__ __noinline__ void collide_masked(const EngineDev &E, const InstDev &I, int g, Rec *in, Rec *out, FarItem<Rec> *fs)
{
    CollideShared<Rec> &S = collide_shared<Rec>();
    const CellHdr &h = E.hdr[g];
    const int lane = threadIdx.x & 31;
    const uint32_t id = cell_id(I, h.i), step = I.step;
    const int run = h.n_in - E.nabs[g], n_tot = run + E.nnew[g];
    const double cm0 = E.cmax[g];
    int64_t nc = ntc_candidates(I, id, step, n_tot, E.psi[5 * g], cm0, E.fmaj[g]);
    if (nc < 0) {
        if (lane == 0) set_err(E.err, kErrOverflow);
        nc = 0;
    }
    double cmax = cm0;
    int na = 0;
    if (nc > 0) {
        // the survivor index
        const uint32_t *mask = survivor_mask(E, g, h.off);
        const int words = (h.n_in + 31) >> 5, stride = max(1, (words + kSelect - 1) / kSelect);
        int before = 0;
        for (int w0 = 0; w0 < words; w0 += 32) {
            const int c = (w0 + lane < words) ? __popc(mask[w0 + lane]) : 0;
            int x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (w0 + lane < words && (w0 + lane) % stride == 0) S.pre[(w0 + lane) / stride] = before + x - c;
            before += __shfl_sync(0xffffffffu, x, 31);
        }
        __syncwarp();
        collide_list<Rec>(I, id, step, MaskedList<Rec>{&h, in, fs, out + h.off, mask, run, words, stride}, n_tot, nc, cmax,
                          na, E.err);
    }
    if (lane == 0) {
        E.ncand[g] = static_cast<int32_t>(nc);
        E.nacc[g] = na;
        if (dbl_bits(cmax) != dbl_bits(cm0)) {
            E.cmax[g] = cmax;
            E.fmaj[g] = majorant_factor(I, cmax);
        }
    }
}

// ------------------------------------------------------------------------------------------
// Block kernel k_cellblock: one block of kBlockThreads per cell, persistent blocks over the work list
// of the cells with many collision candidates (the heavy list: staged cells, P > 0, and direct cells,
// P = 0, whose candidate count is at least heavy_min; the lighter ones run one warp per cell
// in the collision kernel).  Step 2 of Sec. 3.4 in the order the paper gives it:
//   absorption (staged cells): particle k of the arrived list is absorbed into the wave with
//     probability P (Eq. p); the survivors keep their order, compacted by the whole block into the
//     first half of the cell's output block;
//   re-sampling: (1-P) of the wave (Eq. maxsample), after the survivors (staged) or after the
//     arrived positions in the output block (direct), by the whole block;
//   NTC collisions (Appendix A) on that list.  Candidate k touches particles a_k, b_k and must see
//     them as every earlier candidate left them; candidates are taken in windows of kWindow and
//     executed in rounds: a candidate runs in the first round in which no earlier unfinished
//     candidate of the window touches either of its particles (each round every unfinished candidate
//     claims its two particles with atomicMax of (round, -position); the lowest position wins, so the
//     earliest unfinished candidate always runs and a window needs at most kWindow rounds).  The
//     candidates that may run in a round are packed into the first threads of the block, so that
//     only as many warps as there are runnable candidates / 32 execute the scattering.  This is the
//     sequential result whenever c_max stays fixed.  A candidate whose c_r exceeds c_max raises it,
//     and every later candidate must use the raised value: the window is first run with the
//     window's c_max; if any candidate raised it, the records are put back as they were at the
//     window's start and only the candidates up to the first raising one are run again (the raising
//     one accepted, as the sequential loop accepts it), and the next window starts after it with the
//     raised c_max.
// The records live in a shared-memory table during the collisions: the whole list when it has at
// most kBlockSlots records (slot = list position), otherwise the particles a window of
// candidates touches (hashed by list position); the changed records are written back after each
// window.
// ------------------------------------------------------------------------------------------
// What bounds it: the length of the dependent chain of a round (about 20 rounds for 700 candidates among
// 500 particles), not issue (39%) or memory.  So nothing that can be known before the round is left in it:
// pairs, acceptance bounds and scattering angles are formed for a whole window at once, a thread keeps its
// candidates' slots in registers, the runnable ones are listed per warp without an atomic, claims only
// grow, two candidates' draws interleave.  2510 heavy cells of a Kn sweep of Sod tubes:
// 307 -> 227 us in the step (beside the collision kernel), 266 -> 200 us alone.
constexpr int kBlockThreads = 128;
constexpr int kPer = 2;                             // window candidates per thread (window 256: five blocks per SM;
                                                    // 384 was slower on every workload with heavy cells)
constexpr int kWindow = kPer * kBlockThreads;       // candidates per window
constexpr int kBlockSlots = 1024;      // table slots (the hashed form holds at most 2 x kWindow keys)
static_assert(kBlockThreads == 128, "block_rounds: four warps");
static_assert((kBlockSlots & (kBlockSlots - 1)) == 0 && 4 * kWindow <= kBlockSlots && kPer == 2,
              "hashed table: a power of two, at most half full");
constexpr int kAbsorbPer = 4;          // arrived records per thread in flight in the absorption pass

template <typename Rec>
struct BlockShared {
    int key[kBlockSlots];          // hashed form: list position held by the slot, -1 = empty
    unsigned own[kBlockSlots];     // latest claim: (round << 16) | (0xffff - window position)
    unsigned char mod[kBlockSlots];// changed in the current window
    Rec rec[kBlockSlots];          // current values
    float2 wa[kWindow];            // acceptance bounds of the draw (accept_bounds)
    float4 sc[kWindow][2];         // scattering angles (pair_angles)
    unsigned char angok[kWindow];  // they are usable
    uint32_t ready[kWindow];       // the candidates that run in the current round (pack_cand), each warp's
                                   // from its own 32 kPer entries on
    CellHdr hdr;
    MaxwellCell mc;                // the cell's sampling state
    CeCell ce;
    int ce_on;
    int wsum[kAbsorbPer][kBlockThreads / 32];
    double u[2];                   // rounding draws of the re-sampled and the candidate count
    int item, nn, nc, ok, rmin, na;
    alignas(16) int nready[2][kBlockThreads / 32];  // the round's runnable candidates of each warp, by round parity
    // the current window: first candidate, the cell's generator id and step, the raised c_max
    int64_t k0;
    uint32_t id, step;
    double cm_new;
    // the list: in the output block (staged), or the arrived positions and then the output block
    Rec *in, *blk;
    FarItem<Rec> *fs;
    int staged, N;
    float inv_expo;
};

template <typename Rec>
__device__ __forceinline__ BlockShared<Rec> &block_shared()
{
    extern __shared__ __align__(16) unsigned char smraw[];
    return *reinterpret_cast<BlockShared<Rec> *>(smraw);
}

// A candidate in one word: the table slots of its pair and its window position.
__device__ __forceinline__ uint32_t pack_cand(int a, int b, int c)
{
    static_assert(kBlockSlots <= 1024 && kWindow <= 4096, "10 + 10 + 12 bits");
    return static_cast<uint32_t>(a) | (static_cast<uint32_t>(b) << 10) | (static_cast<uint32_t>(c) << 20);
}

// Slot of list position x (inserted if absent; `fresh`: by this call).
__device__ __forceinline__ int block_insert(int *key, int x, bool &fresh, int32_t *err)
{
    uint32_t h = __umulhi(static_cast<uint32_t>(x) * 2654435761u, static_cast<uint32_t>(kBlockSlots));
    for (int it = 0; it < kBlockSlots; ++it) {
        const int old = atomicCAS(&key[h], -1, x);
        if (old == -1 || old == x) {
            fresh = old == -1;
            return static_cast<int>(h);
        }
        h = (h + 1u) & (kBlockSlots - 1);
    }
    set_err(err, kErrOverflow);
    fresh = false;
    return 0;
}

// A candidate of the window (packed: pack_cand) run on the current records; returns whether it was
// accepted.
template <typename Rec>
__device__ __forceinline__ bool block_run_candidate(const InstDev &I, BlockShared<Rec> &S, uint32_t cand,
                                                    const Majorant &M, bool redo)
{
    const int sa = cand & 1023u, sb = (cand >> 10) & 1023u, c = cand >> 20;
    Rec A = S.rec[sa], B = S.rec[sb];
    const float2 bd = S.wa[c];
    const bool angok = S.angok[c] != 0;
    const auto rel = rel_of(A, B);
    double cr = 0.0;
    bool exact, raises;
    const uint32_t k = static_cast<uint32_t>(S.k0 + c);
    const bool a = accept_pair(I, S.id, k, S.step, A, B, rel, bd, M, cr, exact, raises);
    if (raises) {
        atomicMin(&S.rmin, c);
        if (redo) S.cm_new = cr;                   // in the rerun only the first raising candidate runs
    }
    if (a) {
        scatter_pair(I, S.id, k, S.step, A, B, rel, S.sc[c], angok, cr, exact);
        S.rec[sa] = A;
        S.rec[sb] = B;
        S.mod[sa] = 1;
        S.mod[sb] = 1;
    }
    return a;
}

// One pass of rounds over the window's candidates c < live_end (cand: this thread's, packed).  `round`:
// rounds run so far in this cell; claims only grow, so the table needs no clearing between passes.
// Returns the candidates accepted by this thread.
template <typename Rec>
__device__ __forceinline__ int block_rounds(const InstDev &I, BlockShared<Rec> &S, int live_end, const Majorant &M, bool redo,
                                            const uint32_t (&cand)[kPer], unsigned &round)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned lt = (1u << lane) - 1u;
    bool undone[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) undone[u] = t + u * kBlockThreads < live_end;
    // each round: the ready check of the claims made before it, a barrier, then the runs beside
    // the claims of the next round (the runs touch the records, the claims only own), a barrier
    auto claim = [&](unsigned r) {
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const unsigned code = (r << 16) | (0xffffu - static_cast<unsigned>(t + u * kBlockThreads));
            if (undone[u]) {
                atomicMax(&S.own[cand[u] & 1023u], code);
                atomicMax(&S.own[(cand[u] >> 10) & 1023u], code);
            }
        }
    };
    unsigned r = round + 1u;
    claim(r);
    __syncthreads();
    int remaining = live_end, na = 0;
    for (int it = 0; it <= kWindow && remaining > 0; ++it, ++r) {
        const int par = static_cast<int>(r & 1u);
        // the runnable candidates, appended to the round's list (any order: they touch disjoint particles)
        bool rdy[kPer];
        unsigned m[kPer];
        int n = 0;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const unsigned code = (r << 16) | (0xffffu - static_cast<unsigned>(t + u * kBlockThreads));
            rdy[u] = undone[u] && S.own[cand[u] & 1023u] == code && S.own[(cand[u] >> 10) & 1023u] == code;
            m[u] = __ballot_sync(0xffffffffu, rdy[u]);
            n += __popc(m[u]);
        }
        int pos = 32 * kPer * warp;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            if (rdy[u]) {
                S.ready[pos + __popc(m[u] & lt)] = cand[u];
                undone[u] = false;
            }
            pos += __popc(m[u]);
        }
        if (lane == 0) S.nready[par][warp] = n;
        __syncthreads();
        // the j-th of all of them lies j - (those of the warps before) into its warp's part
        const int4 nr = *reinterpret_cast<const int4 *>(S.nready[par]);
        const int n1 = nr.x, n2 = n1 + nr.y, n3 = n2 + nr.z, total = n3 + nr.w;
        claim(r + 1u);
        for (int j = t; j < total; j += kBlockThreads) {
            const int at = j < n2 ? (j < n1 ? j : j - n1 + 32 * kPer) : (j < n3 ? j - n2 + 64 * kPer : j - n3 + 96 * kPer);
            na += block_run_candidate<Rec>(I, S, S.ready[at], M, redo) ? 1 : 0;
        }
        remaining -= total;
        __syncthreads();
    }
    round = r;
    return na;
}

// Record x of the block's list.
template <typename Rec>
__device__ __forceinline__ Rec *block_rec(const BlockShared<Rec> &S, int x)
{
    if (S.staged || x >= S.hdr.n_in) return S.blk + x;
    return arrived_ptr<Rec>(x, S.hdr, S.in, S.fs);
}

// Candidates c0, c0 + kBlockThreads, ... (kU of them, those below nw) of the window: their pairs (packed),
// acceptance bounds and scattering angles.  Lists longer than the table: the pairs' particles are
// hashed into it; the thread that inserts one owns the slot (loads the record here, writes it back,
// frees the slot): bits 2u and 2u + 1 of .w.  Several candidates together, so that their chains of
// dependent operations (two generator calls each) interleave; hashed lists one at a time.
template <typename Rec, int kU>
__device__ __noinline__ uint4 block_draw(const InstDev &I, int c0, int nw, int32_t *err)
{
    static_assert(kU <= 2, "packed candidates");
    BlockShared<Rec> &S = block_shared<Rec>();
    const uint32_t id = S.id, step = S.step, k0 = static_cast<uint32_t>(S.k0 + c0);
    const int N = S.N;
    uint32_t out[4] = {0u, 0u, 0u, 0u};
    int pa[kU], pb[kU];
    Rec ra[kU], rb[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        uint32_t w[4];
        draw(I, id, 2u * (k0 + u * kBlockThreads), step, kCollide, w);
        pa[u] = static_cast<int>(idx32(w[0], static_cast<uint32_t>(N)));
        pb[u] = static_cast<int>(idx32(w[1], static_cast<uint32_t>(N - 1)));
        if (pb[u] >= pa[u]) ++pb[u];
        const float2 bd = accept_bounds(w[2], S.inv_expo);
        if (c0 + u * kBlockThreads < nw) S.wa[c0 + u * kBlockThreads] = bd;
    }
    if (kU == 1 && N > kBlockSlots) {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (c0 + u * kBlockThreads >= nw) continue;
            bool fa, fb;
            const int xa = pa[u], xb = pb[u];
            pa[u] = block_insert(S.key, xa, fa, err);
            pb[u] = block_insert(S.key, xb, fb, err);
            if (fa) ra[u] = ld_rec_rw(block_rec(S, xa));
            if (fb) rb[u] = ld_rec_rw(block_rec(S, xb));
            out[3] |= ((fa ? 1u : 0u) | (fb ? 2u : 0u)) << (2 * u);
        }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        const int c = c0 + u * kBlockThreads;
        float4 ang[2];
        const bool ok = pair_angles(S.rec, I, id, k0 + u * kBlockThreads, step, ang);
        if (c < nw) {
            S.angok[c] = ok ? 1 : 0;
            S.sc[c][0] = ang[0];
            S.sc[c][1] = ang[1];
            out[u] = pack_cand(pa[u], pb[u], c);
        }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        if (out[3] & (1u << (2 * u))) S.rec[pa[u]] = ra[u];
        if (out[3] & (2u << (2 * u))) S.rec[pb[u]] = rb[u];
    }
    return make_uint4(out[0], out[1], out[2], out[3]);
}

// The nc candidates of a list of N records (written earlier by this block or in place).  The list
// in memory holds the state at the start of each window: the changed records are written back after
// every window, and a window rerun after a raise of c_max reloads them from there.
// cm: the cell's c_max; returns it (raised or not), the accepted candidates in S.na.  (A function of its
// own, as block_absorb: the registers of the window loops are not held beside the other phases'.)
template <typename Rec>
__device__ __noinline__ double block_collisions(const EngineDev &E, const InstDev &I, uint32_t id, uint32_t step, Rec *in,
                                                FarItem<Rec> *fs, Rec *blk, bool staged, int N, int64_t nc, double cm)
{
    BlockShared<Rec> &S = block_shared<Rec>();
    const int t = threadIdx.x;
    constexpr int kLd = 4;                        // records per thread in flight
    const bool whole = N <= kBlockSlots;          // the whole list in the table, slot = position
    int na = 0;
    if (t == 0) {
        S.na = 0;
        S.in = in;
        S.blk = blk;
        S.fs = fs;
        S.staged = staged ? 1 : 0;
        S.N = N;
        S.inv_expo = __fdividef(1.0f, I.vhs_expo_f);     // (inf for Maxwell molecules)
    }
    if (N < 2 || nc <= 0) return cm;
    __syncthreads();
    if (whole) {
        for (int x0 = t; x0 < N; x0 += kLd * kBlockThreads) {
            Rec v[kLd];
#pragma unroll
            for (int u = 0; u < kLd; ++u)
                if (x0 + u * kBlockThreads < N) v[u] = ld_rec_rw(block_rec(S, x0 + u * kBlockThreads));
#pragma unroll
            for (int u = 0; u < kLd; ++u) {
                const int x = x0 + u * kBlockThreads;
                if (x < N) { S.rec[x] = v[u]; S.own[x] = 0u; S.mod[x] = 0; }
            }
        }
    } else {
        for (int x = t; x < kBlockSlots; x += kBlockThreads) { S.key[x] = -1; S.own[x] = 0u; S.mod[x] = 0; }
    }
    unsigned round = 0;
    int64_t k_lo = 0;
    while (k_lo < nc) {
        const int nw = static_cast<int>(min(static_cast<int64_t>(kWindow), nc - k_lo));
        __syncthreads();
        if (round + 2u * (kWindow + 2u) > 0xffffu) {       // the claims' round field is full: start over
            for (int x = t; x < kBlockSlots; x += kBlockThreads) S.own[x] = 0u;
            round = 0;
        }
        if (t == 0) {
            S.rmin = kWindow;
            S.k0 = k_lo;
            S.id = id;
            S.step = step;
        }
        __syncthreads();
        uint32_t cand[kPer] = {0u, 0u};
        unsigned owns = 0u;                       // the slots this thread owns: bits 2u (a) and 2u + 1 (b)
        if (whole && (t & ~31) + kBlockThreads < nw) {
            const uint4 d = block_draw<Rec, 2>(I, t, nw, E.err);
            cand[0] = d.x;
            cand[1] = d.y;
        } else {
            // (hashed: one after the other, a candidate's loads beside its angles)
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                if (t + u * kBlockThreads < nw) {
                    const uint4 d = block_draw<Rec, 1>(I, t + u * kBlockThreads, nw, E.err);
                    cand[u] = d.x;
                    owns |= d.w << (2 * u);
                }
            }
        }
        __syncthreads();
        const Majorant M = majorant(cm);
        int upto = nw;
        for (bool redo = false;; redo = true) {
            const int acc = block_rounds<Rec>(I, S, upto, M, redo, cand, round);
            const int r = S.rmin;
            if (redo || r >= nw) {
                if (redo) cm = S.cm_new;
                na += acc;
                break;
            }
            // the candidates after position r saw c_max before its raise: back to the window's start
            // (the records in memory) and again up to r only
            upto = r + 1;
            if (whole) {
                for (int x = t; x < N; x += kBlockThreads) {
                    if (S.mod[x]) S.rec[x] = ld_rec_rw(block_rec(S, x));
                    S.mod[x] = 0;
                }
            } else {
#pragma unroll
                for (int e = 0; e < 2 * kPer; ++e) {
                    const int x = (cand[e >> 1] >> ((e & 1) * 10)) & 1023u;
                    if ((owns >> e) & 1u) {
                        if (S.mod[x]) S.rec[x] = ld_rec_rw(block_rec(S, S.key[x]));
                        S.mod[x] = 0;
                    }
                }
            }
            __syncthreads();
        }
        if (whole) {
            for (int x0 = t; x0 < N; x0 += kLd * kBlockThreads) {
                bool ch[kLd];
#pragma unroll
                for (int u = 0; u < kLd; ++u) {
                    const int x = x0 + u * kBlockThreads;
                    ch[u] = x < N && S.mod[x] != 0;
                }
#pragma unroll
                for (int u = 0; u < kLd; ++u) {
                    const int x = x0 + u * kBlockThreads;
                    if (ch[u]) {
                        st_rec(block_rec(S, x), S.rec[x]);
                        S.mod[x] = 0;
                    }
                }
            }
        } else {
#pragma unroll
            for (int e = 0; e < 2 * kPer; ++e) {
                const int x = (cand[e >> 1] >> ((e & 1) * 10)) & 1023u;
                if ((owns >> e) & 1u) {
                    if (S.mod[x]) st_rec(block_rec(S, S.key[x]), S.rec[x]);
                    S.key[x] = -1;
                    S.mod[x] = 0;
                }
            }
        }
        k_lo += upto;
    }
    na = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(na));
    if ((t & 31) == 0) atomicAdd(&S.na, na);
    __syncthreads();
    return cm;
}

// Staged cell: absorption and compaction of the survivors into the first half of the output block.
// Returns the survivors.
template <typename Rec>
__device__ __noinline__ int block_absorb(const EngineDev &E, const InstDev &I, int g, Rec *in, FarItem<Rec> *fs, Rec *stage,
                                         uint32_t id, uint32_t step)
{
    BlockShared<Rec> &S = block_shared<Rec>();
    const CellHdr &h = S.hdr;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const double P = E.P[g];
    const bool all = !dbl_lt(P, 1.0), none = !dbl_gt(P, 0.0);   // u53 < 1 always
    const uint32_t T = (all || none) ? 0u : frac32(P);
    int run = 0;
    for (int base = 0; base < h.n_in; base += kAbsorbPer * kBlockThreads) {
        Rec v[kAbsorbPer];
        bool keep[kAbsorbPer];
#pragma unroll
        for (int u = 0; u < kAbsorbPer; ++u) {
            const int k = base + u * kBlockThreads + t;
            keep[u] = k < h.n_in;
            if (keep[u]) v[u] = ld_rec_rw(arrived_ptr<Rec>(k, h, in, fs));
        }
#pragma unroll
        for (int u = 0; u < kAbsorbPer; ++u) {
            const int k = base + u * kBlockThreads + t;
            if (keep[u] && !none) {
                uint32_t w[4];
                draw(I, id, static_cast<uint32_t>(k), step, kAbsorb, w);
                keep[u] = !absorbed(w[0], w[1], P, T, all);
            }
            const unsigned m = __ballot_sync(0xffffffffu, keep[u]);
            if (lane == 0) S.wsum[u][warp] = __popc(m);
        }
        __syncthreads();
        int pre = run;
#pragma unroll
        for (int u = 0; u < kAbsorbPer; ++u) {
            int before = 0, tot = 0;
#pragma unroll
            for (int w = 0; w < kBlockThreads / 32; ++w) {
                const int c = S.wsum[u][w];
                before += (w < warp) ? c : 0;
                tot += c;
            }
            const unsigned m = __ballot_sync(0xffffffffu, keep[u]);
            if (keep[u]) st_rec(stage + pre + before + __popc(m & lt), v[u]);
            pre += tot;
        }
        run = pre;
        __syncthreads();
    }
    return run;
}

template <typename Rec>
__device__ void block_cell(const EngineDev &E, int g, BlockShared<Rec> &S, Rec *in, Rec *out, FarItem<Rec> *fs)
{
    const int t = threadIdx.x;
    if (t < static_cast<int>(sizeof(CellHdr) / 16))
        reinterpret_cast<int4 *>(&S.hdr)[t] = reinterpret_cast<const int4 *>(E.hdr + g)[t];
    __syncthreads();
    const CellHdr &h = S.hdr;
    if (h.cls != kClsStaged && h.cls != kClsDirect) return;
    const InstDev &I = E.inst[h.b];
    const bool staged = h.cls == kClsStaged;
    const uint32_t id = cell_id(I, h.i), step = I.step;
    Rec *blk = out + h.off;
    // NS-corrected sampling: the cell's state and coefficients, by one thread of the last warp while the
    // others absorb (without it every sampling thread forms the state itself: waited for here, it held
    // the absorption's barrier for 3.4k of the 10.7k cycles until then)
    const bool ce = I.resample_mode == 1;
    if (ce && t == kBlockThreads - 32 && (!staged || E.valid[g]) && (staged || h.n_new > 0)) {
        S.mc = maxwell_cell(I, E.prim + 5 * g);
        S.ce_on = ce_coefs(I, E.prim, E.valid, g, h.i, S.ce) ? 1 : 0;
    }
    int run = h.n_in;
    const double cm0 = E.cmax[g];
    double rho_t = 0.0, P = 0.0, fmaj = 0.0;
    int valid = 0;
    if (staged) {
        // what the counts need, ahead of the absorption: the state, and the two rounding draws by two lanes
        if (t == 0) {
            rho_t = E.psi[5 * g];
            P = E.P[g];
            fmaj = E.fmaj[g];
            valid = E.valid[g];
        }
        if (t < 2) S.u[t] = round_draw(I, id, static_cast<uint32_t>(t), step);
        __syncwarp();                     // (a cell without arrived particles passes no barrier in block_absorb)
        run = block_absorb<Rec>(E, I, g, in, fs, blk, id, step);
    }
    // re-sampled and candidate counts
    if (t == 0) {
        if (staged) {
            const double rho_w = rho_t - fixed_to_double(run, 0) * I.mp_over_dx;
            const int64_t nn = valid ? resample_count(I, P, rho_w, S.u[0]) : 0;
            const int64_t n_tot = run + nn;
            S.ok = (n_tot <= h.slots) ? 1 : 0;
            S.nn = static_cast<int>(nn < h.slots ? nn : h.slots);
            int64_t nc = 0;
            if (S.ok) {
                nc = ntc_candidates(I, static_cast<int>(n_tot), rho_t, cm0, fmaj, S.u[1]);
                if (nc < 0 || nc > INT32_MAX) {
                    set_err(E.err, kErrOverflow);
                    nc = 0;
                }
            } else {
                set_err(E.err, kErrOverflow);
                E.hdr[g].cls = kClsSkip;
            }
            S.nc = static_cast<int>(nc);
        } else {
            S.ok = 1;
            S.nn = h.n_new;
            S.nc = h.nc;
        }
    }
    __syncthreads();
    if (!S.ok) return;
    const int nn = S.nn;
    const int n_tot = run + nn;
    if (nn > 0 && (staged || !(h.edges & kEdgePresampled))) {   // (otherwise drawn ahead by k_sample)
        if (ce) {
            const MaxwellCell mc = S.mc;
            const CeCell *cc = S.ce_on ? &S.ce : nullptr;
            for (int j = t; j < nn; j += kBlockThreads)
                st_rec(blk + run + j, sample_particle<Rec>(I, id, static_cast<uint32_t>(j), step, mc, cc));
        } else if ((t & ~31) < nn) {
            const MaxwellCell mc = maxwell_cell_for<Rec>(I, E.prim + 5 * g);
            for (int j = t; j < nn; j += kBlockThreads)
                st_rec(blk + run + j, sample_particle<Rec>(I, id, static_cast<uint32_t>(j), step, mc, nullptr));
        }
    }
    __syncthreads();
    const double cmax = block_collisions<Rec>(E, I, id, step, in, fs, blk, staged, n_tot, S.nc, cm0);
    if (t == 0) {
        E.ncand[g] = S.nc;
        E.nacc[g] = S.na;
        if (staged) {
            E.nabs[g] = h.n_in - run;
            E.nnew[g] = nn;
        }
        if (dbl_bits(cmax) != dbl_bits(cm0)) {
            E.cmax[g] = cmax;
            E.fmaj[g] = majorant_factor(I, cmax);
        }
    }
}

template <typename Rec, int kMinB>
__global__ void __launch_bounds__(kBlockThreads, kMinB) k_cellblock(const __grid_constant__ EngineDev E, int rp)
{
    wait_predecessor();
    BlockShared<Rec> &S = block_shared<Rec>();
    Rec *in = static_cast<Rec *>(E.buf[rp]);
    Rec *out = static_cast<Rec *>(E.buf[1 - rp]);
    FarItem<Rec> *fs = static_cast<FarItem<Rec> *>(E.far_sorted);
    const int n_long = E.ticket[kLongLen], n_items = n_long + E.ticket[kListLen + kHeavyList];
    if (n_items == 0) return;                 // (written by the kernel before: the same for every thread)
    const int32_t *list = E.wl + static_cast<size_t>(kHeavyList) * E.G;
    // the block's first cell by its index, the others by ticket (taken when the block is free: taken ahead,
    // cells waited behind long ones while other blocks had finished)
    for (int it = static_cast<int>(blockIdx.x); it < n_items;) {
        block_cell<Rec>(E, it < n_long ? list[E.G - 1 - it] : list[it - n_long], S, in, out, fs);
        if (threadIdx.x == 0) S.item = static_cast<int>(gridDim.x) + atomicAdd(&E.ticket[kHeavyList], 1);
        __syncthreads();
        it = S.item;
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------
// Particles drawn ahead (Eq. maxsample, or its NS-corrected option): the re-sampled particles of
// direct cells with at least kPreSampleMin of them -- every particle of a first step -- in chunks of
// kSampleChunk over all warps of the GPU, into the positions after the cell's arrived list in its
// output block, before the collision kernels collide them there.  First the rounds of the light list.
// ------------------------------------------------------------------------------------------
constexpr int kSampleThreads = 256;

// Rounds of the light list (one item each for the collision kernel): the light cells of each warp of
// k_offsets_flux (consecutive in the list), in order, in groups whose candidates fit in the 32
// lanes of a warp; one descriptor (first position, cells) per round.
// Returns the number of rounds; lane r < (that number) holds round r in `mine`.
__device__ __forceinline__ int pack_rounds(const EngineDev &E, int grp, int lane, int2 &mine)
{
    mine = make_int2(0, 0);
    const int n_groups = (E.G_run + 31) / 32;
    const int2 gr = (grp < n_groups) ? E.wgrp[grp] : make_int2(0, 0);
    if (gr.y <= 0) return 0;
    int ncl = 0;
    if (lane < gr.y) ncl = E.wlnc[gr.x + lane];
    int done = 0, nr = 0;
    while (__any_sync(0xffffffffu, lane >= done && ncl > 0)) {
        int x = (lane >= done) ? ncl : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const unsigned rm = __ballot_sync(0xffffffffu, lane >= done && x <= 32);
        const int last = min(31 - __clz(rm), gr.y - 1);
        if (lane == nr) mine = make_int2(gr.x + done, last + 1 - done);
        ++nr;
        done = last + 1;
    }
    return nr;
}

template <typename Rec>
__global__ void __launch_bounds__(kSampleThreads, 4) k_sample(const __grid_constant__ EngineDev E, int rp)
{
    wait_predecessor();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kW = kSampleThreads / 32;
    const int n_groups = (E.G_run + 31) / 32;
    // one group per warp, one atomic per block for the rounds of its warps
    __shared__ int s_nr[kW], s_base;
    for (int w0 = blockIdx.x * kW; w0 < n_groups; w0 += gridDim.x * kW) {
        int2 mine;
        const int nr = pack_rounds(E, w0 + warp, lane, mine);
        if (lane == 0) s_nr[warp] = nr;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int k = 0; k < kW; ++k) tot += s_nr[k];
            s_base = tot ? atomicAdd(&E.ticket[kRoundLen], tot) : 0;
        }
        __syncthreads();
        int base = s_base;
        for (int k = 0; k < warp; ++k) base += s_nr[k];
        if (lane < nr) {
            if (base + lane < E.G) E.wr[base + lane] = mine;
            else set_err(E.err, kErrOverflow);
        }
        __syncthreads();
    }
    Rec *out = static_cast<Rec *>(E.buf[1 - rp]);
    const int n_chunks = min(E.ticket[kPreLen], E.wls_cap);
    if (n_chunks == 0) return;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&E.ticket[kPreCtr], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= n_chunks) break;
        const int2 it = E.wlp[t];
        const int g = it.x, j0 = it.y;
        const CellHdr &h = E.hdr[g];
        const int b = h.b, n_in = h.n_in, n_new = h.n_new, cls = h.cls, i = h.i;
        const long long off = h.off;
        if (cls != kClsDirect && cls != kClsStream) continue;
        const InstDev &I = E.inst[b];
        const int j1 = min(j0 + kSampleChunk, n_new);
        if (I.resample_mode == 1) {
            sample_run_ce<Rec>(I, E.prim, E.valid, g, i, I.step, out + off + n_in, j0, j1, lane);
            continue;
        }
        // (the draws unrolled here: this kernel's loop is short)
        const MaxwellCell mc = maxwell_cell_for<Rec>(I, E.prim + 5 * g);
        for (int j = j0 + lane; j < j1; j += 32)
            st_rec(out + off + n_in + j, sample_particle<Rec, false>(I, cell_id(I, i), static_cast<uint32_t>(j),
                                                                     I.step, mc, nullptr));
    }
}

// Absorption and re-sampling of the staged cells (P > 0) with few candidates, one warp per cell, in pools with
// the QMC split, where every cell absorbs.  The absorption draws depend only on counters, so they become
// a bit mask of the survivors, no particle is read, and the streaming kernel skips the absorbed ones
// where it reads the list anyway.  The re-sampled particles go to the output block after as many places
// as there are survivors (the stayers written so far never lie beyond the read position).  A kernel of
// its own: beside the collisions the three phases' code did not fit the instruction cache (0.47 ms for
// the two, most of a warp's stalls waits for instructions).  Copying the survivors into the output
// block first, as collide_staged does, reads and writes every particle once more, a load latency per 32
// of them: 0.75 ms of the QMC batch's 1.03 ms step.  Pools without the QMC split keep the copy: their
// staged cells are few, and the streaming kernel's test of the mask costs the others 0.6%.
template <typename Rec>
__global__ void __launch_bounds__(kSampleThreads, 4) k_absorb(const __grid_constant__ EngineDev E, int rp)
{
    wait_predecessor();
    const int lane = threadIdx.x & 31;
    Rec *out = static_cast<Rec *>(E.buf[1 - rp]);
    const int n_items = E.ticket[kListLen + kWarpList];
    const int32_t *list = E.wl + (E.G - 1);     // (backwards)
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&E.ticket[kAbsorbCtr], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= n_items) break;
        const int g = list[-t];
        const CellHdr &h = E.hdr[g];
        if (h.cls != kClsStaged) continue;
        const InstDev &I = E.inst[h.b];
        const uint32_t id = cell_id(I, h.i), step = I.step;
        const double P = E.P[g];
        const bool all = !dbl_lt(P, 1.0), none = !dbl_gt(P, 0.0);   // u53 < 1 always
        const uint32_t T = (all || none) ? 0u : frac32(P);
        const int n_in = h.n_in, slots = h.slots, ci = h.i;
        const int64_t off = h.off;
        uint32_t *mask = survivor_mask(E, g, off);
        const int words = (n_in + 31) >> 5;
        int run = 0;
        constexpr int kU = 4;                    // words per iteration (independent draws)
        for (int w0 = 0; w0 < words; w0 += kU) {
            uint32_t m[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int k = 32 * (w0 + u) + lane;
                uint32_t w[4];
                draw(I, id, static_cast<uint32_t>(k), step, kAbsorb, w);
                m[u] = __ballot_sync(0xffffffffu, k < n_in && (none || !absorbed(w[0], w[1], P, T, all)));
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (lane == u && w0 + u < words) mask[w0 + u] = m[u];
                run += __popc(m[u]);
            }
        }
        const double rho_w = E.psi[5 * g] - fixed_to_double(run, 0) * I.mp_over_dx;
        const int64_t nn = E.valid[g] ? resample_count(I, id, step, P, rho_w) : 0;
        if (run + nn > slots) {
            if (lane == 0) {
                set_err(E.err, kErrOverflow);
                E.hdr[g].cls = kClsSkip;
            }
            continue;
        }
        __syncwarp();
        if (lane == 0) {
            E.hdr[g].cls = kClsMasked;
            E.nabs[g] = n_in - run;
            E.nnew[g] = static_cast<int32_t>(nn);
        }
        Rec *first = out + off + run;
        if (I.resample_mode == 1) {
            sample_run_ce<Rec>(I, E.prim, E.valid, g, ci, step, first, 0, static_cast<int>(nn), lane);
        } else {
            const MaxwellCell mc = maxwell_cell_for<Rec>(I, E.prim + 5 * g);
            for (int j = lane; j < nn; j += 32)
                st_rec(first + j, sample_particle<Rec>(I, id, static_cast<uint32_t>(j), step, mc, nullptr));
        }
    }
}

// Blocks per SM: single-precision records at 64 registers; double-precision records at 80 (the Mach-3 shock of
// 100 cells 79 -> 72 us per step; six blocks were slower for single-precision absorption, 5.16 -> 5.45 ms on
// the QMC batch).
template <typename Rec, bool kMasked>
__global__ void __launch_bounds__(kCollideThreads, sizeof(Rec) == sizeof(RecF) ? 8 : 6) k_collide(const __grid_constant__ EngineDev E, int rp)
{
    wait_predecessor();
    const int lane = threadIdx.x & 31;
    Rec *in = static_cast<Rec *>(E.buf[rp]);
    Rec *out = static_cast<Rec *>(E.buf[1 - rp]);
    FarItem<Rec> *fs = static_cast<FarItem<Rec> *>(E.far_sorted);
    // the other cells of this kernel (direct cells with more than kMaxDirect candidates or with
    // re-sampled particles, staged cells), one per warp, then the rounds of the light direct cells
    // (packed by k_sample: one round is one item); the next ticket is fetched while the current item
    // runs (the heavy cells: k_cellblock)
    {
        const int n_items = E.ticket[kListLen + kWarpList];
        const int32_t *list = E.wl + (E.G - 1);     // (backwards)
        int t = 0;
        if (lane == 0) t = atomicAdd(&E.ticket[kWarpList], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        while (t < n_items) {
            int tn = 0;
            if (lane == 0) tn = atomicAdd(&E.ticket[kWarpList], 1);
            const int g = list[-t];
            const CellHdr h = E.hdr[g];
            if constexpr (kMasked) {
                if (h.cls == kClsMasked) collide_masked<Rec>(E, E.inst[h.b], g, in, out, fs);
            } else {
                if (h.cls == kClsStaged) collide_staged<Rec>(E, E.inst[h.b], h, g, in, out, fs);
            }
            if (h.cls == kClsDirect) collide_big<Rec>(E, g, in, out, fs);
            __syncwarp();
            t = __shfl_sync(0xffffffffu, tn, 0);
        }
    }
    {
        const int n_rounds = min(E.ticket[kRoundLen], E.G);
        const int32_t *list = E.wl + static_cast<size_t>(kLightList) * E.G;
        const int n_light = E.ticket[kListLen + kLightList];
        int t = 0;
        if (lane == 0) t = atomicAdd(&E.ticket[kRoundCtr], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        while (t < n_rounds) {
            int tn = 0;
            if (lane == 0) tn = atomicAdd(&E.ticket[kRoundCtr], 1);
            const int2 r = E.wr[t];
            collide_packed<Rec>(E, list, r.x, min(r.x + min(r.y, 32), n_light), in, out, fs);
            t = __shfl_sync(0xffffffffu, tn, 0);
        }
    }
    // re-sampled particles of cells without collisions (Eq. maxsample), chunk by chunk, into the
    // positions after the cell's arrived list in its output block
    const int n_chunks = min(E.ticket[kSampleLen], E.wls_cap);
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&E.ticket[kSampleCtr], 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= n_chunks) break;
        const int2 it = E.wls[t];
        const int g = it.x, j0 = it.y;
        const CellHdr &h = E.hdr[g];
        const int b = h.b, n_in = h.n_in, n_new = h.n_new, cls = h.cls, i = h.i;
        const long long off = h.off;
        if (cls != kClsStream && cls != kClsReservoir) continue;
        const InstDev &I = E.inst[b];
        const int j1 = min(j0 + kSampleChunk, n_new);
        if (I.resample_mode == 1 && cls == kClsStream) {
            sample_run_ce<Rec>(I, E.prim, E.valid, g, i, I.step, out + off + n_in, j0, j1, lane);
            continue;
        }
        const MaxwellCell mc = maxwell_cell_for<Rec>(I, E.prim + 5 * g);
        for (int j = j0 + lane; j < j1; j += 32)
            st_rec(out + off + n_in + j, sample_particle<Rec>(I, cell_id(I, i), static_cast<uint32_t>(j), I.step, mc,
                                                              nullptr));
    }
}

// ------------------------------------------------------------------------------------------
// Streaming kernel: one warp per cell.
//
// Output block of a cell s (2 x slots records, slots = the bound on its list after re-sampling):
// particles that stay (S) are written forward from the block start, those moving one cell left
// (L) forward from the middle, those moving one cell right (R) backward from the end; each run
// keeps the order the particles had before transport.  The sorted list of cell g for the next
// step reads R(g-1) from its end backwards, then S(g), then L(g+1).  A staged cell's list lies
// in the first half of its own block; its stayers are written back in place, never ahead of the
// read position.  Any split of the list into consecutive groups gives the same stable order, so
// every piece of the list is streamed in its own groups of 32.
//
// Register use decides the bandwidth of this kernel (it needs about 48 resident warps per SM to
// keep HBM busy), so the loop state is small: the piece descriptors live in shared memory and the
// rare cases (walls, wraps, leavers, moves of two or more cells) share one code path.
// ------------------------------------------------------------------------------------------
// One piece of a cell's list: list positions [k0, k0 + n); kind 0: records at p[dir * r], read-only
// loads (arrived runs); 1: records at p[r], plain loads (records written by the collision kernel
// into the output block); 2: the records of the sorted far-list items p[r].
template <typename Rec>
struct Piece {
    const void *p;
    int n, k0, dir, kind;
};

template <typename Rec>
struct StreamShared {
    long long acc[4][32];     // lane-private rare-path sums (u, v, w, |xi|^2/2)
    Piece<Rec> piece[6];
};

// Records of the list in flight: kStreamStages iterations of 32 x groups records, each slot written
// (by an asynchronous copy) and read by the same lane.
constexpr int kStreamStages = 3;
template <typename Rec, int kGroups>
struct StreamRing {
    Rec rec[kStreamStages][32 * kGroups];
};

// Asynchronous 16-byte copy global -> shared (L2 only), its commit and the wait for all but the N
// most recent groups of this thread.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Address of position r of a piece of the list (kind 0: arrived runs, stored forward or backward;
// 1: records in the output block; 2: sorted far-list items).
template <typename Rec>
__device__ __forceinline__ const Rec *piece_rec(const Piece<Rec> &pc, int r)
{
    if (pc.kind == 2) return &static_cast<const FarItem<Rec> *>(pc.p)[r].rec;
    return static_cast<const Rec *>(pc.p) + (pc.kind == 0 ? pc.dir * r : r);
}

struct StreamState {
    int oS, oL, oR;                       // next write offsets in the block: S, L (forward), R (backward)
    int ngone;                            // far movers and removed particles of this lane
    bool range_ok;
};

// Full transport of one particle (Step 3) with 64-bit cell arithmetic and the boundary conditions.
__device__ __forceinline__ int64_t transport_full(const InstDev &I, int64_t cell, float &xl, float &u, bool &refl)
{
    const float s = __fmaf_rn(u, I.dtdx_f, xl);
    if (!(fabsf(s) < 1e15f)) return kGone;
    const float fk = floorf(s);
    float x = __fsub_rn(s, fk);
    int64_t k = static_cast<int64_t>(fk);
    if (x >= 1.0f) { x = 0.0f; k += 1; }
    xl = x;
    return apply_walls<float>(I, cell + k, xl, u, refl);
}
__device__ __forceinline__ int64_t transport_full(const InstDev &I, int64_t cell, double &xl, double &u, bool &refl)
{
    return transport(I, cell, xl, u, refl);
}

// Everything but a move to the same or a neighbouring cell inside the domain: wall reflections,
// periodic wraps, particles that leave the domain or move two or more cells.  The particle is
// transported from its original state with the boundary conditions; particles that move two or
// more cells or leave take their pre-transport moments out of the cell (a far mover is appended to
// the far list), a reflected particle's normal momentum changes sign (+2 u after the reflection).
// Returns the class: 0 one cell left, 1 stays, 2 one cell right, 3 farther, 4 left the domain.
template <typename Rec>
__device__ __forceinline__ int stream_rare(const EngineDev &E, int g, int k, Rec &v, long long *a, StreamState &st)
{
    using T = decltype(Rec().xl);
    const CellHdr &h = E.hdr[g];
    const InstDev &I = E.inst[h.b];
    const int ci = h.i;
    const T u0 = v.u;
    bool refl = false;
    const int64_t d = transport_full(I, ci, v.xl, v.u, refl);
    int c;
    if (d == kGone) c = 4;
    else if (d == ci) c = 1;
    else if (d == ci - 1) c = 0;
    else if (d == ci + 1) c = 2;
    else c = 3;
    if (refl || c >= 3) {
        st.range_ok = st.range_ok && fx_in_range(u0) && fx_in_range(v.v) && fx_in_range(v.w);
        if (c >= 3) {
            ++st.ngone;
            a[0] -= fx_vel(u0);
            a[32] -= fx_vel(v.v);
            a[64] -= fx_vel(v.w);
            a[96] -= fx_energy(u0, v.v, v.w);
        } else {
            a[0] += fx_vel(v.u) - fx_vel(u0);
        }
        if (c == 3) {
            const int slot = atomicAdd(&E.far_count[0], 1);
            if (slot < E.far_cap) {
                FarItem<Rec> it;
                it.dest = I.cell_base + 1 + static_cast<int>(d);
                it.src = g;
                it.q = k;
                it.pad = 0;
                it.rec = v;
                static_cast<FarItem<Rec> *>(E.far_app)[slot] = it;
            } else {
                set_err(E.err, kErrOverflow);
            }
        }
    }
    return c;
}

// Common path of the transport: c in {0, 1, 2} for the same or a neighbouring cell inside the
// cells [lo, lo + width) (the domain, and the phantom cell beyond an end that faces another part of
// a split domain); 4 for a particle of an inflow/outflow reservoir (ci = -1 or C) that stays outside
// the domain on the reservoir's side (discarded: a reservoir keeps only what enters, and its own
// moment sums are not used); -1 for everything else (general path).
__device__ __forceinline__ int move_near(float dtdx, int C, int lo, int width, int ci, float &xl, float u)
{
    const float s = __fmaf_rn(u, dtdx, xl);
    if (!(fabsf(s) < 1073741824.0f)) return -1;
    const float fk = floorf(s);
    float x = __fsub_rn(s, fk);
    int k = __float2int_rz(fk);                  // |fk| <= 2^30: exact
    if (x >= 1.0f) { x = 0.0f; k += 1; }
    const unsigned dd = static_cast<unsigned>(k + 1);
    const int d = ci + k;                        // |ci| <= 2^30, |k| <= 2^30: no overflow
    if (dd >= 3u || static_cast<unsigned>(d - lo) >= static_cast<unsigned>(width)) {
        if ((d < 0 && ci < 0) || (d >= C && ci >= C)) return 4;
        return -1;
    }
    xl = x;
    return static_cast<int>(dd);
}
// FP64 records: of the transport only the fused multiply-add and one addition use the double-precision
// pipe (a warp instruction holds it for 64 cycles); floor, comparisons and conversions are integer
// operations, and so are the fixed-point conversions of the run sums.  With them on that pipe (6 and
// 16 instructions per record and per mover) the pipe, not HBM, set the kernel's time: 1595 -> 1051 us
// (0.59 -> 0.90 of the copy bandwidth) on 1e8 particles in 1e5 cells.
__device__ __forceinline__ int move_near(double dtdx, int C, int lo, int width, int ci, double &xl, double u)
{
    const double s = __fma_rn(u, dtdx, xl);
    double x;
    int k;
    if (!dbl_floor_near(s, x, k)) {
        if (!(fabs(s) < 1073741824.0)) return -1;
        const double fk = floor(s);
        x = __dsub_rn(s, fk);
        k = __double2int_rz(fk);
        if (x >= 1.0) { x = 0.0; k += 1; }
    }
    const unsigned dd = static_cast<unsigned>(k + 1);
    const int d = ci + k;
    if (dd >= 3u || static_cast<unsigned>(d - lo) >= static_cast<unsigned>(width)) {
        if ((d < 0 && ci < 0) || (d >= C && ci >= C)) return 4;
        return -1;
    }
    xl = x;
    return static_cast<int>(dd);
}

// Moment sums of the L run (pL, nL) and the R run (pR, nR) of a block, read back together: the runs
// are taken as one list, two records per thread in flight per iteration (the threads first, first + stride, ...
// share it).
template <typename Rec>
__device__ __forceinline__ void run_sums_lr(const Rec *pL, int nL, const Rec *pR, int nR, int first, int stride,
                                            long long sL[4], long long sR[4], bool &ok)
{
    const int n = nL + nR;
    for (int j = first; j < n; j += 2 * stride) {
        const int j2 = j + stride;
        const Rec a = ld_rec_rw(j < nL ? pL + j : pR + (j - nL));
        Rec b = a;
        if (j2 < n) b = ld_rec_rw(j2 < nL ? pL + j2 : pR + (j2 - nL));
        const long long fa[4] = {fx_vel(a.u), fx_vel(a.v), fx_vel(a.w), fx_energy(a.u, a.v, a.w)};
        ok = ok && fx_in_range(a.u) && fx_in_range(a.v) && fx_in_range(a.w);
        const bool aL = j < nL;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sL[k] += aL ? fa[k] : 0;
            sR[k] += aL ? 0 : fa[k];
        }
        if (j2 < n) {
            const long long fb[4] = {fx_vel(b.u), fx_vel(b.v), fx_vel(b.w), fx_energy(b.u, b.v, b.w)};
            ok = ok && fx_in_range(b.u) && fx_in_range(b.v) && fx_in_range(b.w);
            const bool bL = j2 < nL;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                sL[k] += bL ? fb[k] : 0;
                sR[k] += bL ? 0 : fb[k];
            }
        }
    }
}

// Warp sum of a 64-bit integer whose lane values stay below 2^62 in magnitude: three 32-bit
// reductions of its 21-bit limbs (the limb sums of 32 lanes fit in 32 bits).
__device__ __forceinline__ long long warp_sum_ll(long long x)
{
    const unsigned a0 = static_cast<unsigned>(x) & 0x1fffffu;
    const unsigned a1 = static_cast<unsigned>(x >> 21) & 0x1fffffu;
    const int a2 = static_cast<int>(x >> 42);
    const unsigned s0 = __reduce_add_sync(0xffffffffu, a0);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, a1);
    const int s2 = __reduce_add_sync(0xffffffffu, a2);
    return static_cast<long long>(s2) * (1LL << 42) + static_cast<long long>(s1) * (1LL << 21) + static_cast<long long>(s0);
}

// Outputs of a cell that streams nothing (skipped, or in error).
__device__ __forceinline__ void stream_cell_empty(const EngineDev &E, int g, int wp)
{
    const int lane = threadIdx.x & 31;
    if (lane < 4) { E.AL[4 * g + lane] = 0; E.AR[4 * g + lane] = 0; }
    if (lane < 5) E.Aself[5 * g + lane] = 0;
    if (lane == 0) {
        E.nL[wp][g] = 0; E.nS[wp][g] = 0; E.nR[wp][g] = 0; E.slotsb[wp][g] = 0;
        E.ncand[g] = 0; E.nacc[g] = 0; E.nabs[g] = 0; E.nnew[g] = 0;
    }
}


// kMinBlocks: 512-thread blocks per SM the register budget allows; kStreamGroups: groups of 32 records
// each lane loads before any of them is processed (loads in flight per warp).  Both are launch knobs
// of the autotuner; results do not depend on them.
// kMasked: the pool may have masked cells, whose absorbed particles are skipped.
template <typename Rec, int kMinBlocks, int kStreamGroups, bool kMasked>
__global__ void __launch_bounds__(512, kMinBlocks) k_stream(EngineDev E, int rp)
{
    wait_predecessor();
    using T = decltype(Rec().xl);
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int g = blockIdx.x * (blockDim.x >> 5) + warp;
    if (g >= E.G_run) return;
    if (E.order) g = E.order[g];
    StreamShared<Rec> &SS = reinterpret_cast<StreamShared<Rec> *>(s_raw)[warp];
    const int wp = 1 - rp;
    const CellHdr *hp = E.hdr + g;
    const int cls = hp->cls;
    int n_tot = 0;
    const bool masked = kMasked && cls == kClsMasked;
    if (masked || cls == kClsStaged) n_tot = hp->n_in - E.nabs[g] + E.nnew[g];
    else if (cls != kClsSkip) n_tot = hp->n_in + hp->n_new;
    const int slots = hp->slots;
    if (cls == kClsSkip || n_tot > slots) {
        if (cls != kClsSkip && lane == 0) set_err(E.err, kErrOverflow);
        stream_cell_empty(E, g, wp);
        return;
    }
    Rec *blk = static_cast<Rec *>(E.buf[wp]) + hp->off;
    // pieces of the list, in list order
    if (lane == 0) {
        const Rec *in = static_cast<const Rec *>(E.buf[rp]);
        const FarItem<Rec> *fs = static_cast<const FarItem<Rec> *>(E.far_sorted);
        if (cls == kClsStaged) {
            for (int q = 0; q < 5; ++q) SS.piece[q] = Piece<Rec>{blk, 0, 0, 1, 1};
            SS.piece[5] = Piece<Rec>{blk, n_tot, 0, 1, 1};
        } else {
            int k = 0;
            SS.piece[0] = Piece<Rec>{fs + hp->fb, hp->nfb, k, 1, 2};
            k += hp->nfb;
            SS.piece[1] = Piece<Rec>{in + (hp->Rend - 1), hp->Rn, k, -1, 0};
            k += hp->Rn;
            SS.piece[2] = Piece<Rec>{in + hp->Sa, hp->Sn, k, 1, 0};
            k += hp->Sn;
            SS.piece[3] = Piece<Rec>{in + hp->La, hp->Ln, k, 1, 0};
            k += hp->Ln;
            SS.piece[4] = Piece<Rec>{fs + hp->fb + hp->nfb, hp->nfa, k, 1, 2};
            k += hp->nfa;
            // re-sampled particles, drawn by the collision kernels after the arrived positions (masked: after
            // the survivors; the stayers written so far lie below the read position)
            const int run = masked ? k - E.nabs[g] : k;
            SS.piece[5] = Piece<Rec>{blk + run, n_tot - run, k, 1, 1};
        }
    }
    long long *acc = &SS.acc[0][lane];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[32 * j] = 0;
    __syncwarp();
    T dtdx;
    if constexpr (sizeof(T) == 4) dtdx = hp->dtdx_f;
    else dtdx = E.inst[hp->b].dtdx;
    const int C = hp->C, ci = hp->i;
    const int lo = -(hp->edges & 1), width = C + (hp->edges & 1) + ((hp->edges >> 1) & 1);
    const unsigned lt = (1u << lane) - 1u;
    StreamState st;
    st.oS = 0;
    st.oL = slots;
    st.oR = 2 * slots - 1;
    st.ngone = 0;
    st.range_ok = true;
    // The list, iteration by iteration (32 x groups positions of one piece each): the records of
    // the iteration kStreamStages - 1 ahead are copied into the warp's ring asynchronously while the
    // current one is transported, so the loads' latency is not waited for.
    StreamRing<Rec, kStreamGroups> &RG =
        reinterpret_cast<StreamRing<Rec, kStreamGroups> *>(s_raw + (blockDim.x >> 5) * sizeof(StreamShared<Rec>))[warp];
    constexpr int kIt = 32 * kStreamGroups;
    int qp = 0, bp = 0, sp = 0;                  // producer: piece, offset, stage
    while (qp < 6 && SS.piece[qp].n == 0) ++qp;
    int qc = qp, bc = 0, sc = 0;                 // consumer
    auto issue = [&]() {
        if (qp < 6) {
            const Piece<Rec> pc = SS.piece[qp];
#pragma unroll
            for (int u2 = 0; u2 < kStreamGroups; ++u2) {
                const int r = bp + 32 * u2 + lane;
                if (r < pc.n) {
                    const Rec *src = piece_rec(pc, r);
                    Rec *dst = &RG.rec[sp][32 * u2 + lane];
#pragma unroll
                    for (int h = 0; h < static_cast<int>(sizeof(Rec) / 16); ++h)
                        cp_async16(reinterpret_cast<char *>(dst) + 16 * h, reinterpret_cast<const char *>(src) + 16 * h);
                }
            }
            bp += kIt;
            if (bp >= pc.n) {
                bp = 0;
                do { ++qp; } while (qp < 6 && SS.piece[qp].n == 0);
            }
        }
        cp_async_commit();                        // (an empty group past the end keeps the count aligned)
        sp = (sp + 1 == kStreamStages) ? 0 : sp + 1;
    };
#pragma unroll
    for (int s0 = 0; s0 < kStreamStages - 1; ++s0) issue();
    const uint32_t *mask = masked ? survivor_mask(E, g, hp->off) : nullptr;
    while (qc < 6) {
        issue();
        cp_async_wait<kStreamStages - 1>();       // this iteration's copies (each lane reads its own)
        const int n = SS.piece[qc].n, k0 = SS.piece[qc].k0;
        const int base = bc;
#pragma unroll
        for (int u2 = 0; u2 < kStreamGroups; ++u2) {
            const int r = base + 32 * u2 + lane;
            if (base + 32 * u2 >= n) break;
            Rec v;
            int c = 5;
            bool here = r < n;
            uint32_t bits = 0xffffffffu;         // (loaded beside the record, tested after the transport)
            if (kMasked && mask && here && qc < 5) bits = mask[(k0 + r) >> 5];
            if (here) {
                v = RG.rec[sc][32 * u2 + lane];
                c = move_near(dtdx, C, lo, width, ci, v.xl, v.u);
                if (kMasked && !((bits >> ((k0 + r) & 31)) & 1u)) c = 5;
                if (c < 0) c = stream_rare<Rec>(E, g, k0 + r, v, acc, st);
            }
            const unsigned mL = __ballot_sync(0xffffffffu, c == 0);
            const unsigned mS = __ballot_sync(0xffffffffu, c == 1);
            const unsigned mR = __ballot_sync(0xffffffffu, c == 2);
            const unsigned m = (c == 0) ? mL : ((c == 1) ? mS : mR);
            const int rk = __popc(m & lt);
            const int o = (c == 0) ? st.oL + rk : ((c == 1) ? st.oS + rk : st.oR - rk);
            if (c < 3) st_rec(blk + o, v);
            st.oS += __popc(mS);
            st.oL += __popc(mL);
            st.oR -= __popc(mR);
        }
        bc += kIt;
        if (bc >= n) {
            bc = 0;
            do { ++qc; } while (qc < 6 && SS.piece[qc].n == 0);
        }
        sc = (sc + 1 == kStreamStages) ? 0 : sc + 1;
    }
    cp_async_wait<0>();
    __syncwarp();
    // moments of the L and R runs, read back with every lane busy
    const int nLr = st.oL - slots;
    const int nRr = 2 * slots - 1 - st.oR;
    long long sL[4] = {0, 0, 0, 0}, sR[4] = {0, 0, 0, 0};
    bool ok = st.range_ok;
    run_sums_lr<Rec>(blk + slots, nLr, blk + st.oR + 1, nRr, lane, 32, sL, sR, ok);
    if (!__all_sync(0xffffffffu, ok) && lane == 0) set_err(E.err, kErrOverflow);
    long long lj = 0, rj = 0, gj = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const long long a = warp_sum_ll(sL[j]), b = warp_sum_ll(sR[j]), c = warp_sum_ll(acc[32 * j]);
        if (lane == j) { lj = a; rj = b; gj = c; }
    }
    const int ngone = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(st.ngone));
    if (lane < 4) {
        E.AL[4 * g + lane] = lj;
        E.AR[4 * g + lane] = rj;
        E.Aself[5 * g + 1 + lane] = gj - lj - rj;
    }
    if (lane == 0) {
        E.Aself[5 * g] = -static_cast<int64_t>(ngone + nLr + nRr);
        E.nS[wp][g] = st.oS;
        E.nL[wp][g] = nLr;
        E.nR[wp][g] = nRr;
        E.slotsb[wp][g] = slots;
        if (!masked && cls != kClsStaged) {
            if (cls != kClsDirect) { E.ncand[g] = 0; E.nacc[g] = 0; }
            E.nabs[g] = 0;
            E.nnew[g] = hp->n_new;
        }
        if (cls != kClsReservoir) atomicAdd(&E.inst[hp->b].updates, static_cast<unsigned long long>(n_tot));
    }
}

// Streaming with a block of kW warps per cell: the same runs and sums as k_stream, for pools too small to
// fill the GPU with one warp per cell, where a warp's walk through its list (a memory latency per
// iteration) is the kernel's time.  The list is taken in chunks of kR records per thread, loaded at
// once; position base + u T + t belongs to thread t, so the order is (u, warp, lane).  Each warp's
// class counts of every u go to shared memory, one barrier, and a warp scan gives every (u, warp) its
// place in the runs.  A staged list (in the first half of the output block) is overwritten by its
// stayers only at positions of this and earlier chunks, whose records all threads hold after the
// barrier.
template <typename Rec, int kW, int kR>
__global__ void __launch_bounds__(32 * kW) k_stream_block(EngineDev E, int rp)
{
    wait_predecessor();
    using T = decltype(Rec().xl);
    constexpr int kT = 32 * kW, kE = kR * kW;
    static_assert(kE <= 32 && kE * 32 < 1024, "one warp scans the counts, 10 bits per class");
    __shared__ uint32_t s_cnt[2][kE];
    __shared__ long long s_acc[kW][4][32];
    __shared__ unsigned long long s_sum[12];
    __shared__ int s_gone, s_bad;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int g = blockIdx.x;
    const int wp = 1 - rp;
    const CellHdr h = E.hdr[g];
    const int cls = h.cls;
    int n_tot = 0;
    int n_arr = h.n_in, run = h.n_in;    // arrived positions, and those of them in the list (masked: the survivors)
    if (cls == kClsStaged || cls == kClsMasked) {
        run = h.n_in - E.nabs[g];
        n_tot = run + E.nnew[g];
        if (cls == kClsStaged) { n_arr = 0; run = 0; }        // the whole list in the output block
    } else if (cls != kClsSkip) {
        n_tot = h.n_in + h.n_new;
    }
    const int slots = h.slots;
    if (cls == kClsSkip || n_tot > slots) {
        if (cls != kClsSkip && t == 0) set_err(E.err, kErrOverflow);
        if (t < 32) stream_cell_empty(E, g, wp);
        return;
    }
    Rec *blk = static_cast<Rec *>(E.buf[wp]) + h.off;
    Rec *in = static_cast<Rec *>(E.buf[rp]);
    FarItem<Rec> *fs = static_cast<FarItem<Rec> *>(E.far_sorted);
    const int n_pos = n_arr + (n_tot - run);               // positions to walk: arrived, then from blk + run on
    const uint32_t *mask = cls == kClsMasked ? survivor_mask(E, g, h.off) : nullptr;
    T dtdx;
    if constexpr (sizeof(T) == 4) dtdx = h.dtdx_f;
    else dtdx = E.inst[h.b].dtdx;
    const int C = h.C, ci = h.i;
    const int lo = -(h.edges & 1), width = C + (h.edges & 1) + ((h.edges >> 1) & 1);
    const unsigned lt = (1u << lane) - 1u;
    long long *acc = &s_acc[warp][0][lane];
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[32 * j] = 0;
    if (t < 12) s_sum[t] = 0ull;
    if (t == 0) { s_gone = 0; s_bad = 0; }
    StreamState st;
    st.oS = 0;
    st.oL = slots;
    st.oR = 2 * slots - 1;
    st.ngone = 0;
    st.range_ok = true;
    int par = 0;
    for (int base = 0; base < n_pos; base += kR * kT, par ^= 1) {
        Rec v[kR];
        int c[kR];
#pragma unroll
        for (int u = 0; u < kR; ++u) {
            const int k = base + u * kT + t;
            c[u] = 5;
            if (k < n_pos) {
                c[u] = (mask && k < n_arr && !((mask[k >> 5] >> (k & 31)) & 1u)) ? 5 : 0;
                v[u] = ld_rec_l2(k >= n_arr ? blk + run + (k - n_arr) : arrived_ptr<Rec>(k, h, in, fs));
            }
        }
        unsigned mine = 0;                                  // lane u: the warp's counts of u
#pragma unroll
        for (int u = 0; u < kR; ++u) {
            const int k = base + u * kT + t;
            if (c[u] == 0) {
                c[u] = move_near(dtdx, C, lo, width, ci, v[u].xl, v[u].u);
                if (c[u] < 0) c[u] = stream_rare<Rec>(E, g, k, v[u], acc, st);
            }
            const unsigned n = __popc(__ballot_sync(0xffffffffu, c[u] == 0)) |
                               __popc(__ballot_sync(0xffffffffu, c[u] == 1)) << 10 |
                               __popc(__ballot_sync(0xffffffffu, c[u] == 2)) << 20;
            if (lane == u) mine = n;
        }
        if (lane < kR) s_cnt[par][lane * kW + warp] = mine;
        __syncthreads();
        unsigned x = lane < kE ? s_cnt[par][lane] : 0u;     // inclusive scan over (u, warp)
        const unsigned own = x;
#pragma unroll
        for (int o = 1; o < kE; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const unsigned tot = __shfl_sync(0xffffffffu, x, kE - 1), pre = x - own;
#pragma unroll
        for (int u = 0; u < kR; ++u) {
            const unsigned p = __shfl_sync(0xffffffffu, pre, u * kW + warp);
            const unsigned mL = __ballot_sync(0xffffffffu, c[u] == 0);
            const unsigned mS = __ballot_sync(0xffffffffu, c[u] == 1);
            const unsigned mR = __ballot_sync(0xffffffffu, c[u] == 2);
            const unsigned m = (c[u] == 0) ? mL : ((c[u] == 1) ? mS : mR);
            const int rk = __popc(m & lt);
            const int o = (c[u] == 0)   ? st.oL + static_cast<int>(p & 1023u) + rk
                          : (c[u] == 1) ? st.oS + static_cast<int>((p >> 10) & 1023u) + rk
                                        : st.oR - static_cast<int>(p >> 20) - rk;
            if (c[u] < 3) st_rec(blk + o, v[u]);
        }
        st.oL += static_cast<int>(tot & 1023u);
        st.oS += static_cast<int>((tot >> 10) & 1023u);
        st.oR -= static_cast<int>(tot >> 20);
    }
    __syncthreads();                                        // (the runs are read back below)
    const int nLr = st.oL - slots;
    const int nRr = 2 * slots - 1 - st.oR;
    long long sL[4] = {0, 0, 0, 0}, sR[4] = {0, 0, 0, 0};
    bool ok = st.range_ok;
    run_sums_lr<Rec>(blk + slots, nLr, blk + st.oR + 1, nRr, t, kT, sL, sR, ok);
    const bool rare = st.ngone != 0 || acc[0] != 0;         // (a far mover or leaver, or a reflection)
    if (__any_sync(0xffffffffu, rare)) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long a = warp_sum_ll(acc[32 * j]);
            if (lane == 0) atomicAdd(&s_sum[8 + j], static_cast<unsigned long long>(a));
        }
        const int n = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(st.ngone));
        if (lane == 0) atomicAdd(&s_gone, n);
    }
    if (32 * warp < nLr + nRr) {                            // (the other warps had no record to sum)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const long long a = warp_sum_ll(sL[j]), b = warp_sum_ll(sR[j]);
            if (lane == 0) {
                atomicAdd(&s_sum[j], static_cast<unsigned long long>(a));
                atomicAdd(&s_sum[4 + j], static_cast<unsigned long long>(b));
            }
        }
    }
    if (!ok) s_bad = 1;
    __syncthreads();
    if (t < 4) {
        const long long lj = static_cast<long long>(s_sum[t]), rj = static_cast<long long>(s_sum[4 + t]);
        E.AL[4 * g + t] = lj;
        E.AR[4 * g + t] = rj;
        E.Aself[5 * g + 1 + t] = static_cast<long long>(s_sum[8 + t]) - lj - rj;
    }
    if (t == 0) {
        if (s_bad) set_err(E.err, kErrOverflow);
        E.Aself[5 * g] = -static_cast<int64_t>(s_gone + nLr + nRr);
        E.nS[wp][g] = st.oS;
        E.nL[wp][g] = nLr;
        E.nR[wp][g] = nRr;
        E.slotsb[wp][g] = slots;
        if (cls != kClsStaged && cls != kClsMasked) {
            if (cls != kClsDirect) { E.ncand[g] = 0; E.nacc[g] = 0; }
            E.nabs[g] = 0;
            E.nnew[g] = h.n_new;
        }
        if (cls != kClsReservoir) atomicAdd(&E.inst[h.b].updates, static_cast<unsigned long long>(n_tot));
    }
}

// ------------------------------------------------------------------------------------------
// Far movers: rank sort by (dest, src, q) -- keys are unique.
// ------------------------------------------------------------------------------------------
template <typename Rec>
__global__ void k_far_sort(EngineDev E)
{
    wait_predecessor();
    const FarItem<Rec> *a = static_cast<const FarItem<Rec> *>(E.far_app);
    FarItem<Rec> *s = static_cast<FarItem<Rec> *>(E.far_sorted);
    int n = *(volatile int32_t *)&E.far_count[0];
    if (n > E.far_cap) n = E.far_cap;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) E.far_count[1] = n;
    if (t >= n) return;
    const FarItem<Rec> me = a[t];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
        const FarItem<Rec> &o = a[j];
        const bool less = (o.dest < me.dest) || (o.dest == me.dest && (o.src < me.src || (o.src == me.src && o.q < me.q)));
        rank += less ? 1 : 0;
    }
    s[rank] = me;
}

// s = a + b as 64-bit integers; false when the sum overflows.
__device__ __forceinline__ bool add_no_overflow(long long a, long long b, long long &s)
{
    s = static_cast<long long>(static_cast<unsigned long long>(a) + static_cast<unsigned long long>(b));
    return ((a ^ s) & (b ^ s)) >= 0;
}

// ------------------------------------------------------------------------------------------
// Cell kernel: Eq. (r1) update, time average, primitive state, P, slot bound and plan of the next
// step.  For P = 0 the re-sampled count and the NTC candidate count depend only on cell data and
// counters, so they are decided here, one thread per cell, instead of inside the particle kernels.
// ------------------------------------------------------------------------------------------
template <typename Rec, int B>
__global__ void __launch_bounds__(B) k_cells(EngineDev E, int q, int update)
{
    wait_predecessor();
    __shared__ int64_t s_w[B / 32];
    const int g = blockIdx.x * B + threadIdx.x;
    int64_t myslots = 0;
    if (B == kCellBlockMin && g > 0 && g + 1 < E.G_run) {
        // small pools (one warp per SM): what the cell reads, asked for at once instead of in the order of
        // use, half a dozen L2 latencies one after the other
        prefetch_l1(E.far_count + 1);
        prefetch_l1(E.off[q] + g);
        prefetch_l1(E.slotsb[q] + g);
        prefetch_l1(E.nR[q] + g - 1);
        prefetch_l1(E.nS[q] + g);
        prefetch_l1(E.nL[q] + g + 1);
        prefetch_l1(E.AR + 4 * (g - 1));
        prefetch_l1(E.AL + 4 * (g + 1));
        prefetch_l1(E.Aself + 5 * g);
        prefetch_l1(E.psi + 5 * g);
        prefetch_l1(E.psi + 5 * g + 4);
        prefetch_l1(E.flux + 5 * (g - 1));
        prefetch_l1(E.flux + 5 * g + 4);
        prefetch_l1(E.avg + 5 * g);
        prefetch_l1(E.avg + 5 * g + 4);
        prefetch_l1(E.cmax + g);
        prefetch_l1(E.fmaj + g);
    }
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        if (update) E.far_count[0] = 0;
        for (int q = 0; q < kLists; ++q) E.ticket[kListLen + q] = 0;
        E.ticket[kSampleLen] = 0;
        E.ticket[kPreLen] = 0;
        E.ticket[kRoundLen] = 0;
        E.ticket[kLongLen] = 0;
    }
    if (g < E.G_run) {
        CellHdr hd;
        hd.Rend = hd.Sa = hd.La = hd.off = 0;
        hd.Rn = hd.Sn = hd.Ln = hd.slots = 0;
        hd.fb = hd.nfb = hd.nfa = 0;
        hd.n_in = hd.n_new = hd.nc = 0;
        hd.cls = kClsSkip;
        hd.b = -1;
        hd.i = 0;
        hd.C = 0;
        hd.dtdx_f = 0.0f;
        hd.edges = 0;
        const int b = E.cell_inst[g];
        if (b >= 0) {
            const InstDev &I = E.inst[b];
            const int i = g - I.cell_base - 1;
            const uint32_t step_next = I.step + (update ? 1u : 0u);
            hd.b = b;
            hd.i = i;
            hd.C = I.C;
            hd.dtdx_f = I.dtdx_f;
            hd.edges = (I.bc_left == kBcPhantom ? 1 : 0) | (I.bc_right == kBcPhantom ? 2 : 0);
            if (i < 0 || i >= I.C) {
                const int side = (i < 0) ? 0 : 1;
                const int bc = side ? I.bc_right : I.bc_left;
                if (bc == 0) {
                    double qg[5];
                    const bool ok = ghost_prim(I, side, qg, false, qg);
                    const double Pg = split_fraction(I, qg, ok);
                    myslots = ok ? resample_count(I, cell_id(I, i), step_next, Pg, qg[0]) : 0;
                    for (int k = 0; k < 5; ++k) E.prim[5 * g + k] = qg[k];
                    E.valid[g] = ok ? 1 : 0;
                    E.P[g] = Pg;
                    hd.cls = kClsReservoir;
                    hd.n_new = static_cast<int32_t>(myslots);
                }
                E.cnt[g] = 0;
            } else {
                // particles arriving in g and the sums of what they carry
                int farn = 0, lo = 0, mid = 0;
                double fsum[4] = {0, 0, 0, 0};
                const int nf = E.far_count[1];
                if (nf > 0) {
                    const FarItem<Rec> *fs = static_cast<const FarItem<Rec> *>(E.far_sorted);
                    lo = far_lower(fs, nf, g, INT32_MIN);
                    mid = far_lower(fs, nf, g, g + 1);
                    const int hi = far_lower(fs, nf, g + 1, INT32_MIN);
                    farn = hi - lo;
                    for (int k = lo; k < hi; ++k) {
                        const double u = fs[k].rec.u, v = fs[k].rec.v, w = fs[k].rec.w;
                        fsum[0] += u; fsum[1] += v; fsum[2] += w; fsum[3] += 0.5 * (u * u + v * v + w * w);
                    }
                    hd.fb = lo;
                    hd.nfb = mid - lo;
                    hd.nfa = hi - mid;
                }
                hd.Rend = E.off[q][g - 1] + 2 * static_cast<int64_t>(E.slotsb[q][g - 1]);
                hd.Rn = E.nR[q][g - 1];
                hd.Sa = E.off[q][g];
                hd.Sn = E.nS[q][g];
                hd.La = E.off[q][g + 1] + E.slotsb[q][g + 1];
                hd.Ln = E.nL[q][g + 1];
                const int arrivals = hd.Rn + hd.Sn + hd.Ln + farn;
                double *psi = E.psi + 5 * g;
                if (update) {
                    const int64_t *aR = E.AR + 4 * (g - 1), *aL = E.AL + 4 * (g + 1), *aS = E.Aself + 5 * g;
                    double dp[5];
                    // the three runs' fixed-point sums added as integers and converted once (unless the
                    // sum would overflow)
                    // (conversions by integer operations; the far movers' sums added only where there
                    // are any, the wave fluxes only where one is nonzero: x + 0 and x - 0 are x)
                    dp[0] = fixed_to_double(static_cast<int64_t>(hd.Rn + hd.Ln + farn) + aS[0], 0);
                    for (int k = 0; k < 4; ++k) {
                        const int fr = (k == 3) ? 32 : 40;
                        long long s1, s2;
                        if (add_no_overflow(aR[k], aL[k], s1) && add_no_overflow(s1, aS[k + 1], s2)) {
                            dp[k + 1] = fixed_to_double(s2, fr);
                            if (farn > 0) dp[k + 1] = dp[k + 1] + fsum[k];
                        } else {
                            dp[k + 1] = fixed_to_double(aR[k], fr) + fixed_to_double(aL[k], fr) + fsum[k] +
                                        fixed_to_double(aS[k + 1], fr);
                        }
                    }
                    const double *Fl = E.flux + 5 * (g - 1), *Fr = E.flux + 5 * g;
                    bool zero_flux = true;
                    for (int k = 0; k < 5; ++k) zero_flux = zero_flux && dbl_is_zero(Fl[k]) && dbl_is_zero(Fr[k]);
                    for (int k = 0; k < 5; ++k) {
                        const double fp = I.mp_over_dx * dp[k];
                        if (zero_flux) {
                            psi[k] = psi[k] + fp;
                        } else {
                            const double fw = I.dtdx * (Fr[k] - Fl[k]);
                            psi[k] = psi[k] + fp - fw;
                        }
                    }
                    if (static_cast<int64_t>(step_next) > static_cast<int64_t>(I.avg_start)) {
                        for (int k = 0; k < 5; ++k) E.avg[5 * g + k] += psi[k];
                    }
                }
                double qq[5];
                const bool ok = prim_from_cons(psi, I.inv_cv, qq);
                for (int k = 0; k < 5; ++k) E.prim[5 * g + k] = qq[k];
                E.valid[g] = ok ? 1 : 0;
                const double P = split_fraction(I, qq, ok);
                E.P[g] = P;
                int64_t extra = 0;
                if (ok) {
                    if (dbl_is_zero(P)) {
                        extra = resample_count(I, cell_id(I, i), step_next, 0.0,
                                               psi[0] - fixed_to_double(arrivals, 0) * I.mp_over_dx);
                    } else {
                        extra = static_cast<int64_t>(floor(((1.0 - P) * fmax(psi[0], 0.0)) * I.dx_over_mp)) + 2;
                    }
                }
                E.cnt[g] = arrivals;
                myslots = arrivals + extra;
                hd.n_in = arrivals;
                if (dbl_gt(P, 0.0)) {
                    hd.cls = kClsStaged;
                } else {
                    const int64_t n_tot = arrivals + extra;
                    const int64_t nc = ntc_candidates(I, cell_id(I, i), step_next,
                                                      static_cast<int>(n_tot), psi[0], E.cmax[g], E.fmaj[g]);
                    hd.n_new = static_cast<int32_t>(extra);
                    if (nc < 0 || n_tot > INT32_MAX) {
                        set_err(E.err, kErrOverflow);
                        hd.cls = kClsSkip;
                    } else {
                        hd.nc = static_cast<int32_t>(nc);
                        hd.cls = (nc == 0) ? kClsStream : kClsDirect;
                    }
                }
            }
        }
        if (myslots > INT32_MAX / 2) {
            set_err(E.err, kErrOverflow);
            myslots = 0;
            hd.cls = kClsSkip;
        }
        hd.slots = static_cast<int32_t>(myslots);
        E.slots[g] = static_cast<int32_t>(myslots);
        E.hdr[g] = hd;
    }
    // block sum of the slot bounds
    int64_t x = myslots;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t s = 0;
        for (int w = 0; w < B / 32; ++w) s += s_w[w];
        E.blocksum[blockIdx.x] = 2 * s;
    }
}

// ------------------------------------------------------------------------------------------
// Offsets of the next step's output blocks, the collision kernel's work list, and the wave flux of
// every interface.  With 256-cell blocks (large pools) at 64 registers (a full SM of warps): the
// double-precision flux, which spills there, runs only where P_f > 0, and the offsets and lists
// before it are latency-bound.  Smaller blocks (small pools, one or two blocks per SM) take up to
// 128 registers and keep the flux's double-precision chain out of local memory.
// ------------------------------------------------------------------------------------------
// Whether a cell's collisions are long dependency chains, which the block kernel runs in parallel
// rounds: at least heavy_min NTC candidates (Appendix A), for a staged cell on a list that fits the block's
// shared-memory table.  (On longer lists the pairs rarely share a particle and the collision kernel's
// warp takes them 32 at a time.)  A staged cell is estimated with about (1 - P) of its mass in
// particles after absorption and re-sampling.  Only the choice of kernel depends on this, never a
// result.
// Returns the estimated candidate count, 0 where the block kernel does not take the cell.
__device__ __forceinline__ int staged_heavy(const EngineDev &E, int g)
{
    const InstDev &I = E.inst[E.hdr[g].b];
    const double rho_t = E.psi[5 * g];
    const double n_est = (1.0 - E.P[g]) * fmax(rho_t, 0.0) * I.dx_over_mp;
    if (!(n_est <= 0.9 * kBlockSlots)) return 0;
    const double rr = (I.ntc_rate == 1) ? rho_t * I.inv_rho_ref : n_est * I.ntc_rr;
    const double nsel = I.ntc_A * rr * (n_est - 1.0) * E.fmaj[g] * E.cmax[g];
    return nsel >= static_cast<double>(E.heavy_min) ? static_cast<int>(fmin(nsel, 1e6)) : 0;
}

// Chunks of cell g appended to a sample list (lanes of a warp together: one atomic per warp).
__device__ __forceinline__ void append_chunks(const EngineDev &E, int2 *list, int len_ticket, int g, int chunks, int lane)
{
    int incl = chunks;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (total > 0) {
        int base = 0;
        if (lane == 0) base = atomicAdd(&E.ticket[len_ticket], total);
        base = __shfl_sync(0xffffffffu, base, 0);
        const int first = base + incl - chunks;
        for (int c = 0; c < chunks; ++c) {
            if (first + c < E.wls_cap) list[first + c] = make_int2(g, c * kSampleChunk);
            else set_err(E.err, kErrOverflow);
        }
    }
}

// Wave flux of the interface after cell g (between local cells i and i+1; -1: the left end), and
// the instance's step counter advanced once per step.
__device__ __forceinline__ void interface_flux(const EngineDev &E, int g)
{
    if (g >= E.G_run) return;
    const int b = E.cell_inst[g];
    if (b < 0) return;
    InstDev &I = E.inst[b];
    const int i = g - I.cell_base - 1;   // interface between local cells i and i+1
    if (i >= I.C) return;
    const int gl = (i < 0) ? -1 : g, gr = (i + 1 >= I.C) ? -1 : g + 1;
    double a[5], c[5];
    bool aok, cok;
    const bool periodic = (I.bc_left == 2);
    if (gl >= 0) { for (int k = 0; k < 5; ++k) a[k] = E.prim[5 * gl + k]; aok = E.valid[gl] != 0; }
    if (gr >= 0) { for (int k = 0; k < 5; ++k) c[k] = E.prim[5 * gr + k]; cok = E.valid[gr] != 0; }
    if (gl < 0) {
        if (periodic) {
            const int gg = I.cell_base + I.C;
            for (int k = 0; k < 5; ++k) a[k] = E.prim[5 * gg + k];
            aok = E.valid[gg] != 0;
        } else if (I.bc_left == kBcPhantom) {
            // the neighbouring part's edge cell, copied into the phantom cell g
            for (int k = 0; k < 5; ++k) a[k] = E.prim[5 * g + k];
            aok = E.valid[g] != 0;
        } else {
            aok = ghost_prim(I, 0, c, cok, a);
        }
    }
    if (gr < 0) {
        if (periodic) {
            const int gg = I.cell_base + 1;
            for (int k = 0; k < 5; ++k) c[k] = E.prim[5 * gg + k];
            cok = E.valid[gg] != 0;
        } else if (I.bc_right == kBcPhantom) {
            for (int k = 0; k < 5; ++k) c[k] = E.prim[5 * (g + 1) + k];
            cok = E.valid[g + 1] != 0;
        } else {
            cok = ghost_prim(I, 1, a, aok, c);
        }
    }
    if (I.recon_mode == 1) {
        // the states beyond a and c, as the flux sees them, and whether a and c have slopes
        const bool use0 = periodic || i >= 0, use1 = periodic || i + 1 < I.C;
        const int g0 = I.cell_base + 1;            // local cell 0
        double wm[5] = {0, 0, 0, 0, 0}, w2[5] = {0, 0, 0, 0, 0};
        bool okm = false, ok2 = false;
        if (use0) {
            const int j = i - 1;
            if (j >= 0 || periodic) {
                const int gj = g0 + ((j + I.C) % I.C);
                for (int k = 0; k < 5; ++k) wm[k] = E.prim[5 * gj + k];
                okm = E.valid[gj] != 0;
            } else {
                okm = ghost_prim(I, 0, E.prim + 5 * g0, E.valid[g0] != 0, wm);
            }
        }
        if (use1) {
            const int j = i + 2;
            if (j < I.C || periodic) {
                const int gj = g0 + (j % I.C);
                for (int k = 0; k < 5; ++k) w2[k] = E.prim[5 * gj + k];
                ok2 = E.valid[gj] != 0;
            } else {
                const int gl2 = g0 + I.C - 1;
                ok2 = ghost_prim(I, 1, E.prim + 5 * gl2, E.valid[gl2] != 0, w2);
            }
        }
        double aR[5], cR[5];
        recon_pair(wm, okm, a, aok, c, cok, w2, ok2, use0, use1, aR, cR);
        wave_flux(I, aR, aok, cR, cok, E.flux + 5 * g, a, c);
    } else {
        wave_flux(I, a, aok, c, cok, E.flux + 5 * g, a, c);
    }
}

// End of a step: the instance's step counter (and the count of averaged states) advance, once per
// instance (by the thread of its left reservoir cell).
__device__ __forceinline__ void step_advance(const EngineDev &E, int g)
{
    if (g >= E.G_run) return;
    const int b = E.cell_inst[g];
    if (b < 0) return;
    InstDev &I = E.inst[b];
    if (g - I.cell_base - 1 != -1) return;
    const uint32_t nxt = I.step + 1u;
    if (static_cast<int64_t>(nxt) > static_cast<int64_t>(I.avg_start)) I.navg += 1;
    I.step = nxt;
}

template <int B>
__global__ void __launch_bounds__(B, (B < 256) ? 512 / B : 1024 / B) k_offsets(EngineDev E, int wp, int advance,
                                                                                 int per)
{
    wait_predecessor();
    __shared__ int64_t s_w[B / 32];
    __shared__ int64_t s_pre;
    const int g = blockIdx.x * B + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // sum of the slot bounds of all earlier blocks (the cell kernel's block sums, `per` of its
    // blocks to one of these)
    int64_t acc = 0;
    if (B == kCellBlockMin && g < E.G_run) {               // (as in the cell kernel)
        prefetch_l1(E.slots + g);
        prefetch_l1(E.hdr + g);
        prefetch_l1(&E.hdr[g].nc);
        prefetch_l1(E.psi + 5 * g);
        prefetch_l1(E.P + g);
        prefetch_l1(E.cmax + g);
        prefetch_l1(E.fmaj + g);
    }
    for (int j = threadIdx.x; j < blockIdx.x * per; j += B) acc += E.blocksum[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) s_w[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t s = 0;
        for (int w = 0; w < B / 32; ++w) s += s_w[w];
        s_pre = s;
    }
    __syncthreads();
    // exclusive scan of the slots inside the block
    const int64_t v = (g < E.G_run) ? 2 * static_cast<int64_t>(E.slots[g]) : 0;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    int64_t wpre = 0;
    for (int w = 0; w < warp; ++w) wpre += s_w[w];
    bool listed = false;
    int lq = kWarpList;   // work list (kLightList: direct cells with up to kMaxDirect candidates and
                          // nothing re-sampled; kHeavyList: the cells with many candidates)
    int chunks = 0, pchunks = 0;
    bool longest = false;                      // in the heavy list's front part
    if (g < E.G_run) {
        const int64_t o = s_pre + wpre + x - v;
        E.off[wp][g] = o;
        E.hdr[g].off = o;
        if (o + v > E.capacity) {
            set_err(E.err, kErrOverflow);
            E.hdr[g].cls = kClsSkip;
        } else {
            const int cls = E.hdr[g].cls;
            listed = (cls == kClsDirect) || (cls == kClsStaged);
            if (cls == kClsStaged) {
                const int nc = staged_heavy(E, g);
                if (nc > 0) lq = kHeavyList;
                longest = nc >= kLongCandidates;
            }
            if (cls == kClsDirect) {
                const int nc = E.hdr[g].nc;
                if (nc >= E.heavy_min) lq = kHeavyList;
                else if (light_resampling(E.hdr[g]) && nc <= kMaxDirect) lq = kLightList;
                longest = lq == kHeavyList && nc >= kLongCandidates;
            }
            const bool many = E.hdr[g].n_new >= kPreSampleMin;
            // the few re-sampled particles of cells without collisions, and every reservoir's, are
            // drawn in the collision kernel's tail (beside the collisions)
            if (cls == kClsReservoir || (cls == kClsStream && !many))
                chunks = (E.hdr[g].n_new + kSampleChunk - 1) / kSampleChunk;
            if ((cls == kClsDirect || cls == kClsStream) && many && lq != kHeavyList) {
                // many particles to draw (all of them in a first step): drawn ahead over the whole
                // GPU instead of by the one warp that collides the cell.  (The block kernel's cells
                // draw their own: that kernel then depends on nothing of the sampling kernel and
                // starts beside it.)
                pchunks = (E.hdr[g].n_new + kSampleChunk - 1) / kSampleChunk;
                if (cls == kClsDirect) E.hdr[g].edges |= kEdgePresampled;
            }
        }
    }
    // sample lists (one atomic per warp): chunk c of cell g starts at particle c * kSampleChunk
    append_chunks(E, E.wls, kSampleLen, g, chunks, lane);
    append_chunks(E, E.wlp, kPreLen, g, pchunks, lane);
    // work lists of the collision kernels (one atomic per warp and list)
    int light_base = 0;
#pragma unroll
    for (int q = 0; q < kLists; ++q) {
        const bool mine = listed && lq == q && !longest;
        const unsigned lm = __ballot_sync(0xffffffffu, mine);
        if (lm) {
            int base = 0;
            if (lane == __ffs(lm) - 1) base = atomicAdd(&E.ticket[kListLen + q], __popc(lm));
            base = __shfl_sync(0xffffffffu, base, __ffs(lm) - 1);
            const int pos = base + __popc(lm & ((1u << lane) - 1u));
            if (mine) E.wl[q == kWarpList ? E.G - 1 - pos : static_cast<size_t>(q) * E.G + pos] = g;
            if (q == kLightList) {
                light_base = base;
                if (mine) E.wlnc[pos] = E.hdr[g].nc;
            }
        }
    }
    {
        const bool mine = listed && longest;
        const unsigned lm = __ballot_sync(0xffffffffu, mine);
        if (lm) {
            int base = 0;
            if (lane == __ffs(lm) - 1) base = atomicAdd(&E.ticket[kLongLen], __popc(lm));
            base = __shfl_sync(0xffffffffu, base, __ffs(lm) - 1);
            const int pos = base + __popc(lm & ((1u << lane) - 1u));
            if (mine) E.wl[static_cast<size_t>(kHeavyList) * E.G + (E.G - 1 - pos)] = g;
        }
    }
    if (g == 0) {
        for (int q = 0; q < kLists; ++q) E.ticket[q] = 0;
        E.ticket[kSampleCtr] = 0;
        E.ticket[kPreCtr] = 0;
        E.ticket[kRoundCtr] = 0;
        E.ticket[kAbsorbCtr] = 0;
    }
    if (advance) step_advance(E, g);
    // this warp's light cells (consecutive in the light list), packed into rounds by k_sample
    {
        const unsigned lm = __ballot_sync(0xffffffffu, listed && lq == kLightList);
        if (lane == 0 && g < E.G) E.wgrp[g >> 5] = make_int2(lm ? light_base : 0, __popc(lm));
    }
}

// Wave flux at every interface (Sec. 3.3) from the primitive states of the cell kernel: run at the
// start of the step that applies it (by the cell kernel), on a side stream beside that step's
// collision and streaming kernels, which neither read the flux nor write the states it reads.
template <int B>
__global__ void __launch_bounds__(B, (B < 256) ? 512 / B : 1024 / B) k_flux(EngineDev E)
{
    wait_predecessor();
    interface_flux(E, blockIdx.x * B + threadIdx.x);
}

// ------------------------------------------------------------------------------------------
// Initial cells of one instance: all wave (Psi_p = 0), Psi_t from the two-state profile.
// ------------------------------------------------------------------------------------------
// Initial state of cell g = g0 + t of instance b (all wave, no particles; the left or right state by
// the cell centre's side of x_split).
__device__ __forceinline__ void init_cell(const EngineDev &E, int b, int g, const double *lc, const double *rc,
                                          double x_min, double x_split)
{
    const InstDev &I = E.inst[b];
    E.cell_inst[g] = b;
    const int i = g - I.cell_base - 1;
    for (int p = 0; p < 2; ++p) { E.nL[p][g] = 0; E.nS[p][g] = 0; E.nR[p][g] = 0; E.off[p][g] = 0; E.slotsb[p][g] = 0; }
    for (int k = 0; k < 4; ++k) { E.AL[4 * g + k] = 0; E.AR[4 * g + k] = 0; }
    for (int k = 0; k < 5; ++k) { E.Aself[5 * g + k] = 0; E.avg[5 * g + k] = 0.0; E.flux[5 * g + k] = 0.0; E.psi[5 * g + k] = 0.0; E.prim[5 * g + k] = 0.0; }
    E.ncand[g] = 0; E.nacc[g] = 0; E.nabs[g] = 0; E.nnew[g] = 0; E.cnt[g] = 0; E.slots[g] = 0; E.valid[g] = 0; E.P[g] = 0.0; E.cmax[g] = 0.0; E.fmaj[g] = 1.0;
    if (i < 0 || i >= I.C) return;
    const double xc = x_min + (static_cast<double>(I.id0 + i) + 0.5) * I.dx;
    const bool left = xc < x_split;
    for (int k = 0; k < 5; ++k) E.psi[5 * g + k] = left ? lc[k] : rc[k];
    const double T = left ? I.left[4] : I.right[4];
    E.cmax[g] = 5.0 * sqrt(2.0 * I.R * T);
    E.fmaj[g] = majorant_factor(I, E.cmax[g]);
}

__global__ void k_init_cells(EngineDev E, int b, int g0, int n, double l0, double l1, double l2, double l3, double l4,
                             double r0, double r1, double r2, double r3, double r4, double x_min, double x_split)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double lc[5] = {l0, l1, l2, l3, l4}, rc[5] = {r0, r1, r2, r3, r4};
    init_cell(E, b, g0 + t, lc, rc, x_min, x_split);
}

struct InitCellsBatch {
    InitCellsItem it[kInitBatch];
};

// blockIdx.y: the item (instance); blockIdx.x: cells of that instance
__global__ void k_init_cells_batch(EngineDev E, const __grid_constant__ InitCellsBatch B, int n_items)
{
    const int j = blockIdx.y;
    if (j >= n_items) return;
    const InitCellsItem &q = B.it[j];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= q.n) return;
    init_cell(E, q.b, q.g0 + t, q.lc, q.rc, q.x_min, q.x_split);
}

// ------------------------------------------------------------------------------------------
// Gather of the stable sorted list of instance b (inspection).
// ------------------------------------------------------------------------------------------
// (the values in double precision by integer operations: as conversions, 4 per particle at 64 cycles per
// warp instruction of the double-precision pipe, they took as long as the kernel's traffic)
template <typename Rec>
__global__ void k_gather(EngineDev E, int rp, int g0, int ncell, const int64_t *start, int64_t total, const int64_t *gate,
                         int32_t *cell, double *xl, double *u, double *v, double *w)
{
    const int t = blockIdx.x;
    if (t >= ncell) return;
    if (gate && *gate != total) return;     // the count differs from the caller's size: write nothing
    const int g = g0 + t;
    const Rec *in = static_cast<const Rec *>(E.buf[rp]);
    const FarItem<Rec> *fs = static_cast<const FarItem<Rec> *>(E.far_sorted);
    const int nf = E.far_count[1];
    int lo = 0, mid = 0, hi = 0;
    if (nf > 0) {
        lo = far_lower(fs, nf, g, INT32_MIN);
        mid = far_lower(fs, nf, g, g + 1);
        hi = far_lower(fs, nf, g + 1, INT32_MIN);
    }
    const int64_t Rend = E.off[rp][g - 1] + 2 * static_cast<int64_t>(E.slotsb[rp][g - 1]);
    const int Rn = E.nR[rp][g - 1];
    const int64_t Sa = E.off[rp][g];
    const int Sn = E.nS[rp][g];
    const int64_t La = E.off[rp][g + 1] + E.slotsb[rp][g + 1];
    const int Ln = E.nL[rp][g + 1];
    const int nfb = mid - lo, nfa = hi - mid;
    const int n = nfb + Rn + Sn + Ln + nfa;
    const int64_t o = start[t];
    const int local = g - E.inst[E.cell_inst[g]].cell_base - 1;
    if (o + n > total) {
        if (threadIdx.x == 0) set_err(E.err, kErrOverflow);
        return;
    }
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        int r = k;
        Rec x;
        if (r < nfb) x = fs[lo + r].rec;
        else if ((r -= nfb) < Rn) x = in[Rend - 1 - r];
        else if ((r -= Rn) < Sn) x = in[Sa + r];
        else if ((r -= Sn) < Ln) x = in[La + r];
        else { r -= Ln; x = fs[mid + r].rec; }
        __stcs(cell + o + k, local);
        __stcs(xl + o + k, dbl_of(x.xl));
        __stcs(u + o + k, dbl_of(x.u));
        __stcs(v + o + k, dbl_of(x.v));
        __stcs(w + o + k, dbl_of(x.w));
    }
}

// ------------------------------------------------------------------------------------------
// Normal stress Pi = S_xx and heat flux Q = Q_x of interior cells (Eq. gkt_moment1; inspection,
// not part of the step): the particle part from the central moments of the arrived particles about
// the total velocity U_t,
//   S_p = (m_p/dx) sum (xi_x - U)^2 - rho_p R T_t,   Q_p = (m_p/dx) sum (xi_x - U) |xi - U|^2 / 2,
// rho_p = n m_p / dx; the wave part its NS stress and heat flux (the values of the Chapman-Enskog
// re-sampling: neighbour states as the wave flux sees them, mu_e = eps mu) weighted by
// rho_w / rho_t.  A cell whose total state is not usable reports 0.
// Three passes: one thread per cell splits -U into float pairs; one warp per cell sums its particles
// (single-precision records in double-single arithmetic: the double-precision units are a small
// fraction of the single-precision ones); one thread per cell finishes in double precision.
// ------------------------------------------------------------------------------------------
struct ShCell {
    float nu[6];      // -U, -V, -W as double-single pairs
    double s[2];      // sum (xi_x - U)^2, sum (xi_x - U) |xi - U|^2 / 2 (as (hi, lo) floats for FP32 records)
};

__device__ __forceinline__ bool sh_interior(const EngineDev &E, int g, int &b, int &i)
{
    b = E.cell_inst[g];
    if (b < 0) return false;
    i = g - E.inst[b].cell_base - 1;
    return i >= 0 && i < E.inst[b].C;
}

__global__ void k_sh_split(EngineDev E, int g0, int ncell, ShCell *tmp)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ncell) return;
    const int g = g0 + t;
    int b, i;
    if (!sh_interior(E, g, b, i) || !E.valid[g]) return;
    for (int d = 0; d < 3; ++d) {
        const ds x = ds_neg(ds_of_double(E.prim[5 * static_cast<int64_t>(g) + 1 + d]));
        tmp[g].nu[2 * d] = x.hi;
        tmp[g].nu[2 * d + 1] = x.lo;
    }
}

template <typename Rec>
__global__ void k_sh_sums(EngineDev E, int rp, int g0, int ncell, ShCell *tmp)
{
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= ncell) return;
    const int g = (E.order && g0 == 0 && ncell == E.G_run) ? E.order[t] : g0 + t;
    int b, i;
    if (!sh_interior(E, g, b, i) || !E.valid[g]) return;
    Rec *in = static_cast<Rec *>(E.buf[rp]);
    FarItem<Rec> *fs = static_cast<FarItem<Rec> *>(E.far_sorted);
    const CellHdr h = E.hdr[g];
    const int n = h.n_in;
    constexpr int kIn = 4;   // records per lane in flight
    if constexpr (sizeof(Rec().u) == 4) {
        // single-precision records: c = xi - U formed exactly (TwoSum with the double-single -U) and
        // rounded once, the two terms in single precision, each lane's sums compensated (TwoSum of
        // every addition, the errors summed apart); the arrived runs read as contiguous ranges
        const float v0h = tmp[g].nu[0], v0l = tmp[g].nu[1], v1h = tmp[g].nu[2], v1l = tmp[g].nu[3],
                    v2h = tmp[g].nu[4], v2l = tmp[g].nu[5];
        float s2 = 0.0f, e2 = 0.0f, s3 = 0.0f, e3 = 0.0f;
        auto add = [&](const Rec &r) {
            const ds ax = ds_two_sum(r.u, v0h), ay = ds_two_sum(r.v, v1h), az = ds_two_sum(r.w, v2h);
            const float cx = ax.hi + (ax.lo + v0l), cy = ay.hi + (ay.lo + v1l), cz = az.hi + (az.lo + v2l);
            const float xx = cx * cx;
            const float c2 = fmaf(cz, cz, fmaf(cy, cy, xx));
            const float t3 = (0.5f * cx) * c2;
            const ds a2 = ds_two_sum(s2, xx), a3 = ds_two_sum(s3, t3);
            s2 = a2.hi;
            e2 += a2.lo;
            s3 = a3.hi;
            e3 += a3.lo;
        };
        auto range = [&](const Rec *p, int cnt) {
            for (int k0 = lane; k0 < cnt; k0 += 32 * kIn) {
                Rec x[kIn];
#pragma unroll
                for (int u = 0; u < kIn; ++u)
                    if (k0 + 32 * u < cnt) x[u] = ld_rec(p + k0 + 32 * u);
#pragma unroll
                for (int u = 0; u < kIn; ++u)
                    if (k0 + 32 * u < cnt) add(x[u]);
            }
        };
        range(in + (h.Rend - h.Rn), h.Rn);
        range(in + h.Sa, h.Sn);
        range(in + h.La, h.Ln);
        for (int k = lane; k < h.nfb + h.nfa; k += 32) add(fs[h.fb + k].rec);
        ds f2 = ds_two_sum(s2, e2), f3 = ds_two_sum(s3, e3);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            f2 = ds_add(f2, {__shfl_xor_sync(0xffffffffu, f2.hi, o), __shfl_xor_sync(0xffffffffu, f2.lo, o)});
            f3 = ds_add(f3, {__shfl_xor_sync(0xffffffffu, f3.hi, o), __shfl_xor_sync(0xffffffffu, f3.lo, o)});
        }
        if (lane == 0) {
            float *o = reinterpret_cast<float *>(tmp[g].s);
            o[0] = f2.hi; o[1] = f2.lo; o[2] = f3.hi; o[3] = f3.lo;
        }
    } else {
        const double *W0 = E.prim + 5 * static_cast<int64_t>(g);
        const double U = W0[1], V = W0[2], Wz = W0[3];
        double s2 = 0.0, s3 = 0.0;
        for (int k0 = lane; k0 < n; k0 += 32 * kIn) {
            Rec x[kIn];
#pragma unroll
            for (int u = 0; u < kIn; ++u) {
                const int r = k0 + 32 * u;
                if (r >= n) break;
                x[u] = ld_rec(arrived_ptr<Rec>(r, h, in, fs));
            }
#pragma unroll
            for (int u = 0; u < kIn; ++u) {
                if (k0 + 32 * u >= n) break;
                const double cx = x[u].u - U, cy = x[u].v - V, cz = x[u].w - Wz;
                s2 += cx * cx;
                s3 += cx * (0.5 * (cx * cx + cy * cy + cz * cz));
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            s3 += __shfl_xor_sync(0xffffffffu, s3, o);
        }
        if (lane == 0) { tmp[g].s[0] = s2; tmp[g].s[1] = s3; }
    }
}

__global__ void k_sh_finish(EngineDev E, int fp32, int g0, int ncell, const ShCell *tmp, int accumulate, double *out)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ncell) return;
    const int g = g0 + t;
    int b, i;
    if (!sh_interior(E, g, b, i)) return;
    double pi = 0.0, q = 0.0;
    if (E.valid[g]) {
        const InstDev &I = E.inst[b];
        double s2, s3;
        if (fp32) {
            const float *o = reinterpret_cast<const float *>(tmp[g].s);
            s2 = static_cast<double>(o[0]) + static_cast<double>(o[1]);
            s3 = static_cast<double>(o[2]) + static_cast<double>(o[3]);
        } else {
            s2 = tmp[g].s[0];
            s3 = tmp[g].s[1];
        }
        const double rho_p = static_cast<double>(E.hdr[g].n_in) * I.mp_over_dx;
        pi = I.mp_over_dx * s2 - rho_p * I.R * E.prim[5 * static_cast<int64_t>(g) + 4];
        q = I.mp_over_dx * s3;
        CeCell m;
        ce_coefs(I, E.prim, E.valid, g, i, m);   // sets the stress and heat flux of a usable cell
        const double rho_t = E.psi[5 * static_cast<int64_t>(g)];
        const double wgt = (rho_t - rho_p) / rho_t;
        pi += wgt * m.sxx;
        q += wgt * m.qx;
    }
    if (accumulate) {
        out[g] += pi;
        out[E.G + g] += q;
    } else {
        out[g] = pi;
        out[E.G + g] = q;
    }
}

// ------------------------------------------------------------------------------------------
// Macroscopic profiles of all instances in one pass (inspection): out = [rho | u | T | wave
// fraction] x total, instance b's interior cell i at base[b] + i (base[b] < 0: not reported).
// ------------------------------------------------------------------------------------------
__global__ void k_moments(EngineDev E, int which, const int64_t *base, int64_t total, double *out)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= E.G) return;
    const int b = E.cell_inst[g];
    if (b < 0 || base[b] < 0) return;
    const InstDev &I = E.inst[b];
    const int i = g - I.cell_base - 1;
    if (i < 0 || i >= I.C) return;
    const int64_t o = base[b] + i;
    if (o >= total) return;
    const double *c = (which == 1 ? E.avg : E.psi) + 5 * static_cast<int64_t>(g);
    const int64_t navg = I.navg;
    const double scale = (which == 1) ? (navg > 0 ? 1.0 / static_cast<double>(navg) : 0.0) : 1.0;
    // one reciprocal per density instead of five divisions (each double-precision instruction holds
    // an SM sub-partition for 64 cycles on this GPU); the read-out, not a decision of the method
    const double r = c[0] * scale;
    const double mx = c[1] * scale, my = c[2] * scale, mz = c[3] * scale, e5 = c[4] * scale;
    const double ir = r > 0 ? 1.0 / r : 0.0;
    const double ux = mx * ir, uy = my * ir, uz = mz * ir;
    const double tt = r > 0 ? (e5 * ir - 0.5 * (ux * ux + uy * uy + uz * uz)) * I.inv_cv : 0.0;
    const double rt = E.psi[5 * static_cast<int64_t>(g)];
    const double irt = (which == 1) ? (rt > 0 ? 1.0 / rt : 0.0) : ir;
    out[o] = r;
    out[total + o] = ux;
    out[2 * total + o] = tt;
    out[3 * total + o] = rt > 0 ? 1.0 - (static_cast<double>(E.cnt[g]) * I.mp_over_dx) * irt : 0.0;
}

// ------------------------------------------------------------------------------------------
// Launchers
// ------------------------------------------------------------------------------------------
size_t stream_smem_bytes(int fp32, int threads, int groups)
{
    const size_t ring = (groups == 3) ? (fp32 ? sizeof(StreamRing<RecF, 3>) : sizeof(StreamRing<RecD, 3>))
                                      : (fp32 ? sizeof(StreamRing<RecF, 2>) : sizeof(StreamRing<RecD, 2>));
    return static_cast<size_t>(threads / 32) * ((fp32 ? sizeof(StreamShared<RecF>) : sizeof(StreamShared<RecD>)) + ring);
}
size_t stress_tmp_bytes() { return sizeof(ShCell); }
size_t collide_smem_bytes(int fp32)
{
    return (fp32 ? sizeof(CollideShared<RecF>) : sizeof(CollideShared<RecD>)) * (kCollideThreads / 32);
}
int collide_threads() { return kCollideThreads; }

// Sets the kernel's dynamic shared-memory limit to smem_max (the largest any launch shape uses, so
// that engines with different shapes can coexist) and returns blocks per SM at `threads`, `smem`.
template <typename K>
static int occupancy_of(K kern, int threads, size_t smem, size_t smem_max)
{
    int n = 0;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem_max));
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

// The streaming kernel for a register budget (variant 0/1/2: 1/2/3 blocks of 512 threads per SM) and
// 2 or 3 record groups per lane.
template <typename Rec, bool kMasked>
static void (*stream_kernel_m(int variant, int groups))(EngineDev, int)
{
    if (groups == 3) {
        if (variant == 2) return k_stream<Rec, 3, 3, kMasked>;
        if (variant == 1) return k_stream<Rec, 2, 3, kMasked>;
        return k_stream<Rec, 1, 3, kMasked>;
    }
    if (variant == 2) return k_stream<Rec, 3, 2, kMasked>;
    if (variant == 1) return k_stream<Rec, 2, 2, kMasked>;
    return k_stream<Rec, 1, 2, kMasked>;
}
template <typename Rec>
static void (*stream_kernel(int variant, int groups, int masked))(EngineDev, int)
{
    return masked ? stream_kernel_m<Rec, true>(variant, groups) : stream_kernel_m<Rec, false>(variant, groups);
}

// The streaming kernel with a block of 2, 4 or 8 warps per cell.
template <typename Rec>
static void (*stream_block_kernel(int warps))(EngineDev, int)
{
    if (warps == 8) return k_stream_block<Rec, 8, 3>;
    if (warps == 4) return k_stream_block<Rec, 4, 4>;
    return k_stream_block<Rec, 2, 4>;
}

// Warps per cell of the streaming kernel for a pool of `cells` cells with about `particles` particles, at
// most about `longest` of them in a cell: the smallest sum of the longest list's walk (a memory latency
// per iteration of a warp, shared by the cell's warps) and of the whole pool's work, which several warps
// per cell make dearer (counts exchanged through shared memory).  Coefficients in ns per record of the
// longest list, per particle and per cell, fitted to Mach-8 shocks of 60 to 15000 cells with 60 and 415
// particles per upstream cell, 26 pools in each precision (profiles/launch_rules.md): the choice is 1.3%
// slower than the best on average, 14% at worst.  (100 cells, FP64 records: 24.5 us with a warp per cell,
// 8.2 us with eight; 1000 cells, FP32: 13.8 and 8.0 us with four; FP32 pools of 6000 cells of 1000 particles
// are the fastest with one warp per cell.)
int stream_warps(int fp32, int64_t cells, double particles, double longest)
{
    static const int w[4] = {1, 2, 4, 8};
    static const double walk[2][4] = {{34.0, 21.5, 15.4, 12.3}, {25.6, 17.6, 12.5, 9.7}};
    static const double work[2][4] = {{0.0105, 0.0120, 0.0131, 0.0197}, {0.0055, 0.0073, 0.0086, 0.0123}};
    static const double cell[4] = {0.9, 1.2, 2.1, 4.5};
    int best = 0;
    double tb = 0.0;
    for (int k = 0; k < 4; ++k) {
        double t = walk[fp32 ? 1 : 0][k] * longest + work[fp32 ? 1 : 0][k] * particles + cell[k] * static_cast<double>(cells);
        if (k == 0) t *= 0.9;      // (its walk and work overlap best)
        if (k == 0 || t < tb) {
            best = k;
            tb = t;
        }
    }
    return w[best];
}

int stream_occupancy(int fp32, int variant, int groups, int threads)
{
    // the limit: the largest shape's shared memory, within what a block may opt in to
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const size_t smem = stream_smem_bytes(fp32, threads, groups);
    if (smem > static_cast<size_t>(optin)) return 0;
    const size_t mx = std::min(stream_smem_bytes(fp32, 512, 3), static_cast<size_t>(optin));
    int n = 0;
    for (int masked = 0; masked < 2; ++masked)
        n = fp32 ? occupancy_of(stream_kernel<RecF>(variant, groups, masked), threads, smem, mx)
                 : occupancy_of(stream_kernel<RecD>(variant, groups, masked), threads, smem, mx);
    return n;
}

size_t staged_smem_bytes(int fp32)
{
    return fp32 ? sizeof(BlockShared<RecF>) : sizeof(BlockShared<RecD>);
}

// The block kernel at five blocks per SM (96 registers) or, wide, four (128 registers, fewer spills).
int staged_occupancy(int fp32, int wide)
{
    const size_t smem = staged_smem_bytes(fp32);
    if (wide)
        return fp32 ? occupancy_of(k_cellblock<RecF, 4>, kBlockThreads, smem, smem)
                    : occupancy_of(k_cellblock<RecD, 4>, kBlockThreads, smem, smem);
    return fp32 ? occupancy_of(k_cellblock<RecF, 5>, kBlockThreads, smem, smem)
                : occupancy_of(k_cellblock<RecD, 5>, kBlockThreads, smem, smem);
}

int sample_occupancy(int fp32)
{
    return fp32 ? occupancy_of(k_sample<RecF>, kSampleThreads, 0, 0) : occupancy_of(k_sample<RecD>, kSampleThreads, 0, 0);
}

template <typename Rec>
static void (*collide_kernel(int masked))(EngineDev, int)
{
    return masked ? k_collide<Rec, true> : k_collide<Rec, false>;
}

int collide_occupancy(int fp32)
{
    const size_t smem = collide_smem_bytes(fp32);
    int n = 0;
    for (int masked = 0; masked < 2; ++masked)
        n = fp32 ? occupancy_of(collide_kernel<RecF>(masked), kCollideThreads, smem, smem)
                 : occupancy_of(collide_kernel<RecD>(masked), kCollideThreads, smem, smem);
    return n;
}

namespace {
// Launch with a scheduling priority (blocks of higher-priority launches are dispatched first) and
// programmatic stream serialization (see wait_predecessor).
template <typename... Args>
cudaError_t launch_prio(void (*kernel)(Args...), int grid, int threads, size_t smem, cudaStream_t s, int prio,
                        Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributePriority;
    attr[0].val.priority = prio;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
}  // namespace


// Launch with programmatic stream serialization (see wait_predecessor).
template <typename... Args>
static cudaError_t launch_pdl(void (*kernel)(Args...), dim3 grid, int threads, cudaStream_t s, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
cudaError_t launch_sample(const EngineDev &E, int fp32, int rp, int grid, cudaStream_t s, int prio)
{
    const cudaError_t e = fp32 ? launch_prio(k_sample<RecF>, grid, kSampleThreads, 0, s, prio, E, rp)
                               : launch_prio(k_sample<RecD>, grid, kSampleThreads, 0, s, prio, E, rp);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_absorb(const EngineDev &E, int fp32, int rp, int grid, cudaStream_t s, int prio)
{
    const cudaError_t e = fp32 ? launch_prio(k_absorb<RecF>, grid, kSampleThreads, 0, s, prio, E, rp)
                               : launch_prio(k_absorb<RecD>, grid, kSampleThreads, 0, s, prio, E, rp);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_collide(const EngineDev &E, int fp32, int masked, int rp, int grid, cudaStream_t s, int prio)
{
    const size_t smem = collide_smem_bytes(fp32);
    cudaError_t e = fp32 ? launch_prio(collide_kernel<RecF>(masked), grid, kCollideThreads, smem, s, prio, E, rp)
                         : launch_prio(collide_kernel<RecD>(masked), grid, kCollideThreads, smem, s, prio, E, rp);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_staged(const EngineDev &E, int fp32, int wide, int rp, int grid, cudaStream_t s, int prio)
{
    const size_t smem = staged_smem_bytes(fp32);
    cudaError_t e;
    if (wide)
        e = fp32 ? launch_prio(k_cellblock<RecF, 4>, grid, kBlockThreads, smem, s, prio, E, rp)
                 : launch_prio(k_cellblock<RecD, 4>, grid, kBlockThreads, smem, s, prio, E, rp);
    else
        e = fp32 ? launch_prio(k_cellblock<RecF, 5>, grid, kBlockThreads, smem, s, prio, E, rp)
                 : launch_prio(k_cellblock<RecD, 5>, grid, kBlockThreads, smem, s, prio, E, rp);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_stream(const EngineDev &E, int fp32, int variant, int groups, int masked, int rp, int threads,
                          int warps, cudaStream_t s, int prio)
{
    if (warps > 1) {
        const cudaError_t eb = fp32 ? launch_prio(stream_block_kernel<RecF>(warps), E.G_run, 32 * warps, 0, s, prio, E, rp)
                                    : launch_prio(stream_block_kernel<RecD>(warps), E.G_run, 32 * warps, 0, s, prio, E, rp);
        return eb != cudaSuccess ? eb : cudaGetLastError();
    }
    const int wpb = threads / 32;
    const int grid = (E.G_run + wpb - 1) / wpb;
    const size_t smem = stream_smem_bytes(fp32, threads, groups);
    const cudaError_t e =
        fp32 ? launch_prio(stream_kernel<RecF>(variant, groups, masked), grid, threads, smem, s, prio, E, rp)
             : launch_prio(stream_kernel<RecD>(variant, groups, masked), grid, threads, smem, s, prio, E, rp);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_far_sort(const EngineDev &E, int fp32, cudaStream_t s)
{
    const int grid = (E.far_cap + 255) / 256;
    if (fp32) launch_pdl(k_far_sort<RecF>, dim3(grid), 256, s, E);
    else launch_pdl(k_far_sort<RecD>, dim3(grid), 256, s, E);
    return cudaGetLastError();
}

// Cells per block of the offset and flux kernels (and of the cell kernel on small pools).  Their
// per-cell work is a chain of double-precision operations (primitive state, Eq. (p), the wave flux),
// and an SM's double-precision units are few: a small pool is spread over as many SMs as it can fill
// (two blocks each) instead of a few full blocks.
static int cell_block(int cells, int nsm)
{
    for (int b = kCellBlockMin; b < kCellBlock; b *= 2)
        if (cells <= b * 2 * nsm) return b;
    return kCellBlock;
}

// Cells per block of the cell kernel alone: on a large pool, blocks of kCellBlockLarge instead of
// kCellBlock spread its double-precision chains evenly over the SMs' sub-partitions (all blocks are
// resident at once; with 256-cell blocks some SMs hold a block more than others).  The offset
// kernel keeps its own blocks and reads the cell kernel's block sums in their units.
static int cells_kernel_block(int cells, int nsm)
{
    const int b = cell_block(cells, nsm);
    return b == kCellBlock ? kCellBlockLarge : b;
}

template <typename Rec>
static cudaError_t launch_cells_b(const EngineDev &E, int b, int grid, int q, int update, cudaStream_t s)
{
    if (b == 32) launch_pdl(k_cells<Rec, 32>, dim3(grid), 32, s, E, q, update);
    else if (b == 64) launch_pdl(k_cells<Rec, 64>, dim3(grid), 64, s, E, q, update);
    else if (b == 128) launch_pdl(k_cells<Rec, 128>, dim3(grid), 128, s, E, q, update);
    else launch_pdl(k_cells<Rec, kCellBlock>, dim3(grid), kCellBlock, s, E, q, update);
    return cudaGetLastError();
}

cudaError_t launch_cells(const EngineDev &E, int fp32, int q, int update, cudaStream_t s)
{
    const int b = cells_kernel_block(E.G_run, E.nsm > 0 ? E.nsm : 1);
    const int grid = (E.G_run + b - 1) / b;
    return fp32 ? launch_cells_b<RecF>(E, b, grid, q, update, s) : launch_cells_b<RecD>(E, b, grid, q, update, s);
}

cudaError_t launch_offsets(const EngineDev &E, int wp, int advance, cudaStream_t s)
{
    const int nsm = E.nsm > 0 ? E.nsm : 1;
    const int b = cell_block(E.G_run, nsm);
    const int per = b / cells_kernel_block(E.G_run, nsm);
    const int grid = (E.G_run + b - 1) / b;
    if (b == 32) launch_pdl(k_offsets<32>, dim3(grid), 32, s, E, wp, advance, per);
    else if (b == 64) launch_pdl(k_offsets<64>, dim3(grid), 64, s, E, wp, advance, per);
    else if (b == 128) launch_pdl(k_offsets<128>, dim3(grid), 128, s, E, wp, advance, per);
    else launch_pdl(k_offsets<kCellBlock>, dim3(grid), kCellBlock, s, E, wp, advance, per);
    return cudaGetLastError();
}

cudaError_t launch_flux(const EngineDev &E, cudaStream_t s, int prio)
{
    const int b = cell_block(E.G_run, E.nsm > 0 ? E.nsm : 1);
    const int grid = (E.G_run + b - 1) / b;
    cudaError_t e;
    if (b == 32) e = launch_prio(k_flux<32>, grid, 32, 0, s, prio, E);
    else if (b == 64) e = launch_prio(k_flux<64>, grid, 64, 0, s, prio, E);
    else if (b == 128) e = launch_prio(k_flux<128>, grid, 128, 0, s, prio, E);
    else e = launch_prio(k_flux<kCellBlock>, grid, kCellBlock, 0, s, prio, E);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_stress_heat(const EngineDev &E, int fp32, int rp, int g0, int ncell, int accumulate, double *out,
                               void *tmp, cudaStream_t s)
{
    if (ncell <= 0) return cudaSuccess;
    ShCell *t = static_cast<ShCell *>(tmp);
    const int gt = (ncell + 255) / 256;
    if (fp32) k_sh_split<<<gt, 256, 0, s>>>(E, g0, ncell, t);
    const int gw = (ncell + 3) / 4;   // one warp per cell
    if (fp32) k_sh_sums<RecF><<<gw, 128, 0, s>>>(E, rp, g0, ncell, t);
    else k_sh_sums<RecD><<<gw, 128, 0, s>>>(E, rp, g0, ncell, t);
    k_sh_finish<<<gt, 256, 0, s>>>(E, fp32, g0, ncell, t, accumulate, out);
    return cudaGetLastError();
}

cudaError_t launch_init_turn(cudaStream_t s)
{
    k_init_turn<<<1, (kTurnTable > kLogTable ? kTurnTable : kLogTable), 0, s>>>();
    return cudaGetLastError();
}

cudaError_t launch_init_cells_batch(const EngineDev &E, const InitCellsItem *items, int n_items, cudaStream_t s)
{
    for (int j0 = 0; j0 < n_items; j0 += kInitBatch) {
        const int m = std::min(kInitBatch, n_items - j0);
        InitCellsBatch B;
        int max_n = 0;
        for (int j = 0; j < m; ++j) {
            B.it[j] = items[j0 + j];
            max_n = std::max(max_n, items[j0 + j].n);
        }
        if (max_n <= 0) continue;
        const dim3 grid((max_n + 255) / 256, m);
        k_init_cells_batch<<<grid, 256, 0, s>>>(E, B, m);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// order[start + i] = g0 + i for each item's n cells (one block row per item).
struct OrderBatch {
    OrderItem it[kOrderBatch];
};
__global__ void k_fill_order(int32_t *order, const __grid_constant__ OrderBatch B)
{
    const OrderItem &q = B.it[blockIdx.y];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < q.n) order[q.start + i] = q.g0 + i;
}

cudaError_t launch_fill_order(int32_t *order, const OrderItem *items, int n_items, cudaStream_t s)
{
    for (int j0 = 0; j0 < n_items; j0 += kOrderBatch) {
        const int m = std::min(kOrderBatch, n_items - j0);
        OrderBatch B;
        int max_n = 0;
        for (int j = 0; j < m; ++j) {
            B.it[j] = items[j0 + j];
            max_n = std::max(max_n, items[j0 + j].n);
        }
        if (max_n <= 0) continue;
        k_fill_order<<<dim3((max_n + 255) / 256, m), 256, 0, s>>>(order, B);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// A restored checkpoint's warp list (wl[G], wl[G + 1], ...) to its place on the device (wl[G - 1], wl[G - 2], ...).
__global__ void k_place_warp_list(EngineDev E)
{
    const int n = min(E.ticket[kListLen + kWarpList], E.G);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) E.wl[E.G - 1 - t] = E.wl[E.G + t];
}

cudaError_t launch_place_warp_list(const EngineDev &E, cudaStream_t s)
{
    k_place_warp_list<<<std::min(1024, (E.G + 255) / 256), 256, 0, s>>>(E);
    return cudaGetLastError();
}

cudaError_t launch_init_cells(const EngineDev &E, int b, int g0, int n, const double *lc, const double *rc, double x_min,
                              double x_split, cudaStream_t s)
{
    const int grid = (n + 255) / 256;
    k_init_cells<<<grid, 256, 0, s>>>(E, b, g0, n, lc[0], lc[1], lc[2], lc[3], lc[4], rc[0], rc[1], rc[2], rc[3], rc[4],
                                      x_min, x_split);
    return cudaGetLastError();
}

cudaError_t launch_moments(const EngineDev &E, int which, const int64_t *d_base, int64_t total, double *d_out,
                           cudaStream_t s)
{
    k_moments<<<(E.G + 255) / 256, 256, 0, s>>>(E, which, d_base, total, d_out);
    return cudaGetLastError();
}

cudaError_t launch_gather(const EngineDev &E, int fp32, int rp, int b, int g0, int ncell, const int64_t *d_start,
                          int64_t total, const int64_t *gate, int32_t *cell, double *xl, double *u, double *v,
                          double *w, cudaStream_t s)
{
    (void)b;
    if (ncell <= 0) return cudaSuccess;
    if (fp32) k_gather<RecF><<<ncell, 128, 0, s>>>(E, rp, g0, ncell, d_start, total, gate, cell, xl, u, v, w);
    else k_gather<RecD><<<ncell, 128, 0, s>>>(E, rp, g0, ncell, d_start, total, gate, cell, xl, u, v, w);
    return cudaGetLastError();
}

}  // namespace duwp
