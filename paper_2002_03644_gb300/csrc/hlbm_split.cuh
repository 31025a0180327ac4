// hlbm_split.cuh -- the FP64 time step of Algorithm 1 as two passes of one
// thread per cell, so that no value is computed twice.
//
// GB300's FP64 pipe retires about 1.7 multiply-adds per clock and SM, and
// the FP64 step is bound by the number of FP64 instructions per cell-update,
// not by bytes.  The tiled and the marching kernels recompute the halo of
// every tile or strip, and each cell evaluates its neighbours' limited
// slopes and closure defects again.  Here every such value is computed once
// and stored in a plane (HBM is at a tenth of its rate):
//   level pass    (split_level_kernel)   level n+1 of a cell from level n:
//                 entropy update (eq sequaalgo), pull and moments (eqs streamalgo,
//                 rhoalgo, ualgo), theta (eq Entropie expression), and the cell's
//                 closure defects Gamma_x, Gamma_y (Sec. 3.2);
//   collide pass  (split_collide_kernel)  E1, E2, a1 and the collision (eqs
//                 Psialgo, Equilibrium, a1sigalgo, streamalgo) from level n+1 of
//                 the cell and its neighbours, and for the next level pass the
//                 cell's two Van Albada slopes of s(n+1) and mu / (2 mu + p).
// A face of the MUSCL scheme needs the slopes of the cell and of its upwind
// neighbour only, so two slopes per cell serve what took four per cell, and
// one reciprocal serves omega (eq. streamalgo) and the Phi of the next level
// (eq. viscous heat discret).  That leaves five reciprocals per cell-update
// (1 / (rho theta), 1 / rho, 1 / (2 mu + p) and the slopes' two) instead of
// eight divisions.
//
// Measured on GB300, per step: 1024^2 vortex 369 us (764 on the marching
// kernel), Sod tube 400 x 4 13 us (39 on the tiled kernel).  The level pass
// takes 83 FP64 instructions per cell, the collide pass 92.5; the FP64 pipe is
// busy for 85 and 86 % of their cycles, which is what 19 cycles per warp
// instruction, the most that eight warps of dependent multiply-adds reach,
// come to.
//
// Against the time step in 80-bit arithmetic (13 cases of 700 to 10000 cells,
// all sides but walls, sigma 0 to 0.9): after one step the rms errors of rho,
// u, theta, s and a1 are 0.997 to 1.000 times (geometric mean) those of the
// tiled and the marching kernel with IEEE divisions and CUDA's functions;
// after 10 to 40 steps 0.88 to 1.07 times in every smooth case.
//
// CANON (grids of up to 768^2 cells, whose checkpoints hold the 13 planes of
// the tiled kernel): the cache planes a level pass reads are derived from
// the F and s that the state holds, in the collide pass, so that a run
// resumed from those planes continues bitwise; larger grids carry the four
// cache planes in their checkpoints, and the level pass's own values stay in
// them, which saves the second log and exp per cell-update.
//
// Boundaries are the index maps of the other kernels.  Beyond a Dirichlet
// or zero-gradient side s does not vary along the normal, so the slope there
// is zero, as is that of the zero-gradient side's edge cell.
#pragma once

#include "hlbm_march.cuh"

namespace hlbm {

// Planes that live between the two passes of a step (or from the collide
// pass to the next level pass), [ny][pitch] each; sigma > 0 alone needs the
// second moments.
struct SplitPlanes {
    double *dx, *dy, *mp;      // limited slopes of s, mu / (2 mu + p): collide pass -> next level pass
    double *gx, *gy;           // Gamma_x, Gamma_y of level n+1: level pass -> collide pass
    double *mxx, *myy, *mxy;   // second moments of the pulled populations: level pass -> collide pass
    double *rho, *ux, *uy, *th;  // level n+1: level pass -> collide pass (CANON: not the state's own cache planes)
    // constants of the case that would each cost an FP64 instruction per cell
    double two_mu, m_half_mu, quarter_mu, half_tmg, one_m_sigma;
};
// planes that go from the level pass to the collide pass
constexpr int SPLIT_NHAND = 5, SPLIT_NHAND_CANON = 9;

// x > 0 and x < 0, false for NaN as the comparisons are, on the integer pipe (a
// comparison of doubles takes the FP64 pipe like a multiply-add): the bits of
// the smallest subnormal to infinity, and the same with the sign.
__device__ __forceinline__ bool positive64(double x)
{
    return (unsigned long long)__double_as_longlong(x) - 1 < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool negative64(double x)
{
    return (unsigned long long)__double_as_longlong(x) - 0x8000000000000001ull < 0x7ff0000000000000ull;
}

// rho and momentum of nine populations (moments(), every operation rounded).
// The pairs are mirror images, so that u keeps its small values, and its
// sign, where the flow across an axis nearly vanishes; sums that share
// f5 - f7 and f8 - f6 save two operations, but their rounding errors have the
// size of the mean flow's populations.
__device__ __forceinline__ void moments64(const double f[9], double &rho, double &jx, double &jy)
{
    rho = __dadd_rn(__dadd_rn(__dadd_rn(__dadd_rn(f[0], f[1]), __dadd_rn(f[2], f[3])),
                              __dadd_rn(__dadd_rn(f[4], f[5]), __dadd_rn(f[6], f[7]))), f[8]);
    jx = __dadd_rn(__dadd_rn(__dsub_rn(f[1], f[3]), __dsub_rn(f[5], f[6])), __dsub_rn(f[8], f[7]));
    jy = __dadd_rn(__dadd_rn(__dsub_rn(f[2], f[4]), __dsub_rn(f[5], f[8])), __dsub_rn(f[6], f[7]));
}

// Van Albada slope of the one-sided differences a, b (va_slope).
__device__ __forceinline__ double va_slope64(double a, double b)
{
    const double ab = a * b;
    return positive64(ab) ? quot64(ab * (a + b), fma(a, a, b * b)) : 0.0;
}

// p and 2 mu + p, rounded operation by operation: the collide pass and
// split_prepare_kernel give the same bits, so a resumed run continues bitwise.
__device__ __forceinline__ double pressure64(double rho, double th) { return __dmul_rn(__dmul_rn(rho, th), 1.0 / 3.0); }

// omega = (2 mu - p) / (2 mu + p) (eq. streamalgo) and mu / (2 mu + p), the
// factor of the Phi of the next level (eq. viscous heat discret).
__device__ __forceinline__ void relaxation64(double two_mu, double mu, double p, double &omega, double &mp)
{
    const double b = __dadd_rn(two_mu, p);
    if (rcp64_ok(b)) {
        const double ib = rcp64(b);
        omega = __dmul_rn(two_mu - p, ib);
        mp = __dmul_rn(mu, ib);
    } else {
        omega = (two_mu - p) / b;
        mp = mu / b;
    }
}

// u = j / rho (eq. ualgo)
__device__ __forceinline__ void velocity64(double jx, double jy, double rho, double &ux, double &uy)
{
    if (rcp64_ok(rho)) {
        const double ir = rcp64(rho);
        ux = __dmul_rn(jx, ir);
        uy = __dmul_rn(jy, ir);
    } else {
        ux = jx / rho;
        uy = jy / rho;
    }
}

// rho, u and theta of a cell from the stored F and s.  The sums are rounded
// one by one (never fused with the products that made f), so that values
// taken from registers and from memory give the same bits.
__device__ __forceinline__ void canon_macros64(const Tables64 &tab, const double f[9], double s, const KParams &kp, double &rho,
                                               double &ux, double &uy, double &th)
{
    double jx, jy;
    moments64(f, rho, jx, jy);
    velocity64(jx, jy, rho, ux, uy);
    th = theta64(tab, kp, rho, s);
}

// Offsets of a cell's neighbours (or -(side + 1) on a Dirichlet side).
struct Cross {
    int w, e, s, n;
};
__device__ __forceinline__ Cross cross_of(int x, int y, const KParams &kp)
{
    const int xw = map_col(x - 1, kp), xe = map_col(x + 1, kp), ys = map_row(y - 1, kp), yn = map_row(y + 1, kp);
    return Cross{join_map(y, xw, kp.pitch), join_map(y, xe, kp.pitch), join_map(ys, x, kp.pitch), join_map(yn, x, kp.pitch)};
}

// A plane's value at a neighbour's offset, or a Dirichlet side's constant
// (DIR: some side is a Dirichlet side).  Every read of another cell goes
// through here, where the debug build checks it.
template <bool DIR, int SITE>
__device__ __forceinline__ double plane_at(const double *p, int o, const double *side, const KParams &kp)
{
    if (DIR && o < 0) return side ? side[-o - 1] : 0.0;
    return HLBM_CELL_OK(o / kp.pitch, o % kp.pitch, 1, kp, SITE) ? p[o] : 0.0;
}

template <bool SIG, bool PHI0, bool DIR>
__global__ void __launch_bounds__(256)
split_level_kernel(const double *F, const double *A, double *__restrict__ outA,
                   const SplitPlanes sp, const KParams kp)
{
    __shared__ Tables64 tab;
    load_tables64(tab);
    step_begin();
    step_next();  // at the start: Sod tube 12.9 us per step against 14.1 at the end, 1024^2 alike
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= kp.nx || y >= kp.ny) return;
    const long long P = kp.plane;
    const int o = y * kp.pitch + x;
    const int xw = map_col(x - 1, kp), xe = map_col(x + 1, kp), ys = map_row(y - 1, kp), yn = map_row(y + 1, kp);
    const int pitch = kp.pitch;
    const int oW = join_map(y, xw, pitch), oE = join_map(y, xe, pitch), oS = join_map(ys, x, pitch), oN = join_map(yn, x, pitch);
    if (!HLBM_CELL_OK(y, x, 1, kp, 31)) return;
    // pull: population i comes from (x - c_ix, y - c_iy)
    double f[9];
    {
        const int src[9] = {o, oW, oS, oE, oN, join_map(ys, xw, pitch), join_map(ys, xe, pitch), join_map(yn, xe, pitch),
                            join_map(yn, xw, pitch)};
#pragma unroll
        for (int i = 0; i < 9; i++) {
            if (DIR && src[i] < 0) f[i] = kp.d_F[-src[i] - 1][i];
            else f[i] = HLBM_CELL_OK(src[i] / pitch, src[i] % pitch, 1, kp, 31) ? F[i * P + src[i]] : 0.0;
        }
    }
    const double *pu = A + A_UX * P, *pv = A + A_UY * P, *pt = A + A_TH * P, *ps = A + A_S * P;
    const double rho0 = A[A_RHO * P + o], ux0 = pu[o], uy0 = pv[o], th0 = pt[o], s0 = ps[o];
    auto at = [&](const double *p, int q, const double *side) { return plane_at<DIR, 31>(p, q, side, kp); };
    // twice the central differences
    const double dxux = at(pu, oE, kp.d_ux) - at(pu, oW, kp.d_ux);
    const double dyux = at(pu, oN, kp.d_ux) - at(pu, oS, kp.d_ux);
    const double dxuy = at(pv, oE, kp.d_uy) - at(pv, oW, kp.d_uy);
    const double dyuy = at(pv, oN, kp.d_uy) - at(pv, oS, kp.d_uy);
    const double lap = (at(pt, oE, kp.d_th) + at(pt, oW, kp.d_th)) +
                       (at(pt, oN, kp.d_th) + at(pt, oS, kp.d_th)) - 4.0 * th0;
    // u ds/dx with limited upwind faces (muscl_adv): (s0 + d0/2) - (sq + dq/2)
    // from the upwind side q, times |u|; on the mirrored stencil of u < 0 the
    // slopes change sign.  Both sides are loaded before u is known.
    auto face = [&](double u, int om, int op, const double *pd) {
        const double sm = at(ps, om, kp.d_s), sq = at(ps, op, kp.d_s);
        const double dm = at(pd, om, nullptr), dq = at(pd, op, nullptr);  // no slope on a Dirichlet side
        const bool pos = positive64(u);
        return fma(pos ? 0.5 : -0.5, pd[o] - (pos ? dm : dq), s0 - (pos ? sm : sq));
    };
    const double fx = face(ux0, oW, oE, sp.dx), fy = face(uy0, oS, oN, sp.dy);
    const double ad = fma(fabs(ux0), fx, fabs(uy0) * fy);
    double phi;
    if (PHI0) {
        const double a_xx = A[A_XX * P + o], a_xy = A[A_XY * P + o], a_yy = A[A_YY * P + o];
        phi = -sp.mp[o] * (a_xx * dxux + a_xy * (dyux + dxuy) + a_yy * dyuy);
    } else {
        const double d1 = dxux - dyuy, d2 = dyux + dxuy;
        phi = sp.quarter_mu * (d1 * d1 + d2 * d2);
    }
    const double rt = rho0 * th0, heat = fma(kp.lambda, lap, phi);
    const double s = rcp64_ok(rt) ? fma(heat, rcp64(rt), s0 - ad) : (s0 - ad) + heat / rt;
    double rho, jx, jy, ux, uy;
    moments64(f, rho, jx, jy);
    velocity64(jx, jy, rho, ux, uy);
    const double th = theta64(tab, kp, rho, s);
    outA[A_S * P + o] = s;
    sp.rho[o] = rho;
    sp.ux[o] = ux;
    sp.uy[o] = uy;
    sp.th[o] = th;
    const double omt = 1.0 - th;
    sp.gx[o] = rho * ux * fma(-ux, ux, omt);
    sp.gy[o] = rho * uy * fma(-uy, uy, omt);
    if (SIG) {
        const double diag = (f[5] + f[6]) + (f[7] + f[8]);
        sp.mxx[o] = (f[1] + f[3]) + diag;
        sp.myy[o] = (f[2] + f[4]) + diag;
        sp.mxy[o] = (f[5] - f[6]) + (f[7] - f[8]);
    }
}

// Populations after the collision (build_populations) with fewer operations:
//   - the recurrence of Sec. 3.3 for a1_xxyy, its off-equilibrium trace term
//     included, is m2(u_x) a1_yy + m2(u_y) a1_xx + 4 u_x u_y a1_xy with m2(u) =
//     u^2 + theta / 3 (the products of the lower coefficients expand and
//     cancel), three operations instead of eleven;
//   - the inverse transform works on halved and quartered moments, so that
//     its factors 1/2 cost nothing.
// 54 FP64 operations instead of 72.
__device__ __forceinline__ void populations64(double rho, double ux, double uy, double th, double axx, double axy, double ayy,
                                              double ex, double ey, double omega, double f[9])
{
    const double t3 = th * (1.0 / 3.0);
    const double mx = fma(ux, ux, t3), my = fma(uy, uy, t3);
    const double ux2 = 2.0 * ux, uy2 = 2.0 * uy, m = ux2 * axy;
    const double axxy = fma(uy, axx, m), ayyx = fma(ux, ayy, uy2 * axy);
    const double axxyy = fma(uy2, m, fma(my, axx, mx * ayy));
    const double rh = 0.5 * rho, rq = 0.25 * rho, oh = 0.5 * omega, oq = 0.25 * omega;
    const double exq = 0.25 * ex, eyq = 0.25 * ey;
    const double rqx = rq * ux, rqm = rq * mx;
    // h_ab = R_ab / 2, q_ab = R_ab / 4
    const double h10 = rh * ux, h01 = rh * uy;
    const double h20 = fma(rh, mx, fma(oh, axx, exq)), h02 = fma(rh, my, fma(oh, ayy, eyq));
    const double q11 = fma(rqx, uy, oq * axy), q21 = fma(rqm, uy, oq * axxy), q12 = fma(rqx, my, oq * ayyx);
    const double q22 = fma(rqm, my, fma(oq, axxyy, (exq + eyq) * (1.0 / 6.0)));
    const double x0z = fma(-2.0, h20, rho), x0p = h20 + h10, x0m = h20 - h10;
    const double x1z = fma(-2.0, q21, h01), x1p = q21 + q11, x1m = q21 - q11;  // halves
    const double x2z = fma(-2.0, q22, h02), x2p = q22 + q12, x2m = q22 - q12;  // halves
    f[0] = fma(-2.0, x2z, x0z);
    f[1] = fma(-2.0, x2p, x0p);
    f[3] = fma(-2.0, x2m, x0m);
    f[2] = x2z + x1z;
    f[4] = x2z - x1z;
    f[5] = x2p + x1p;
    f[8] = x2p - x1p;
    f[6] = x2m + x1m;
    f[7] = x2m - x1m;
}

// The two limited slopes of s at a cell.
template <bool DIR, int SITE>
__device__ __forceinline__ void slopes64(const double *ps, int o, const Cross &c, const KParams &kp,
                                         const SplitPlanes &sp)
{
    const double s0 = ps[o];
    auto at = [&](int q) { return plane_at<DIR, SITE>(ps, q, kp.d_s, kp); };
    sp.dx[o] = va_slope64(s0 - at(c.w), at(c.e) - s0);
    sp.dy[o] = va_slope64(s0 - at(c.s), at(c.n) - s0);
}

// A: the auxiliary planes of level n+1 (split_level_kernel wrote s); a1 goes
// there, and with CANON the derived macros, the populations to F.
template <bool SIG, bool DIR, bool CANON>
__global__ void __launch_bounds__(256)
split_collide_kernel(double *__restrict__ F, double *A, const SplitPlanes sp, const KParams kp)
{
    __shared__ Tables64 tab;
    if (CANON) load_tables64(tab);
    step_begin();
    step_next();
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= kp.nx || y >= kp.ny) return;
    const long long P = kp.plane;
    const int o = y * kp.pitch + x;
    const Cross c = cross_of(x, y, kp);
    if (!HLBM_CELL_OK(y, x, 1, kp, 32)) return;
    auto at = [&](const double *q, int oq, const double *side) { return plane_at<DIR, 32>(q, oq, side, kp); };
    const double *pu = sp.ux, *pv = sp.uy;
    const double rho = sp.rho[o], ux = pu[o], uy = pv[o], th = sp.th[o];
    const double dxux = at(pu, c.e, kp.d_ux) - at(pu, c.w, kp.d_ux);
    const double dyux = at(pu, c.n, kp.d_ux) - at(pu, c.s, kp.d_ux);
    const double dxuy = at(pv, c.e, kp.d_uy) - at(pv, c.w, kp.d_uy);
    const double dyuy = at(pv, c.n, kp.d_uy) - at(pv, c.s, kp.d_uy);
    const double p = pressure64(rho, th);
    const double e2 = p * sp.half_tmg * (dxux + dyuy);
    // E1 upwind by the cell's velocity; u = 0 (or the ablation) takes the
    // centred difference
    const bool cen = kp.e1_centred != 0;
    auto closure = [&](double u, double gm, double gc, double gp) {
        const bool up = positive64(u) && !cen, down = negative64(u) && !cen;
        return fma(up || down ? 1.0 : 0.5, (up ? gc : gp) - (down ? gc : gm), e2);
    };
    const double ex = closure(ux, at(sp.gx, c.w, kp.d_gx), sp.gx[o], at(sp.gx, c.e, kp.d_gx));
    const double ey = closure(uy, at(sp.gy, c.s, kp.d_gy), sp.gy[o], at(sp.gy, c.n, kp.d_gy));
    const double cfd = fma(-0.25, p, sp.m_half_mu);  // half of -(mu + p / 2): the differences are doubled
    const double fdxx = cfd * (dxux - dyuy), fdxy = cfd * (dyux + dxuy);
    double axx, axy, ayy;
    if (SIG) {
        const double sg = kp.sigma, om = sp.one_m_sigma;
        const double prxx = sp.mxx[o] - rho * ux * ux - p + 0.5 * ex;
        const double pryy = sp.myy[o] - rho * uy * uy - p + 0.5 * ey;
        const double prxy = sp.mxy[o] - rho * ux * uy;
        axx = sg * prxx + om * fdxx;
        ayy = sg * pryy - om * fdxx;
        axy = sg * prxy + om * fdxy;
    } else {
        axx = fdxx; ayy = -fdxx; axy = fdxy;
    }
    double omega, mp;
    relaxation64(sp.two_mu, kp.mu, p, omega, mp);
    double f[9];
    populations64(rho, ux, uy, th, axx, axy, ayy, ex, ey, omega, f);
#pragma unroll
    for (int i = 0; i < 9; i++) F[i * P + o] = f[i];
    A[A_XX * P + o] = axx;
    A[A_XY * P + o] = axy;
    A[A_YY * P + o] = ayy;
    if (CANON) {
        double r, u, v, t;
        canon_macros64(tab, f, A[A_S * P + o], kp, r, u, v, t);
        A[A_RHO * P + o] = r;
        A[A_UX * P + o] = u;
        A[A_UY * P + o] = v;
        A[A_TH * P + o] = t;
        relaxation64(sp.two_mu, kp.mu, pressure64(r, t), omega, mp);
    }
    sp.mp[o] = mp;
    slopes64<DIR, 32>(A + A_S * P, o, c, kp, sp);
}

// What the first level pass reads beside F, s and a1, from the expressions of
// the collide pass, after init or a checkpoint set the state: the slopes,
// mu / (2 mu + p), and (DERIVE) the cache planes.
template <bool DIR, bool DERIVE>
__global__ void __launch_bounds__(256)
split_prepare_kernel(const double *__restrict__ F, double *A, const SplitPlanes sp, const KParams kp)
{
    __shared__ Tables64 tab;
    if (DERIVE) load_tables64(tab);
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= kp.nx || y >= kp.ny) return;
    const long long P = kp.plane;
    const int o = y * kp.pitch + x;
    if (!HLBM_CELL_OK(y, x, 1, kp, 33)) return;
    double r, t;
    if (DERIVE) {
        double f[9], u, v;
#pragma unroll
        for (int i = 0; i < 9; i++) f[i] = F[i * P + o];
        canon_macros64(tab, f, A[A_S * P + o], kp, r, u, v, t);
        A[A_RHO * P + o] = r;
        A[A_UX * P + o] = u;
        A[A_UY * P + o] = v;
        A[A_TH * P + o] = t;
    } else {
        r = A[A_RHO * P + o];
        t = A[A_TH * P + o];
    }
    double omega, mp;
    relaxation64(sp.two_mu, kp.mu, pressure64(r, t), omega, mp);
    sp.mp[o] = mp;
    slopes64<DIR, 33>(A + A_S * P, o, cross_of(x, y, kp), kp, sp);
}

}  // namespace hlbm
