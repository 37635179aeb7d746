// lbm_node.cuh -- what the step kernels share: the loads of the pull with the wall rules, the
// stencils on rows in shared memory and the update of one node (forces, macros, the three
// collisions, the stores), in one order of operations, so that every kernel gives the
// same bits.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

template <typename Real> struct Vec2;
template <> struct Vec2<float> { using T = float2; };
template <> struct Vec2<double> { using T = double2; };

// The RX_N reference values of a staged row (16-byte aligned) in registers: two or four
// 16-byte loads instead of one load per value.
template <typename Real>
__device__ __forceinline__ void load_rowref_(const Real *rx, Real *v)
{
    if constexpr (std::is_same<Real, float>::value) {
        const float4 a = reinterpret_cast<const float4 *>(rx)[0], b = reinterpret_cast<const float4 *>(rx)[1];
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < RX_N / 2; ++i) {
            const double2 d = reinterpret_cast<const double2 *>(rx)[i];
            v[2 * i] = d.x, v[2 * i + 1] = d.y;
        }
    }
}
static_assert(RX_N == 8, "load_rowref_ reads eight values");

// grad phi = grad (phi - phi0) + (0, d_y phi0), isotropic, at column c of the phi - phi0 rows rm, r0, rp.
__device__ __forceinline__ void grad_ref_(const float *rm, const float *r0, const float *rp, int c, float gref, float &gx,
                                          float &gy)
{
    // diagonal terms from (NE, NW) +- (SE, SW): (NE + SE) - (NW + SW) and (NE - SE) + (NW - SW), both
    // halves of a pair in one packed instruction
    const float c1 = float(1.0 / 3.0), c2 = float(1.0 / 12.0);
    const float2 P = f2_(rp[c + 1], rp[c - 1]), Q = f2_(rm[c + 1], rm[c - 1]);
    const float2 S = add2_(P, Q), D = sub2_(P, Q);
    const float2 G = fma2_(bc2_(c1), f2_(r0[c + 1] - r0[c - 1], rp[c] - rm[c]),
                           mul2_(bc2_(c2), f2_(S.x - S.y, D.x + D.y)));
    gx = G.x, gy = G.y + gref;
}
// FP64: (4 (E - W) + (NE - SW) + (SE - NW)) / 12, (4 (N - S) + (NE - SW) - (SE - NW)) / 12
__device__ __forceinline__ void grad_ref_(const double *rm, const double *r0, const double *rp, int c, double gref,
                                          double &gx, double &gy)
{
    const double a = rp[c + 1] - rm[c - 1], b = rm[c + 1] - rp[c - 1], d = 1.0 / 12.0;
    gx = fma(4.0, r0[c + 1] - r0[c - 1], a + b) * d;
    gy = fma(d, fma(4.0, rp[c] - rm[c], a - b), gref);
}

// Loads of one node for the pull: populations of one lattice (plane base pointers `pl`,
// wall rule KIND) at row y and column x, with the wall rules of Sec. 5.1.  WALLS = false: no link of
// the row crosses a wall.
//   KIND 0: phase field, specular reflection (free slip, no flux through the wall)
//   KIND 1: flow, halfway bounce-back (no slip)
//   KIND 2: energy, anti-bounce-back to the wall temperature where the link crosses the wall
// Values come out in stored units (for FP16 storage: times its scale; wscale multiplies
// the anti-bounce-back wall term accordingly).  Addresses are a plane's base plus an unsigned 32-bit
// byte offset (base plus element index took a 64-bit multiply-add per load).
template <int KIND, int Q, bool WALLS = true, typename Real, typename Store>
__device__ __forceinline__ void pull_row_(const Store *const *pl, int pitch, int ny, int nx, int y, int x, int xm,
                                          int xp, Real wscale, const Real *__restrict__ twall, Real dTcold, Real *out)
{
    const uint32_t S = sizeof(Store), r0 = uint32_t(y) * uint32_t(pitch) * S, dr = uint32_t(pitch) * S;
    auto at = [&](const Store *base, uint32_t row, int col) {
        return ld_<Real, Store>(
            reinterpret_cast<const Store *>(reinterpret_cast<const char *>(base) + (row + uint32_t(col) * S)));
    };
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const int ex = ex_(a), ey = ey_(a);
        const int xs = ex > 0 ? xm : (ex < 0 ? xp : x);
        const bool wall = WALLS && ((ey > 0 && y == 0) || (ey < 0 && y == ny - 1));
        Real v;
        if (!wall) v = at(pl[a], ey > 0 ? r0 - dr : (ey < 0 ? r0 + dr : r0), xs);
        else if (KIND == 0) v = at(pl[mir_(a)], r0, xs);
        else v = at(pl[opp_(a)], r0, x);
        if (KIND == 2 && wall) {
            const Real tw = ey > 0 ? twall[(1 - ex) * nx + x] : dTcold;
            Real t = Real(2.0 * w_<Q>(a)) * tw;
            if constexpr (scaled_<Store>()) t *= wscale;
            v = -v + t;
        }
        out[a] = v;
    }
}

// Pulled populations of one lattice -> what the step keeps of them, in one order of
// operations for every kernel (FP16 storage: the sums are rescaled, not each value).
// phi - phi0 of a row from the pulled deviations and that row's dR (high and low parts)
template <int QF, typename Real, typename Store>
__device__ __forceinline__ Real phi_dev_(const StepArgs<Real, Store> &A, const Real *f, Real dr, Real drlo)
{
    Real dphi = f[0];
#pragma unroll
    for (int a = 1; a < QF; ++a) dphi += f[a];
    if constexpr (scaled_<Store>()) dphi *= A.isf;
    if constexpr (std::is_same<Real, double>::value) return dphi + dr;
    else return (dphi + drlo) + dr;
}
// T - T_ref
template <int QT, typename Real, typename Store>
__device__ __forceinline__ Real temp_dev_(const StepArgs<Real, Store> &A, const Real *h)
{
    Real dT = h[0];
#pragma unroll
    for (int a = 1; a < QT; ++a) dT += h[a];
    if constexpr (scaled_<Store>()) dT *= A.ish;
    return dT;
}
// (sigma - sigma0, p - p0) of row r at column x from dT of the pulled populations (of row r
// itself, or of the row next to the wall for the ghost rows r = -1 and r = ny)
template <typename Real, typename Store>
__device__ __forceinline__ typename Vec2<Real>::T sig_p_(const StepArgs<Real, Store> &A, int r, int x, Real dT, Real dp)
{
    Real dTs = dT;
    if (r == -1) dTs = Real(2) * A.twall[A.nx + x] - dT;   // T_ghost = 2 T_w - T_adjacent
    else if (r == A.ny) dTs = Real(2) * A.P.dTcold - dT;
    typename Vec2<Real>::T v;
    v.x = dTs * (A.P.sigma1 + A.P.sigma2 * dTs);
    v.y = dp;
    return v;
}
// first raw moments of f, and (T - T_ref, first raw moments) of h
template <int QF, typename Real, typename Store>
__device__ __forceinline__ void keep_f_(const StepArgs<Real, Store> &A, const Real *f, Real *m)
{
    raw_first_<QF>(f, m[0], m[1]);
    if constexpr (scaled_<Store>()) m[0] *= A.isf, m[1] *= A.isf;
}
template <int QT, typename Real, typename Store>
__device__ __forceinline__ void keep_h_(const StepArgs<Real, Store> &A, const Real *h, Real dT, Real *m)
{
    m[0] = dT;
    raw_first_<QT>(h, m[1], m[2]);
    if constexpr (scaled_<Store>()) m[1] *= A.ish, m[2] *= A.ish;
}
// the unit normal of a gradient as (n_x, n_y - 1)
template <typename Real, typename R2 = typename Vec2<Real>::T>
__device__ __forceinline__ R2 normal_(Real gx, Real gy, Real g2min)
{
    R2 n;
    unit_normal_dev_(gx, gy, g2min, n.x, n.y);
    return n;
}

// Row y, column x of the step: from phi - phi0 = dphi and grad phi = (gpx, gpy) of the node, the
// unit normal (n_x, n_y - 1) and (sigma - sigma0, p - p0) around it (rows m, 0, p at column s),
// what the collisions keep of the pulled populations (fm: first raw moments of f; hm: T - T_ref
// and first raw moments of h; g: the nine flow populations) and the row's reference values,
// the post-collision populations, the stored pressure and, if asked for, the fields.
template <typename Real, typename Store, int QF, int QT, typename R2 = typename Vec2<Real>::T>
__device__ __forceinline__ void node_step_(const StepArgs<Real, Store> &A, int x, int y, Real dphi, Real gpx, Real gpy,
                                           int s, const R2 *nm, const R2 *n0, const R2 *np, const R2 *qm, const R2 *q0,
                                           const R2 *qp, const Real *fm, const Real *hm, Real *g, Real phi_ref, Real th0,
                                           Real c01, Real p1)
{
    const Phys<Real> &P = A.P;
    const Real c2 = Real(1.0 / 3.0), hf = Real(0.5);
    constexpr bool SCALED = scaled_<Store>();
    const Real phi = phi_ref + dphi;
    const Real g2 = norm2_(gpx, gpy), dT = hm[0];
    const R2 nC = n0[s], nE = n0[s + 1], nW = n0[s - 1], nN = np[s], nS = nm[s];
    const R2 nNE = np[s + 1], nNW = np[s - 1], nSE = nm[s + 1], nSW = nm[s - 1];
    const R2 qE = q0[s + 1], qW = q0[s - 1], qN = qp[s], qS = qm[s];
    const R2 qNE = qp[s + 1], qNW = qp[s - 1], qSE = qm[s + 1], qSW = qm[s - 1];
    const Real nxv = nC.x, nyv = Real(1) + nC.y;
    Real fo[QF], ho[QT], ux, uy, dp;
    if constexpr (std::is_same<Real, float>::value) {
        // the stencils with the (n_x, n_y) and (sigma, p) halves paired; the diagonal terms of
        // div n summed as (NE - SW) +- (SE - NW)
        const Real c1 = Real(1.0 / 3.0), cd = Real(1.0 / 12.0);
        const float2 T1 = sub2_(nNE, nSW), T2 = sub2_(nSE, nNW);
        const Real divn = c1 * ((nE.x - nW.x) + (nN.y - nS.y)) + cd * ((T1.x + T2.x) + (T1.y - T2.y));
        const float2 X = fma2_(bc2_(c1), sub2_(qE, qW), mul2_(bc2_(cd), add2_(sub2_(qNE, qNW), sub2_(qSE, qSW))));
        const float2 Y = fma2_(bc2_(c1), sub2_(qN, qS), mul2_(bc2_(cd), add2_(sub2_(qNE, qSE), sub2_(qNW, qSW))));
        const Real dsx = X.x, dpx = X.y, dsy = Y.x, dpy = Y.y;
        const Real sigma = P.sigma0 + dT * (P.sigma1 + P.sigma2 * dT);
        const Real Fsx = P.csf * (-sigma * g2 * divn * nxv + g2 * ((Real(1) - nxv * nxv) * dsx - nxv * nyv * dsy));
        const Real Fsy = P.csf * (-sigma * g2 * divn * nyv + g2 * ((Real(1) - nyv * nyv) * dsy - nxv * nyv * dsx));
        const Real Ftx = Fsx + P.Fx, Fty = Fsy + P.Fy;
        const Real Fpx = -dpx + c2 * P.drho * gpx, Fpy = -dpy + c2 * P.drho * gpy;
        const Real rho = P.rhoA + phi * P.drho;
        const Real irho = rcp_(rho);
        Real s0, sx, sy, r20, r02, r11;
        flow_raw_moments_(g, s0, sx, sy, r20, r02, r11);
        if constexpr (SCALED) s0 *= A.isg, sx *= A.isg, sy *= A.isg, r20 *= A.isg, r02 *= A.isg, r11 *= A.isg;
        const Real irc2 = Real(3) * irho;
        ux = (sx + hf * c2 * Ftx) * irc2;
        uy = (sy + hf * c2 * Fty) * irc2;
        dp = s0 + hf * (Fpx * ux + Fpy * uy);
        const Real om_nu = rcp_(Real(3) * (P.muA + phi * P.dmu) * irho + hf);
        const Real om_T = rcp_(Real(3) * (P.kA + phi * P.dk) * irho + hf);
        // theta(phi) - theta(phi0) = (4 / W) dphi (1 - 2 phi0 - dphi)
        const Real dth = P.W4 * dphi * (Real(1) - Real(2) * phi_ref - dphi);
        // (FP16 storage: the results come out in stored units)
        collide_phase_dev_<QF, SCALED>(fo, fm[0], fm[1], dphi, phi, ux, uy, nxv, nC.y, th0, dth, c01, P.Mphi,
                                       P.omega_phi, A.sf);
        collide_flow_<SCALED>(g, rho, dp, ux, uy, Fpx, Fpy, Ftx, Fty, om_nu, s0, sx, sy, r20, r02, r11, A.sg);
        collide_energy_<QT, SCALED>(ho, hm[1], hm[2], dT, ux, uy, P.T_ref, om_T, A.sh);
    } else {
        // the same with as few FP64 instructions as it takes: stencils times 12 (the factor goes into
        // constants), F_s = delta_s (grad sigma - (sigma div n + n . grad sigma) n), no division
        // where a property is constant
        const Real divn = fma(Real(4), (nE.x - nW.x) + (nN.y - nS.y),
                              ((nNE.x - nSW.x) + (nSE.x - nNW.x)) + ((nNE.y - nSW.y) - (nSE.y - nNW.y)));
        const Real a = qNE.x - qSW.x, b = qSE.x - qNW.x, u = qNE.y - qSW.y, v = qSE.y - qNW.y;
        const Real dsx = fma(Real(4), qE.x - qW.x, a + b), dsy = fma(Real(4), qN.x - qS.x, a - b);
        const Real dpx = fma(Real(4), qE.y - qW.y, u + v), dpy = fma(Real(4), qN.y - qS.y, u - v);
        const Real csf = P.csf12 * g2, nf = -fma(P.sigma0 + q0[s].x, divn, fma(nxv, dsx, nyv * dsy));
        const Real Ftx = fma(csf, fma(nxv, nf, dsx), P.Fx), Fty = fma(csf, fma(nyv, nf, dsy), P.Fy);
        const Real Fpx = fma(P.c2drho, gpx, Real(-1.0 / 12.0) * dpx), Fpy = fma(P.c2drho, gpy, Real(-1.0 / 12.0) * dpy);
        const Real rho = fma(phi, P.drho, P.rhoA);
        const Real irho = P.constant & 1 ? P.irhoA : rcp_(rho);
        const Real om_nu = P.constant & 2 ? P.omnuA : rcp_(fma(fma(phi, P.dmu3, P.mu3A), irho, hf));
        const Real om_T = P.constant & 4 ? P.omTA : rcp_(fma(fma(phi, P.dk3, P.k3A), irho, hf));
        Real s0, sx, sy, d2, r11;
        flow_raw_moments_(g, s0, sx, sy, d2, r11);
        const Real irc2 = Real(3) * irho;
        ux = fma(hf * c2, Ftx, sx) * irc2;
        uy = fma(hf * c2, Fty, sy) * irc2;
        const Real Gh = hf * fma(Fpx, ux, Fpy * uy);
        dp = s0 + Gh;
        const Real dth = (P.W4 * dphi) * (p1 - dphi);   // p1 = 1 - 2 phi0
        collide_phase_raw_<QF>(fo, fm[0], fm[1], dphi, phi, ux, uy, nxv, nC.y, th0, dth, c01, P.Mphi, P.omega_phi);
        collide_flow_raw_(g, rho, dp, ux, uy, Fpx, Fpy, Ftx, Fty, Gh, om_nu, sx, sy, d2, r11);
        collide_energy_raw_<QT>(ho, hm[1], hm[2], dT, ux, uy, P.T_ref, om_T);
    }
    const int o = y * A.pitch + x;
    // one unsigned 32-bit byte offset from every plane's base (measured 2 % faster than
    // plane base + element index)
    const uint32_t ob = uint32_t(o) * uint32_t(sizeof(Store));
    auto at = [&](Store *base) { return reinterpret_cast<Store *>(reinterpret_cast<char *>(base) + ob); };
#pragma unroll
    for (int a = 0; a < QF; ++a) {
        st_(at(A.fo[a]), fo[a]);
    }
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        st_(at(A.go[a]), g[a]);
    }
#pragma unroll
    for (int a = 0; a < QT; ++a) {
        st_(at(A.ho[a]), ho[a]);
    }
    A.dp_out[o] = dp;
    if (A.macro) {
        const long long N = (long long)A.nx * A.ny, m = (long long)y * A.nx + x;
        A.macro[m] = A.phi0[y] + double(dphi);
        A.macro[N + m] = double(ux);
        A.macro[2 * N + m] = double(uy);
        A.macro[3 * N + m] = double(P.T_ref) + double(dT);
        A.macro[4 * N + m] = double(dp);
    }
}

}  // namespace lbm
