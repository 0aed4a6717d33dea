// Per-cell / per-face / per-edge arithmetic of the MHD bunch update (device code).
//
// Method: Haahr et al., Sec. 2.1 (ideal MHD, state vector and x-flux of Eq. 6, adiabatic
// EOS), Sec. 2.1.2 (HLLD solver, after Miyoshi & Kusano 2005), Sec. 2.1.3 (staggered
// field, arithmetic edge EMF of Eqs. 7-11, constrained transport Eq. 12, 2D Riemann
// problem at cell edges from the LB/RB/LT/RT corner states of Fig. 3), Sec. 2.1.4 (MUSCL
// slopes and Hancock half-step predictor).  Readings for what the paper leaves open are
// stated where they are used (EMF = u x B with dB/dt = +curl EMF; minmod/MC limiter;
// two-dimensional HLL edge EMF; HLLD degenerate threshold eps * Bn^2).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "mhd_ops.cuh"

namespace mhd {

// Variable order of the state and of the primitive vector.
enum { V_RHO = 0, V_MX = 1, V_MY = 2, V_MZ = 3, V_EN = 4, V_BX = 5, V_BY = 6, V_BZ = 7 };
// Primitive order: rho, u, v, w, P_gas, Bx_c, By_c, Bz_c.
enum { Q_RHO = 0, Q_U = 1, Q_V = 2, Q_W = 3, Q_P = 4, Q_BX = 5, Q_BY = 6, Q_BZ = 7 };

// max/min with ties going to the first argument (the subgradient choice of the adjoint)
template <typename R>
MHD_HD R fmax1(R a, R b) { return a >= b ? a : b; }
template <typename R>
MHD_HD R fmin1(R a, R b) { return a <= b ? a : b; }

// Limited undivided slope from the two one-sided differences a = q_i - q_{i-1},
// b = q_{i+1} - q_i (Sec. 2.1.4).  limiter 0: minmod, 1: monotonised central (the smallest of
// 2a, 2b and (a + b)/2 in magnitude).  Zero when a and b differ in sign or one is 0.
template <typename R>
MHD_HD R limited(R a, R b, int limiter) {
    const R m = minmod_(a, b);
    if (limiter == 0) return m;
    return minmod_(R(0.5) * (a + b), m + m);
}

// Fast magnetosonic speed along a normal with field component bn (transverse bt1, bt2).
// cf^2 = 1/2 (cs^2 + ca^2 + sqrt(disc)), disc = (cs^2 + ca^2)^2 - 4 cs^2 can^2 evaluated
// as (cs^2 - can^2)^2 + cat^2 (2 (cs^2 + can^2) + cat^2) (identical, no cancellation).
// EXACT: correctly rounded square roots (the CFL rates), else near ones (the solvers).
template <bool EXACT, typename R>
MHD_HD R fast_speed(R rho_inv, R gP, R bn, R bt1, R bt2) {
    // (products that feed sums are unfusable: every kernel rounds the speed the same way)
    const R cs2 = mul_(gP, rho_inv);
    const R can2 = mul_(mul_(bn, bn), rho_inv);
    const R cat2 = mul_(fma_(bt1, bt1, bt2 * bt2), rho_inv);
    const R d = cs2 - can2;
    const R disc = fma_(d, d, cat2 * fma_(R(2), cs2 + can2, cat2));
    // 1/2 (s + sqrt(disc)) as one fused step after the square root (halving is exact, so
    // this rounds as 1/2 * (s + sqrt(disc)) does)
    auto root = [](R x) { return EXACT ? rsqrt_(x) : rsqrt_near_(x); };
    return root(fma_(R(0.5), root(disc), R(0.5) * (cs2 + can2 + cat2)));
}

// Primitive state from the conserved one; the cell-centred field is the mean of the two
// faces of the cell (Sec. 2.1 EOS: P = (gamma-1)(E - rho u^2/2 - B^2/2)).
template <typename R>
MHD_HD void cons_to_prim(R rho, R mx, R my, R mz, R E, R bxc, R byc, R bzc, R gm1, R q[8]) {
    const R ri = rcp_(rho);
    const R u = mx * ri, v = my * ri, w = mz * ri;
    q[Q_RHO] = rho;
    q[Q_U] = u;
    q[Q_V] = v;
    q[Q_W] = w;
    // P = (gamma-1) (E - rho |u|^2 / 2 - |B|^2 / 2), both subtractions fused
    const R kin = fma_(u, u, fma_(v, v, w * w));
    const R mag = fma_(bxc, bxc, fma_(byc, byc, bzc * bzc));
    q[Q_P] = gm1 * fma_(R(-0.5), mag, fma_(R(-0.5) * rho, kin, E));
    q[Q_BX] = bxc;
    q[Q_BY] = byc;
    q[Q_BZ] = bzc;
}

// Hancock half step in primitive form (Sec. 2.1.4): W^{n+1/2} = W - dt/2 * (A_x W_x +
// A_y W_y + A_z W_z) for (rho, u, v, w, P) with the ideal-MHD primitive Jacobians; the
// field components of the result are set by the caller from the predicted faces.
// D[d][k]: slope of primitive k along d divided by dx_d (zero on collapsed axes).
template <typename R>
MHD_HD void hancock(const R q[8], const R D[3][8], R hdt, R gamma, R out[5]) {
    const R u = q[Q_U], v = q[Q_V], w = q[Q_W], rho = q[Q_RHO], P = q[Q_P];
    const R divu = D[0][Q_U] + D[1][Q_V] + D[2][Q_W];
    const R ri = rcp_(rho);
    // advective derivative u . grad of primitive k
    auto adv = [&](int k) { return fma_(u, D[0][k], fma_(v, D[1][k], w * D[2][k])); };
    out[0] = rho - hdt * fma_(rho, divu, adv(Q_RHO));
    out[4] = P - hdt * fma_(gamma * P, divu, adv(Q_P));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int a = (c + 1) % 3, b = (c + 2) % 3;
        // (1/rho)[d_c P + B_a d_c B_a + B_b d_c B_b - B_a d_a B_c - B_b d_b B_c]
        const R lor = fma_(q[Q_BX + a], D[c][Q_BX + a] - D[a][Q_BX + c],
                           fma_(q[Q_BX + b], D[c][Q_BX + b] - D[b][Q_BX + c], D[c][Q_P]));
        out[1 + c] = q[Q_U + c] - hdt * fma_(lor, ri, adv(Q_U + c));
    }
}

// The same half step from the undivided slopes dW[d][k] and the inverse cell sizes dxi[d]
// (D = dW * dxi folded into the products that use it; equal to hancock up to rounding).
// The step kernel's prep uses this form: one multiply less on each slope's path.  ND: active
// axes; the slopes of the others are 0, and what they multiply is left out (the compiler keeps
// products with 0), which leaves the values as they are.
template <int ND, typename R>
MHD_HD void hancock_dw(const R q[8], const R dW[3][8], const R dxi[3], R hdt, R gamma, R out[5]) {
    const R u = q[Q_U], v = q[Q_V], w = q[Q_W], rho = q[Q_RHO], P = q[Q_P];
    const R us = u * dxi[0], vs = v * dxi[1], ws = w * dxi[2];
    // x dW[0][k] + y dW[1][l] + z dW[2][m] over the active axes
    auto sum = [&](R x, int k, R y, int l, R z, int m) {
        if constexpr (ND == 3) return fma_(x, dW[0][k], fma_(y, dW[1][l], z * dW[2][m]));
        else if constexpr (ND == 2) return fma_(x, dW[0][k], y * dW[1][l]);
        else return x * dW[0][k];
    };
    const R divu = sum(dxi[0], Q_U, dxi[1], Q_V, dxi[2], Q_W);
    const R ri = rcp_(rho);
    auto adv = [&](int k) { return sum(us, k, vs, k, ws, k); };
    // d_c B_a - d_a B_c
    auto twist = [&](int c, int a) {
        if (c >= ND) return -(dxi[a] * dW[a][Q_BX + c]);
        if (a >= ND) return dxi[c] * dW[c][Q_BX + a];
        return fma_(dxi[c], dW[c][Q_BX + a], -(dxi[a] * dW[a][Q_BX + c]));
    };
    out[0] = rho - hdt * fma_(rho, divu, adv(Q_RHO));
    out[4] = P - hdt * fma_(gamma * P, divu, adv(Q_P));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int a = (c + 1) % 3, b = (c + 2) % 3;
        R lor;
        if (c < ND) lor = fma_(q[Q_BX + a], twist(c, a), fma_(q[Q_BX + b], twist(c, b), dxi[c] * dW[c][Q_P]));
        else if (a < ND && b < ND) lor = fma_(q[Q_BX + a], twist(c, a), q[Q_BX + b] * twist(c, b));
        else lor = a < ND ? q[Q_BX + a] * twist(c, a) : q[Q_BX + b] * twist(c, b);
        out[1 + c] = q[Q_U + c] - hdt * fma_(lor, ri, adv(Q_U + c));
    }
}

// Fast speeds as the double-precision Riemann solvers of the step take them: 2 rho c_f^2 = s + sqrt(disc) with
// s = gamma P + B^2 and disc = (gamma P - B^2)^2 + 4 gamma P Bt^2 (Bt^2 the transverse part of
// B^2): the value of fast_speed with the density divided out once at the end and both terms of
// disc non-negative, so that nothing cancels when gamma P ~ Bn^2 and B is along n.  disc's
// first term and s do not depend on the direction: a corner's two speeds share them.
// Returns 2 rho c_f^2; root: sqrt(disc).
template <typename R>
MHD_HD R fast_h(R gP4, R s, R dd, R bt2, R& root) {
    root = rsqrt_near_(fma_(gP4, bt2, dd));
    return s + root;
}
template <typename R>
MHD_HD R fast_h(R gP4, R s, R dd, R bt2) {
    R root;
    return fast_h(gP4, s, dd, bt2, root);
}

// HLLD flux (Sec. 2.1.2; Miyoshi & Kusano 2005) through a face with normal field bn.
// Left/right states: rho, un, ut1, ut2, P, bt1, bt2.  F receives the fluxes of
// (rho, rho*un, rho*ut1, rho*ut2, E) of the region covering x/t = 0.
// Wave speeds S_L = min(un_L, un_R) - max(cf_L, cf_R), S_R = max(..) + max(..);
// the star state is degenerate when |D| <= eps*bn^2 (then transverse v, B keep their
// outer values); ties at x/t = 0 take the left state.  Every lane takes the same path.
// The contact speed decides the side (left when S_M >= 0 or S_L >= 0), so what only one side
// needs (energies, v.B, the Alfven speed) is formed once, from the selected side.
//
// The two precisions end differently.  Single precision forms F + S (U* - U) + S* (U** - U*)
// in that order, whose rounding runs are compared by.  Double precision, where the FP64 pipe
// bounds every kernel, takes the ideal-MHD flux function at the selected region's state and
// total pressure instead, which the jump conditions make equal (in the star regions the normal
// velocity is S_M and the total pressure p_T*), and the shared form of the fast speed: about a
// third fewer FP64 operations.
template <typename R>
MHD_HD void hlld(const R L[7], const R Rt[7], R bn, R gamma, R gm1i, R eps, R F[5]) {
    constexpr bool F64 = sizeof(R) == 8;
    const R zero = R(0), half = R(0.5);
    const R bn2 = bn * bn;
    const R rl = L[0], ul = L[1], vl = L[2], wl = L[3], pl = L[4], byl = L[5], bzl = L[6];
    const R rr = Rt[0], ur = Rt[1], vr = Rt[2], wr = Rt[3], pr = Rt[4], byr = Rt[5], bzr = Rt[6];
    R b2l, b2r, cmax;
    if constexpr (F64) {
        const R btl = fma_(byl, byl, bzl * bzl), btr = fma_(byr, byr, bzr * bzr), g4 = R(4) * gamma;
        b2l = bn2 + btl;
        b2r = bn2 + btr;
        // the larger fast speed with one square root for the two sides (the root is monotone)
        const R dfl = fma_(gamma, pl, -b2l), dfr = fma_(gamma, pr, -b2r);
        const R hl = fast_h(g4 * pl, fma_(gamma, pl, b2l), dfl * dfl, btl);
        const R hr = fast_h(g4 * pr, fma_(gamma, pr, b2r), dfr * dfr, btr);
        cmax = rsqrt_near_(half * fmax_(hl * rcp_near_(rl), hr * rcp_near_(rr)));
    } else {
        b2l = fma_(byl, byl, fma_(bzl, bzl, bn2));
        b2r = fma_(byr, byr, fma_(bzr, bzr, bn2));
        cmax = fmax_(fast_speed<false>(rcp_near_(rl), gamma * pl, bn, byl, bzl), fast_speed<false>(rcp_near_(rr), gamma * pr, bn, byr, bzr));
    }
    const R ptl = fma_(half, b2l, pl), ptr = fma_(half, b2r, pr);
    const R sl = fmin_(ul, ur) - cmax;
    const R sr = fmax_(ul, ur) + cmax;
    const R sul = sl - ul, sur = sr - ur;
    const R dl = sul * rl, dr = sur * rr;
    const R deni = rcp_near_(dr - dl);
    const R sm = (fma_(dr, ur, -dl * ul) - ptr + ptl) * deni;

    // star states (transverse velocity and field)
    const R sml = sl - sm, smr = sr - sm;
    const R sli = rcp_near_(sml), sri = rcp_near_(smr);
    const R rsl = dl * sli, rsr = dr * sri;
    const R Dl = fma_(dl, sml, -bn2), Dr = fma_(dr, smr, -bn2);
    const R epb = eps * bn2;
    const auto degl = le_mag_(rabs(Dl), epb), degr = le_mag_(rabs(Dr), epb);
    const R Dli = sel(degl, zero, rcp_near_(Dl)), Dri = sel(degr, zero, rcp_near_(Dr));
    const R nul = bn * (sm - ul) * Dli, nur = bn * (sm - ur) * Dri;   // 0 when degenerate
    const R nbl = sel(degl, R(1), fma_(dl, sul, -bn2) * Dli), nbr = sel(degr, R(1), fma_(dr, sur, -bn2) * Dri);
    const R vsl = fma_(-byl, nul, vl), wsl = fma_(-bzl, nul, wl);
    const R vsr = fma_(-byr, nur, vr), wsr = fma_(-bzr, nur, wr);
    const R bysl = byl * nbl, bzsl = bzl * nbl;
    const R bysr = byr * nbr, bzsr = bzr * nbr;

    // double-star states (sign of bn: at bn = 0 their region has zero width and is never the
    // one selected, so the value there does not matter)
    const R sql = rsqrt_near_(rsl), sqr = rsqrt_near_(rsr);
    const R sgn = copysign(R(1), bn);
    const R isum = rcp_near_(sql + sqr);
    const R vss = fma_(sql, vsl, fma_(sqr, vsr, (bysr - bysl) * sgn)) * isum;
    const R wss = fma_(sql, wsl, fma_(sqr, wsr, (bzsr - bzsl) * sgn)) * isum;
    const R sq2 = sql * sqr * sgn;
    const R byss = fma_(sql, bysr, fma_(sqr, bysl, sq2 * (vsr - vsl))) * isum;
    const R bzss = fma_(sql, bzsr, fma_(sqr, bzsl, sq2 * (wsr - wsl))) * isum;

    // the side of x/t = 0 and what is needed of it
    const auto gl = nonneg_(sl), left = mor(gl, nonneg_(sm));
    const R S = sel(left, sl, sr), su = sel(left, sul, sur), si = sel(left, sli, sri);
    const R r0 = sel(left, rl, rr), u0 = sel(left, ul, ur), v0 = sel(left, vl, vr), w0 = sel(left, wl, wr);
    const R p0 = sel(left, pl, pr), by0 = sel(left, byl, byr), bz0 = sel(left, bzl, bzr);
    const R b20 = sel(left, b2l, b2r), pt0 = sel(left, ptl, ptr);
    const R rs = sel(left, rsl, rsr), vs = sel(left, vsl, vsr), ws = sel(left, wsl, wsr);
    const R bys = sel(left, bysl, bysr), bzs = sel(left, bzsl, bzsr);
    const R sq = sel(left, -sql, sqr);
    R pts;
    if constexpr (F64) pts = fma_(sel(left, dl, dr), sm - u0, pt0);
    else pts = fma_(dl * dr, ur - ul, fma_(dr, ptl, -dl * ptr)) * deni;
    const R e0 = fma_(p0, gm1i, half * fma_(r0, fma_(u0, u0, fma_(v0, v0, w0 * w0)), b20));
    const R vb0 = fma_(u0, bn, fma_(v0, by0, w0 * bz0));
    const R vbs = fma_(sm, bn, fma_(vs, bys, ws * bzs)), vbss = fma_(sm, bn, fma_(vss, byss, wss * bzss));
    const R es = fma_(su, e0, fma_(-pt0, u0, fma_(pts, sm, bn * (vb0 - vbs)))) * si;
    const R ess = fma_(sq * sgn, vbs - vbss, es);
    R sa;   // Alfven speed of the side (sq < 0 on the left)
    if constexpr (F64) sa = fma_(rabs(bn), rcp_near_(sq), sm);
    else sa = sm + rdiv(rabs(bn), sq);

    // region: outer (L, R), star or double star
    const auto outer = sel(left, gl, mnot(nonneg_(S)));
    const auto ahead = nonneg_(sa);
    const auto dstar = mand(mnot(outer), sel(left, mnot(ahead), ahead));
    if constexpr (F64) {
        const R rf = sel(outer, r0, rs), uf = sel(outer, u0, sm), ptf = sel(outer, pt0, pts);
        const R vf = sel(dstar, vss, sel(outer, v0, vs)), wf = sel(dstar, wss, sel(outer, w0, ws));
        const R byf = sel(dstar, byss, sel(outer, by0, bys)), bzf = sel(dstar, bzss, sel(outer, bz0, bzs));
        const R ef = sel(dstar, ess, sel(outer, e0, es)), vbf = sel(dstar, vbss, sel(outer, vb0, vbs));
        const R m = rf * uf;
        F[0] = m;
        F[1] = fma_(m, uf, ptf - bn2);
        F[2] = fma_(m, vf, -byf * bn);
        F[3] = fma_(m, wf, -bzf * bn);
        F[4] = fma_(ef + ptf, uf, -bn * vbf);
    } else {
        // flux of the outer state, F* = F + S (U* - U), F** = F* + S* (U** - U*) (the density
        // and normal momentum of ** are those of *)
        const R m0 = r0 * u0;
        const R f0 = m0;
        const R f1 = fma_(m0, u0, pt0 - bn2);
        const R f2v = fma_(m0, v0, -by0 * bn);
        const R f3 = fma_(m0, w0, -bz0 * bn);
        const R f4 = fma_(e0 + pt0, u0, -bn * vb0);
        const R us1 = rs * sm, us2 = rs * vs, us3 = rs * ws;
        const R g0 = fma_(S, rs - r0, f0);
        const R g1 = fma_(S, us1 - m0, f1);
        const R g2 = fma_(S, fma_(-r0, v0, us2), f2v);
        const R g3 = fma_(S, fma_(-r0, w0, us3), f3);
        const R g4 = fma_(S, es - e0, f4);
        const R h2 = fma_(sa, fma_(rs, vss, -us2), g2);
        const R h3 = fma_(sa, fma_(rs, wss, -us3), g3);
        const R h4 = fma_(sa, ess - es, g4);
        F[0] = sel(outer, f0, g0);
        F[1] = sel(outer, f1, g1);
        F[2] = sel(outer, f2v, sel(dstar, h2, g2));
        F[3] = sel(outer, f3, sel(dstar, h3, g3));
        F[4] = sel(outer, f4, sel(dstar, h4, g4));
    }
}

// HLL flux (Harten, Lax & van Leer 1983; the simple solver of the paper's mockup, Sec. 2.4)
// through a face with normal field bn: one intermediate state between the fastest signals
// S_L, S_R (the same estimates as hlld).  States and result as in hlld; the flux at x/t = 0
// is F_L when S_L >= 0, the HLL flux when S_R >= 0 > S_L, otherwise F_R.
template <typename R>
MHD_HD void hll(const R L[7], const R Rt[7], R bn, R gamma, R gm1i, R F[5]) {
    const R zero = R(0), half = R(0.5);
    const R bn2 = bn * bn;
    const R rl = L[0], ul = L[1], vl = L[2], wl = L[3], pl = L[4], byl = L[5], bzl = L[6];
    const R rr = Rt[0], ur = Rt[1], vr = Rt[2], wr = Rt[3], pr = Rt[4], byr = Rt[5], bzr = Rt[6];
    const R b2l = fma_(byl, byl, fma_(bzl, bzl, bn2)), b2r = fma_(byr, byr, fma_(bzr, bzr, bn2));
    const R ptl = fma_(half, b2l, pl), ptr = fma_(half, b2r, pr);
    const R el = fma_(pl, gm1i, half * fma_(rl, fma_(ul, ul, fma_(vl, vl, wl * wl)), b2l));
    const R er = fma_(pr, gm1i, half * fma_(rr, fma_(ur, ur, fma_(vr, vr, wr * wr)), b2r));
    const R cfl = fast_speed<false>(rcp_near_(rl), gamma * pl, bn, byl, bzl);
    const R cfr = fast_speed<false>(rcp_near_(rr), gamma * pr, bn, byr, bzr);
    const R vbl = fma_(ul, bn, fma_(vl, byl, wl * bzl)), vbr = fma_(ur, bn, fma_(vr, byr, wr * bzr));
    const R cmax = fmax_(cfl, cfr);
    const R sl = fmin_(ul, ur) - cmax;
    const R sr = fmax_(ul, ur) + cmax;
    const R ml = rl * ul, mr = rr * ur;
    const R UL[5] = {rl, ml, rl * vl, rl * wl, el};
    const R UR[5] = {rr, mr, rr * vr, rr * wr, er};
    const R FL[5] = {ml, fma_(ml, ul, ptl - bn2), fma_(ml, vl, -byl * bn), fma_(ml, wl, -bzl * bn),
                     fma_(el + ptl, ul, -bn * vbl)};
    const R FR[5] = {mr, fma_(mr, ur, ptr - bn2), fma_(mr, vr, -byr * bn), fma_(mr, wr, -bzr * bn),
                     fma_(er + ptr, ur, -bn * vbr)};
    const R di = rcp_near_(sr - sl);
    const R slr = sl * sr;
    const auto gl = nonneg_(sl), gr = nonneg_(sr);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        const R fh = fma_(sr, FL[c], fma_(-sl, FR[c], slr * (UR[c] - UL[c]))) * di;
        F[c] = sel(gl, FL[c], sel(gr, fh, FR[c]));
    }
}

// A predicted state at a cell corner around an edge (Fig. 3): density, gas pressure,
// the velocity components along the edge's two transverse axes a, b, and the field
// components along a, b and the edge direction e.
template <typename R>
struct Corner {
    R rho, p, ua, ub, Ba, Bb, Be;
};

// fast speeds of a corner state along a and b (double precision: and their inner square roots)
template <typename R>
MHD_HD void corner_speeds(const Corner<R>& s, R gamma, R& cfa, R& cfb, R& ra, R& rb) {
    if constexpr (sizeof(R) == 8) {
        const R hri = R(0.5) * rcp_near_(s.rho), gP4 = R(4) * gamma * s.p;
        const R be2 = s.Be * s.Be;
        const R ta = fma_(s.Bb, s.Bb, be2), tb = fma_(s.Ba, s.Ba, be2);   // transverse to a, to b
        const R b2 = fma_(s.Ba, s.Ba, ta);
        const R sf = fma_(gamma, s.p, b2), df = fma_(gamma, s.p, -b2);
        const R dd = df * df;
        cfa = rsqrt_near_(fast_h(gP4, sf, dd, ta, ra) * hri);
        cfb = rsqrt_near_(fast_h(gP4, sf, dd, tb, rb) * hri);
    } else {   // the rounding of fast_speed (see hlld)
        ra = rb = R(0);
        const R ri = rcp_near_(s.rho), gP = gamma * s.p;
        cfa = fast_speed<false>(ri, gP, s.Ba, s.Bb, s.Be);
        cfb = fast_speed<false>(ri, gP, s.Bb, s.Ba, s.Be);
    }
}

// Two-dimensional HLL upwind EMF at an edge from the four corner states SW, SE, NW, NE
// (E/W along a, N/S along b), with E_e = ua*Bb - ub*Ba per state:
// E = [S_E S_N E_SW - S_E S_S E_NW - S_W S_N E_SE + S_W S_S E_NE] / ((S_E-S_W)(S_N-S_S))
//     + S_E S_W/(S_E-S_W) (Bb_E - Bb_W) - S_N S_S/(S_N-S_S) (Ba_N - Ba_S),
// S_E = max(0, max ua+cf_a), S_W = min(0, min ua-cf_a), S_N, S_S likewise along b.
// It reduces to the 1D HLL induction flux when the states do not vary along a or b.
template <typename R>
MHD_HD R emf2d(const Corner<R>& SW, const Corner<R>& SE, const Corner<R>& NW, const Corner<R>& NE, R gamma) {
    R ap[4], am[4], bp[4], bm[4];
    const Corner<R>* st[4] = {&SW, &SE, &NW, &NE};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const Corner<R>& s = *st[k];
        R cfa, cfb, ra, rb;
        corner_speeds(s, gamma, cfa, cfb, ra, rb);
        ap[k] = s.ua + cfa;
        am[k] = s.ua - cfa;
        bp[k] = s.ub + cfb;
        bm[k] = s.ub - cfb;
    }
    const R sE = max0_(ap[0], ap[1], ap[2], ap[3]), sW = min0_(am[0], am[1], am[2], am[3]);
    const R sN = max0_(bp[0], bp[1], bp[2], bp[3]), sS = min0_(bm[0], bm[1], bm[2], bm[3]);
    const R da = sE - sW, db = sN - sS;
    const R eSW = fma_(SW.ua, SW.Bb, -SW.ub * SW.Ba);
    const R eSE = fma_(SE.ua, SE.Bb, -SE.ub * SE.Ba);
    const R eNW = fma_(NW.ua, NW.Bb, -NW.ub * NW.Ba);
    const R eNE = fma_(NE.ua, NE.Bb, -NE.ub * NE.Ba);
    // [S_E (S_N E_SW - S_S E_NW) - S_W (S_N E_SE - S_S E_NE)] / (da db)
    const R num = fma_(sE, fma_(sN, eSW, -sS * eNW), -sW * fma_(sN, eSE, -sS * eNE));
    const R ida = rcp_near_(da), idb = rcp_near_(db);
    return fma_(sE * sW * ida, SE.Bb - SW.Bb, fma_(num * ida, idb, -(sN * sS * idb) * (NW.Ba - SW.Ba)));
}

// The same where one of the two axes is collapsed (2D: E_x, E_y; 1D: E_y, E_z), from the states s0, s1
// of the active axis (a if along_a, else b): the four corners are two states twice over.
// Double precision: the speeds along the collapsed axis cancel, and what stays is the HLL induction
// flux E = [S_1 e_0 - S_0 e_1 + S_1 S_0 dB] / (S_1 - S_0), S_1 = max(0, max u+cf), S_0 = min(0, min u-cf):
// 2 fast speeds instead of 8.  Single precision keeps emf2d's rounding; the compiler shares the states
// that are the same (4 speeds).  512^2 box of 32^2 patches: FP64, 2 steps, 1754 -> 1388 us; FP32, 4 steps,
// 125.8 -> 118.7 us; 1D, 256 cells, FP64, 8 steps, 98.2 -> 82.5 us (FP64 with the short roots throughout;
// 1429 and 85.8 us with the rounded ones outside the solvers).
template <typename R>
MHD_HD R emf_line(const Corner<R>& s0, const Corner<R>& s1, bool along_a, R gamma) {
    if constexpr (sizeof(R) == 4) {
        return along_a ? emf2d(s0, s1, s0, s1, gamma) : emf2d(s0, s0, s1, s1, gamma);
    } else {
        auto speed = [&](const Corner<R>& s) {
            const R bn = along_a ? s.Ba : s.Bb, bt = along_a ? s.Bb : s.Ba;
            const R bt2 = fma_(bt, bt, s.Be * s.Be), b2 = fma_(bn, bn, bt2);
            const R df = fma_(gamma, s.p, -b2);
            return rsqrt_near_(fast_h(R(4) * gamma * s.p, fma_(gamma, s.p, b2), df * df, bt2) * (R(0.5) * rcp_near_(s.rho)));
        };
        const R c0 = speed(s0), c1 = speed(s1);
        const R u0 = along_a ? s0.ua : s0.ub, u1 = along_a ? s1.ua : s1.ub;
        const R S1 = fmax_(fmax_(u0 + c0, u1 + c1), R(0)), S0 = fmin_(fmin_(u0 - c0, u1 - c1), R(0));
        const R e0 = fma_(s0.ua, s0.Bb, -s0.ub * s0.Ba), e1 = fma_(s1.ua, s1.Bb, -s1.ub * s1.Ba);
        const R dB = along_a ? s1.Bb - s0.Bb : s0.Ba - s1.Ba;
        return fma_(S1 * S0, dB, fma_(S1, e0, -S0 * e1)) * rcp_near_(S1 - S0);
    }
}

}  // namespace mhd
