// Hand-written reverse-mode derivatives (vector-Jacobian products) of the per-element
// arithmetic in mhd_math.cuh, for the discrete adjoint of one bunch step at fixed dt.
//
// Each *_vjp function re-evaluates the values it needs of the forward expression and then
// accumulates (+=) the cotangents of its inputs from the cotangent of its output, sweeping the
// assignments in reverse order.  It differentiates the expression, not its rounding: where the
// forward code of a precision writes the same value in another form (the double-precision HLLD
// flux, the edge EMF's speeds) the two differ by rounding, also in a choice between branches
// whose arguments are equal to rounding.
// Non-differentiable points take the branch the forward took: the limiter passes the
// cotangent to the argument it selected (ties: the first; none when the arguments differ
// in sign or one is zero), max/min pass it to the selected argument (ties: the first),
// sqrt has derivative 0 at 0, and the HLLD region / degenerate-star choices are constant.
#pragma once

#include "mhd_math.cuh"

namespace mhd {

// d limited(a, b): lo -> la, lb
template <typename R>
MHD_HD void limited_vjp(R a, R b, int limiter, R lo, R& la, R& lb) {
    if (!same_sign_(a, b)) return;
    if (limiter == 0) {
        if (le_mag_(rabs(a), rabs(b))) la += lo;
        else lb += lo;
    } else {
        const R c = R(0.5) * (a + b);
        const bool pa = le_mag_(rabs(a), rabs(b));
        const R m2 = pa ? R(2) * a : R(2) * b;
        if (le_mag_(rabs(c), rabs(m2))) {
            la += R(0.5) * lo;
            lb += R(0.5) * lo;
        } else if (pa) {
            la += R(2) * lo;
        } else {
            lb += R(2) * lo;
        }
    }
}

// slope of q from (qm, q0, qp): lo -> lqm, lq0, lqp
template <typename R>
MHD_HD void slope_vjp(R qm, R q0, R qp, int limiter, R lo, R& lqm, R& lq0, R& lqp) {
    R la = R(0), lb = R(0);
    limited_vjp(q0 - qm, qp - q0, limiter, lo, la, lb);
    lqm -= la;
    lq0 += la - lb;
    lqp += lb;
}

// d fast_speed (in terms of rho and P): lcf -> lrho, lP, lbn, lbt1, lbt2
template <typename R>
MHD_HD void fast_speed_vjp(R rho, R P, R bn, R bt1, R bt2, R gamma, R lcf, R& lrho, R& lP, R& lbn, R& lbt1,
                           R& lbt2) {
    const R ri = rcp_near_(rho);
    const R cs2 = gamma * P * ri;
    const R can2 = bn * bn * ri;
    const R cat2 = (bt1 * bt1 + bt2 * bt2) * ri;
    const R d = cs2 - can2;
    const R disc = d * d + cat2 * (R(2) * (cs2 + can2) + cat2);
    const R s = rsqrt_near_(disc);
    const R h = R(0.5) * (cs2 + can2 + cat2 + s);
    const R cf = rsqrt_near_(h);
    const R lh = positive_(cf) ? quot_(R(0.5) * lcf, cf, rcp_near_(cf)) : R(0);
    const R ldisc = positive_(disc) ? quot_(R(0.25) * lh, s, rcp_near_(s)) : R(0);
    const R lcs2 = R(0.5) * lh + ldisc * (R(2) * d + R(2) * cat2);
    const R lcan2 = R(0.5) * lh + ldisc * (R(-2) * d + R(2) * cat2);
    const R lcat2 = R(0.5) * lh + ldisc * (R(2) * (cs2 + can2) + R(2) * cat2);
    lP += lcs2 * gamma * ri;
    lbn += lcan2 * R(2) * bn * ri;
    lbt1 += lcat2 * R(2) * bt1 * ri;
    lbt2 += lcat2 * R(2) * bt2 * ri;
    lrho -= (lcs2 * cs2 + lcan2 * can2 + lcat2 * cat2) * ri;
}

// The same for the form the double-precision solvers take, c_f = sqrt((s + root) / (2 rho)), root =
// sqrt(disc) (fast_h), from the speed and the root that the forward code found: no square root and
// half the operations.
template <typename R>
MHD_HD void fast_h_vjp(R rho, R P, R bn, R bt1, R bt2, R gamma, R cf, R root, R lcf, R& lrho, R& lP, R& lbn, R& lbt1,
                       R& lbt2) {
    const R hri = R(0.5) * rcp_near_(rho), gP = gamma * P;
    const R t = fma_(bt1, bt1, bt2 * bt2), d = gP - fma_(bn, bn, t);
    const R lx = lcf * hri;
    const R lh = positive_(cf) ? quot_(R(0.5) * lx, cf, rcp_near_(cf)) : R(0);      // of s + root
    const R ld = positive_(root) ? quot_(lh, root, rcp_near_(root)) : R(0);      // of disc, twice
    const R lb = fma_(-ld, d, lh);                                   // of B^2
    const R l2 = R(2) * lb, lt = fma_(R(4) * gP, ld, l2);
    lP += gamma * fma_(ld, fma_(R(2), t, d), lh);
    lbn += l2 * bn;
    lbt1 += lt * bt1;
    lbt2 += lt * bt2;
    lrho -= lx * cf;
}

// d cons_to_prim: lq[8] -> lU (rho, mx, my, mz, E) and lbc[3] (cell-centred field)
template <typename R>
MHD_HD void cons_to_prim_vjp(R rho, R mx, R my, R mz, R E, R bxc, R byc, R bzc, R gm1, const R lq[8], R lU[5],
                             R lbc[3]) {
    (void)E;
    const R ri = rcp_(rho);
    const R u = mx * ri, v = my * ri, w = mz * ri;
    const R lP = lq[Q_P];
    // P = gm1 (E - rho |u|^2 / 2 - |bc|^2 / 2), u = m / rho
    R lu = lq[Q_U] - lP * gm1 * rho * u;
    R lv = lq[Q_V] - lP * gm1 * rho * v;
    R lw = lq[Q_W] - lP * gm1 * rho * w;
    R lrho = lq[Q_RHO] - lP * gm1 * R(0.5) * (u * u + v * v + w * w);
    lU[4] += lP * gm1;
    lbc[0] += lq[Q_BX] - lP * gm1 * bxc;
    lbc[1] += lq[Q_BY] - lP * gm1 * byc;
    lbc[2] += lq[Q_BZ] - lP * gm1 * bzc;
    lU[1] += lu * ri;
    lU[2] += lv * ri;
    lU[3] += lw * ri;
    lrho -= (lu * u + lv * v + lw * w) * ri;
    lU[0] += lrho;
}

// d hancock: lout[5] -> lq[8] (primitives at time n) and lD[3][8] (slopes / dx)
template <typename R>
MHD_HD void hancock_vjp(const R q[8], const R D[3][8], R hdt, R gamma, const R lout[5], R lq[8], R lD[3][8]) {
    const R u = q[Q_U], v = q[Q_V], w = q[Q_W], rho = q[Q_RHO], P = q[Q_P];
    const R vel[3] = {u, v, w};
    const R divu = D[0][Q_U] + D[1][Q_V] + D[2][Q_W];
    const R ri = rcp_(rho);
    R ladv[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) ladv[k] = R(0);
    R ldivu = R(0), lri = R(0);
    // out0 = rho - hdt (adv0 + rho divu)
    lq[Q_RHO] += lout[0] * (R(1) - hdt * divu);
    ldivu -= hdt * lout[0] * rho;
    ladv[Q_RHO] -= hdt * lout[0];
    // out4 = P - hdt (adv4 + gamma P divu)
    lq[Q_P] += lout[4] * (R(1) - hdt * gamma * divu);
    ldivu -= hdt * lout[4] * gamma * P;
    ladv[Q_P] -= hdt * lout[4];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int a = (c + 1) % 3, b = (c + 2) % 3;
        const R lor = D[c][Q_P] + q[Q_BX + a] * D[c][Q_BX + a] + q[Q_BX + b] * D[c][Q_BX + b]
                      - q[Q_BX + a] * D[a][Q_BX + c] - q[Q_BX + b] * D[b][Q_BX + c];
        const R lo = lout[1 + c];
        lq[Q_U + c] += lo;
        ladv[Q_U + c] -= hdt * lo;
        const R llor = -hdt * lo * ri;
        lri -= hdt * lo * lor;
        lD[c][Q_P] += llor;
        lq[Q_BX + a] += llor * (D[c][Q_BX + a] - D[a][Q_BX + c]);
        lq[Q_BX + b] += llor * (D[c][Q_BX + b] - D[b][Q_BX + c]);
        lD[c][Q_BX + a] += llor * q[Q_BX + a];
        lD[c][Q_BX + b] += llor * q[Q_BX + b];
        lD[a][Q_BX + c] -= llor * q[Q_BX + a];
        lD[b][Q_BX + c] -= llor * q[Q_BX + b];
    }
    // adv(k) = u D0k + v D1k + w D2k
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (k == Q_BX || k == Q_BY || k == Q_BZ) continue;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            lq[Q_U + d] += ladv[k] * D[d][k];
            lD[d][k] += ladv[k] * vel[d];
        }
    }
    lD[0][Q_U] += ldivu;
    lD[1][Q_V] += ldivu;
    lD[2][Q_W] += ldivu;
    lq[Q_RHO] -= lri * ri * ri;
}

// d hlld: lF[5] -> lL[7], lR[7], lbn: the derivative of F + S (U* - U) + S* (U** - U*) in the region at
// x/t = 0, in both precisions (hlld in double precision takes the flux function at the region's state,
// which the jump conditions make equal).
template <typename R>
MHD_HD void hlld_vjp(const R L[7], const R Rt[7], R bn, R gamma, R gm1i, R eps, const R lF[5], R lL[7], R lR[7],
                     R& lbn) {
    // ----- forward (as hlld)
    const R bn2 = bn * bn;
    const R rl = L[0], ul = L[1], vl = L[2], wl = L[3], pl = L[4], byl = L[5], bzl = L[6];
    const R rr = Rt[0], ur = Rt[1], vr = Rt[2], wr = Rt[3], pr = Rt[4], byr = Rt[5], bzr = Rt[6];
    const R btl = byl * byl + bzl * bzl, btr = byr * byr + bzr * bzr;
    const R b2l = bn2 + btl, b2r = bn2 + btr;
    const R ptl = pl + R(0.5) * b2l, ptr = pr + R(0.5) * b2r;
    bool cl;   // max picks cf_L
    R cmax, croot = 0;
    if constexpr (sizeof(R) == 8) {
        const R g4 = R(4) * gamma, gpl = gamma * pl, gpr = gamma * pr;
        R rootl, rootr;
        const R hl = fast_h(g4 * pl, gpl + b2l, (gpl - b2l) * (gpl - b2l), btl, rootl) * rcp_near_(rl);
        const R hr = fast_h(g4 * pr, gpr + b2r, (gpr - b2r) * (gpr - b2r), btr, rootr) * rcp_near_(rr);
        cl = number_(hl) && !greater_(hr, hl);
        cmax = rsqrt_near_(R(0.5) * (cl ? hl : hr));
        croot = cl ? rootl : rootr;
    } else {
        const R cfl = fast_speed<false>(rcp_near_(rl), gamma * pl, bn, byl, bzl);
        const R cfr = fast_speed<false>(rcp_near_(rr), gamma * pr, bn, byr, bzr);
        cl = number_(cfl) && !greater_(cfr, cfl);
        cmax = cl ? cfl : cfr;
    }
    const bool ml = !greater_(ul, ur);     // min picks u_L
    const bool Ml = !greater_(ur, ul);     // max picks u_L
    const R sl = (ml ? ul : ur) - cmax;
    const R sr = (Ml ? ul : ur) + cmax;
    const R dl = (sl - ul) * rl, dr = (sr - ur) * rr;
    const R den = dr - dl;
    const R deni = rcp_near_(den);
    const R smn = dr * ur - dl * ul - ptr + ptl;
    const R ptn = dr * ptl - dl * ptr + dl * dr * (ur - ul);
    const R sm = smn * deni;
    const R pts = ptn * deni;
    // density of the star states, Alfven speeds, and the region at x/t = 0
    struct Side {   // a side's state and what all regions need of its star state
        R r, u, v, w, p, by, bz, b2, pt, S, sa, ssm, ssmi, rs, sq, isq;
    };
    auto side = [&](const R* W, R b2, R pt, R S) {
        Side t{W[0], W[1], W[2], W[3], W[4], W[5], W[6], b2, pt, S};
        t.sa = S - t.u;
        t.ssm = S - sm;
        t.ssmi = rcp_near_(t.ssm);
        t.rs = t.r * t.sa * t.ssmi;
        t.sq = rsqrt_near_(t.rs);
        t.isq = rcp_near_(t.sq);
        return t;
    };
    const Side A = side(L, b2l, ptl, sl), B = side(Rt, b2r, ptr, sr);
    const R abn = rabs(bn);
    const R sgn = nonzero_(bn) ? copysign(R(1), bn) : R(0);
    int reg = 5;
    if (nonneg_(sr)) reg = 4;
    if (nonneg_(sm + abn * B.isq)) reg = 3;
    if (nonneg_(sm)) reg = 2;
    if (nonneg_(sm - abn * A.isq)) reg = 1;
    if (nonneg_(sl)) reg = 0;
    const bool left = reg <= 2, dstar = reg == 2 || reg == 3;

    // ----- reverse, in terms of the near side (that of x/t = 0: field by field, so that lanes of either
    // side take one path) and the far side, whose star state only the double star uses; with sg =
    // sgn on the left, -sgn on the right, and tau = 1, -1 the formulas of the two sides are one.
    auto pick = [&](bool l) {
        Side t;
        t.r = sel(l, A.r, B.r); t.u = sel(l, A.u, B.u); t.v = sel(l, A.v, B.v); t.w = sel(l, A.w, B.w);
        t.p = sel(l, A.p, B.p); t.by = sel(l, A.by, B.by); t.bz = sel(l, A.bz, B.bz); t.b2 = sel(l, A.b2, B.b2);
        t.pt = sel(l, A.pt, B.pt); t.S = sel(l, A.S, B.S); t.sa = sel(l, A.sa, B.sa); t.ssm = sel(l, A.ssm, B.ssm);
        t.ssmi = sel(l, A.ssmi, B.ssmi); t.rs = sel(l, A.rs, B.rs); t.sq = sel(l, A.sq, B.sq); t.isq = sel(l, A.isq, B.isq);
        return t;
    };
    const Side N = pick(left), O = pick(!left);
    const R sg = left ? sgn : -sgn, tabn = left ? abn : -abn;
    struct SideGrad {   // cotangents of a side's state (pt, e and v.B as they come), its wave speed
        R r = 0, u = 0, v = 0, w = 0, p = 0, by = 0, bz = 0, pt = 0, e = 0, vb = 0, S = 0;
    } gn, go;
    R g_bn = 0, g_bn2 = 0, g_sm = 0, g_pts = 0, g_tabn = 0;
    struct Energy {
        R kin, e, vb;
    };
    auto energy = [&](const Side& T) {   // u^2 / 2, e = p gm1i + r u^2 / 2 + b2 / 2, v.B
        const R kin = R(0.5) * (T.u * T.u + T.v * T.v + T.w * T.w);
        return Energy{kin, T.p * gm1i + T.r * kin + R(0.5) * T.b2, T.u * bn + T.v * T.by + T.w * T.bz};
    };
    auto energy_rev = [&](const Side& T, const Energy& E, SideGrad& g) {   // (b2 / 2 comes with pt's)
        g.u += g.vb * bn; g_bn += g.vb * T.u; g.v += g.vb * T.by; g.by += g.vb * T.v; g.w += g.vb * T.bz; g.bz += g.vb * T.w;
        g.p += g.e * gm1i;
        g.r += g.e * E.kin;
        const R er = g.e * T.r;
        g.u += er * T.u; g.v += er * T.v; g.w += er * T.w;
    };
    struct Star {
        R Di, nu, nb, vs, ws, bys, bzs, vbs, es;
        bool deg;
    };
    auto star = [&](const Side& T, const Energy& E) {
        Star t;
        const R D = T.r * T.sa * T.ssm - bn2;
        t.deg = le_mag_(rabs(D), eps * bn2);
        t.Di = t.deg ? R(0) : rcp_near_(D);
        t.nu = bn * (sm - T.u) * t.Di;
        t.nb = (T.r * T.sa * T.sa - bn2) * t.Di;
        t.vs = t.deg ? T.v : T.v - T.by * t.nu;
        t.ws = t.deg ? T.w : T.w - T.bz * t.nu;
        t.bys = t.deg ? T.by : T.by * t.nb;
        t.bzs = t.deg ? T.bz : T.bz * t.nb;
        t.vbs = sm * bn + t.vs * t.bys + t.ws * t.bzs;
        t.es = (T.sa * E.e - T.pt * T.u + pts * sm + bn * (E.vb - t.vbs)) * T.ssmi;
        return t;
    };
    struct StarGrad {
        R rs = 0, vs = 0, ws = 0, bys = 0, bzs = 0, vbs = 0, es = 0, sq = 0;
    };
    auto star_rev = [&](const Side& T, const Energy& E, const Star& t, StarGrad h, SideGrad& g) {
        // sq = sqrt(rs)
        h.rs += quot_(R(0.5) * h.sq, T.sq, T.isq);
        // es = nes * ssmi
        const R g_nes = h.es * T.ssmi;
        R g_ssm = -g_nes * t.es;
        // nes = sa e - pt u + pts sm + bn (vb - vbs)
        R g_sa = g_nes * E.e;
        g.e += g_nes * T.sa;
        g.pt -= g_nes * T.u;
        g.u -= g_nes * T.pt;
        g_pts += g_nes * sm;
        g_sm += g_nes * pts;
        g_bn += g_nes * (E.vb - t.vbs);
        g.vb += g_nes * bn;
        h.vbs -= g_nes * bn;
        // vbs = sm bn + vs bys + ws bzs
        g_sm += h.vbs * bn;
        g_bn += h.vbs * sm;
        h.vs += h.vbs * t.bys;
        h.bys += h.vbs * t.vs;
        h.ws += h.vbs * t.bzs;
        h.bzs += h.vbs * t.ws;
        g.v += h.vs;
        g.w += h.ws;
        if (!t.deg) {
            g.by += h.bys * t.nb - h.vs * t.nu;
            g.bz += h.bzs * t.nb - h.ws * t.nu;
            // nu = bn (sm - u) / D, nb = (r sa^2 - bn2) / D
            const R g_nu = -(h.vs * T.by + h.ws * T.bz) * t.Di, g_nb = (h.bys * T.by + h.bzs * T.bz) * t.Di;
            g_bn += g_nu * (sm - T.u);
            g_sm += g_nu * bn;
            g.u -= g_nu * bn;
            const R g_D = -(g_nu * t.nu + g_nb * t.nb);
            const R bsa = g_nb * T.sa;
            g.r += bsa * T.sa;
            g_sa += R(2) * bsa * T.r;
            g_bn2 -= g_nb + g_D;
            // D = r sa ssm - bn2
            const R dss = g_D * T.ssm, dr_ = g_D * T.r;
            g.r += dss * T.sa;
            g_sa += dss * T.r;
            g_ssm += dr_ * T.sa;
        } else {
            g.by += h.bys;
            g.bz += h.bzs;
        }
        // rs = r sa ssmi
        const R rsi = h.rs * T.ssmi;
        g.r += rsi * T.sa;
        g_sa += rsi * T.r;
        g_ssm -= rsi * T.rs;
        // ssm = S - sm ; sa = S - u
        g.S += g_ssm + g_sa;
        g_sm -= g_ssm;
        g.u -= g_sa;
    };

    // the near side's flux
    const Energy En = energy(N);
    {
        const R lv = lF[1] * N.u + lF[2] * N.v + lF[3] * N.w;
        const R ru = N.r * N.u;
        gn.r = (lF[0] + lv) * N.u;
        gn.u = N.r * (lF[0] + lv) + lF[1] * ru + lF[4] * (En.e + N.pt);
        gn.v = lF[2] * ru;
        gn.w = lF[3] * ru;
        gn.pt = lF[1] + lF[4] * N.u;
        g_bn2 -= lF[1];
        gn.by = -lF[2] * bn;
        gn.bz = -lF[3] * bn;
        g_bn -= lF[2] * N.by + lF[3] * N.bz + lF[4] * En.vb;
        gn.e = lF[4] * N.u;
        gn.vb = -lF[4] * bn;
        if (reg != 0 && reg != 5) {
            const Star T = star(N, En);
            // f += S (U* - U), U* = (rs, rs sm, rs vs, rs ws, es)
            const R ls = lF[0] + lF[1] * sm + lF[2] * T.vs + lF[3] * T.ws;
            // (difference by difference: of the two sums the larger parts cancel)
            gn.S += lF[0] * (N.rs - N.r) + lF[1] * (N.rs * sm - ru) + lF[2] * (N.rs * T.vs - N.r * N.v) +
                    lF[3] * (N.rs * T.ws - N.r * N.w) + lF[4] * (T.es - En.e);
            const R Sr = N.S * N.r, Srs = N.S * N.rs;
            gn.r -= N.S * (lF[0] + lv);
            gn.u -= Sr * lF[1];
            gn.v -= Sr * lF[2];
            gn.w -= Sr * lF[3];
            gn.e -= N.S * lF[4];
            StarGrad h;
            h.rs = N.S * ls;
            g_sm += Srs * lF[1];
            h.vs = Srs * lF[2];
            h.ws = Srs * lF[3];
            h.es = N.S * lF[4];
            if (dstar) {
                const Energy Eo = energy(O);
                const Star F = star(O, Eo);
                StarGrad k;
                const R isum = rcp_near_(N.sq + O.sq), sq2 = N.sq * O.sq * sg;
                const R dvs = (F.vs - T.vs) * sg, dws = (F.ws - T.ws) * sg;
                const R vss = (N.sq * T.vs + O.sq * F.vs + (F.bys - T.bys) * sg) * isum;
                const R wss = (N.sq * T.ws + O.sq * F.ws + (F.bzs - T.bzs) * sg) * isum;
                const R byss = (N.sq * F.bys + O.sq * T.bys + sq2 * (F.vs - T.vs)) * isum;
                const R bzss = (N.sq * F.bzs + O.sq * T.bzs + sq2 * (F.ws - T.ws)) * isum;
                const R vbss = sm * bn + vss * byss + wss * bzss;
                // f += S* (U** - U*), S* = sm - tau abn / sq,
                // U** - U* = (0, 0, rs (vss - vs), rs (wss - ws), -sq (vbs - vbss) sg)
                const R Ss = sm - tabn * N.isq, dvb = (T.vbs - vbss) * sg;
                const R ld = lF[2] * (vss - T.vs) + lF[3] * (wss - T.ws);
                const R gSs = N.rs * ld - lF[4] * N.sq * dvb;
                h.rs += Ss * ld;
                const R Ssrs = Ss * N.rs;
                const R g_vss = Ssrs * lF[2], g_wss = Ssrs * lF[3];
                h.vs -= g_vss;
                h.ws -= g_wss;
                const R g_ess = Ss * lF[4];
                h.sq -= g_ess * dvb;
                const R g_vbss = g_ess * N.sq * sg;
                h.vbs -= g_vbss;
                const R gsi = quot_(gSs, N.sq, N.isq);
                g_sm += gSs;
                g_tabn -= gsi;
                h.sq += quot_(gsi * tabn, N.sq, N.isq);
                // vbss = sm bn + vss byss + wss bzss
                g_sm += g_vbss * bn;
                g_bn += g_vbss * sm;
                // x = n * isum
                const R g_nv = (g_vss + g_vbss * byss) * isum, g_nw = (g_wss + g_vbss * bzss) * isum;
                const R g_nby = g_vbss * vss * isum, g_nbz = g_vbss * wss * isum;
                const R g_sum = g_nv * vss + g_nw * wss + g_nby * byss + g_nbz * bzss;   // isum = 1 / (sq + sq_o)
                // nv = sq vs + sq_o vs_o + (bys_o - bys) sg, nw alike;
                // nby = sq bys_o + sq_o bys + sq sq_o (vs_o - vs) sg, nbz alike
                h.sq += g_nv * T.vs + g_nw * T.ws + g_nby * (F.bys + O.sq * dvs) + g_nbz * (F.bzs + O.sq * dws) - g_sum;
                k.sq = g_nv * F.vs + g_nw * F.ws + g_nby * (T.bys + N.sq * dvs) + g_nbz * (T.bzs + N.sq * dws) - g_sum;
                h.vs += g_nv * N.sq - g_nby * sq2;
                k.vs = g_nv * O.sq + g_nby * sq2;
                h.ws += g_nw * N.sq - g_nbz * sq2;
                k.ws = g_nw * O.sq + g_nbz * sq2;
                h.bys = g_nby * O.sq - g_nv * sg;
                k.bys = g_nby * N.sq + g_nv * sg;
                h.bzs = g_nbz * O.sq - g_nw * sg;
                k.bzs = g_nbz * N.sq + g_nw * sg;
                star_rev(O, Eo, F, k, go);
                energy_rev(O, Eo, go);
            }
            star_rev(N, En, T, h, gn);
        }
    }
    energy_rev(N, En, gn);
    const R g_abn = left ? g_tabn : -g_tabn;
    R g_rl = sel(left, gn.r, go.r), g_rr = sel(left, go.r, gn.r), g_ul = sel(left, gn.u, go.u), g_ur = sel(left, go.u, gn.u);
    const R g_vl = sel(left, gn.v, go.v), g_vr = sel(left, go.v, gn.v), g_wl = sel(left, gn.w, go.w), g_wr = sel(left, go.w, gn.w);
    R g_pl = sel(left, gn.p, go.p), g_pr = sel(left, go.p, gn.p), g_byl = sel(left, gn.by, go.by), g_byr = sel(left, go.by, gn.by);
    R g_bzl = sel(left, gn.bz, go.bz), g_bzr = sel(left, go.bz, gn.bz), g_ptl = sel(left, gn.pt, go.pt), g_ptr = sel(left, go.pt, gn.pt);
    const R g_el = sel(left, gn.e, go.e), g_er = sel(left, go.e, gn.e);
    R g_sl = sel(left, gn.S, go.S), g_sr = sel(left, go.S, gn.S);
    // sm = smn / den ; pts = ptn / den
    const R g_smn = g_sm * deni, g_ptn = g_pts * deni;
    R g_den = -(g_sm * sm + g_pts * pts) * deni;
    // ptn = dr ptl - dl ptr + dl dr (ur - ul)
    R g_dr = g_ptn * (ptl + dl * (ur - ul));
    R g_dl = g_ptn * (-ptr + dr * (ur - ul));
    g_ptl += g_ptn * dr;
    g_ptr -= g_ptn * dl;
    g_ur += g_ptn * dl * dr;
    g_ul -= g_ptn * dl * dr;
    // smn = dr ur - dl ul - ptr + ptl
    g_dr += g_smn * ur;
    g_ur += g_smn * dr;
    g_dl -= g_smn * ul;
    g_ul -= g_smn * dl;
    g_ptr -= g_smn;
    g_ptl += g_smn;
    // den = dr - dl
    g_dr += g_den;
    g_dl -= g_den;
    // dl = (sl - ul) rl ; dr = (sr - ur) rr
    g_sl += g_dl * rl;
    g_ul -= g_dl * rl;
    g_rl += g_dl * (sl - ul);
    g_sr += g_dr * rr;
    g_ur -= g_dr * rr;
    g_rr += g_dr * (sr - ur);
    // sl = min(ul, ur) - cmax ; sr = max(ul, ur) + cmax
    const R g_cmax = g_sr - g_sl;
    if (ml) g_ul += g_sl;
    else g_ur += g_sl;
    if (Ml) g_ul += g_sr;
    else g_ur += g_sr;
    // the fast speed of the side that the max picked
    {
        R h_r = 0, h_p = 0, h_by = 0, h_bz = 0;
        const R r0 = cl ? rl : rr, p0 = cl ? pl : pr, by0 = cl ? byl : byr, bz0 = cl ? bzl : bzr;
        if constexpr (sizeof(R) == 8)
            fast_h_vjp(r0, p0, bn, by0, bz0, gamma, cmax, croot, g_cmax, h_r, h_p, g_bn, h_by, h_bz);
        else
            fast_speed_vjp(r0, p0, bn, by0, bz0, gamma, g_cmax, h_r, h_p, g_bn, h_by, h_bz);
        if (cl) {
            g_rl += h_r; g_pl += h_p; g_byl += h_by; g_bzl += h_bz;
        } else {
            g_rr += h_r; g_pr += h_p; g_byr += h_by; g_bzr += h_bz;
        }
    }
    // pt = p + b2 / 2 (and the b2 / 2 of e)
    const R g_b2l = R(0.5) * g_el + R(0.5) * g_ptl, g_b2r = R(0.5) * g_er + R(0.5) * g_ptr;
    g_pl += g_ptl;
    g_pr += g_ptr;
    // b2 = bn2 + by^2 + bz^2
    g_bn2 += g_b2l + g_b2r;
    g_byl += R(2) * byl * g_b2l; g_bzl += R(2) * bzl * g_b2l;
    g_byr += R(2) * byr * g_b2r; g_bzr += R(2) * bzr * g_b2r;
    // bn2 = bn^2 ; abn = |bn|
    g_bn += R(2) * bn * g_bn2 + g_abn * sgn;
    lL[0] += g_rl; lL[1] += g_ul; lL[2] += g_vl; lL[3] += g_wl; lL[4] += g_pl; lL[5] += g_byl; lL[6] += g_bzl;
    lR[0] += g_rr; lR[1] += g_ur; lR[2] += g_vr; lR[3] += g_wr; lR[4] += g_pr; lR[5] += g_byr; lR[6] += g_bzr;
    lbn += g_bn;
}

// d hll: lF[5] -> lL[7], lR[7], lbn.  Same forward sequence as hll(); the region (L, HLL
// state, R) and the max / min selections of the wave speeds are constant.
template <typename R>
MHD_HD void hll_vjp(const R L[7], const R Rt[7], R bn, R gamma, R gm1i, const R lF[5], R lL[7], R lR[7], R& lbn) {
    // ----- forward (as hll)
    const R bn2 = bn * bn;
    const R* st[2] = {L, Rt};
    R U[2][5], F[2][5], cf[2], e[2], pt[2], vb[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const R r = st[k][0], u = st[k][1], v = st[k][2], w = st[k][3], p = st[k][4], by = st[k][5], bz = st[k][6];
        const R b2 = bn2 + by * by + bz * bz;
        pt[k] = p + R(0.5) * b2;
        e[k] = p * gm1i + R(0.5) * r * (u * u + v * v + w * w) + R(0.5) * b2;
        cf[k] = fast_speed<false>(rcp_near_(r), gamma * p, bn, by, bz);
        vb[k] = u * bn + v * by + w * bz;
        U[k][0] = r;
        U[k][1] = r * u;
        U[k][2] = r * v;
        U[k][3] = r * w;
        U[k][4] = e[k];
        F[k][0] = r * u;
        F[k][1] = r * u * u + pt[k] - bn2;
        F[k][2] = r * v * u - by * bn;
        F[k][3] = r * w * u - bz * bn;
        F[k][4] = (e[k] + pt[k]) * u - bn * vb[k];
    }
    const R ul = L[1], ur = Rt[1];
    const bool cl = number_(cf[0]) && !greater_(cf[1], cf[0]);
    const R cmax = cl ? cf[0] : cf[1];
    const bool ml = !greater_(ul, ur), Ml = !greater_(ur, ul);
    const R sl = (ml ? ul : ur) - cmax;
    const R sr = (Ml ? ul : ur) + cmax;
    // ----- reverse
    R lU[2][5] = {{0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}}, lFs[2][5] = {{0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}};
    R lsl = R(0), lsr = R(0);
    if (nonneg_(sl)) {
        for (int c = 0; c < 5; ++c) lFs[0][c] = lF[c];
    } else if (nonneg_(sr)) {
        const R di = rcp_near_(sr - sl);
        for (int c = 0; c < 5; ++c) {
            const R dU = U[1][c] - U[0][c];
            const R fh = (sr * F[0][c] - sl * F[1][c] + sl * sr * dU) * di;
            lFs[0][c] = lF[c] * sr * di;
            lFs[1][c] = -lF[c] * sl * di;
            lU[1][c] = lF[c] * sl * sr * di;
            lU[0][c] = -lF[c] * sl * sr * di;
            lsr += lF[c] * (F[0][c] + sl * dU - fh) * di;
            lsl += lF[c] * (-F[1][c] + sr * dU + fh) * di;
        }
    } else {
        for (int c = 0; c < 5; ++c) lFs[1][c] = lF[c];
    }
    // wave speeds: sl = min(ul, ur) - cmax, sr = max(ul, ur) + cmax
    R* lst[2] = {lL, lR};
    lL[1] += (ml ? lsl : R(0)) + (Ml ? lsr : R(0));
    lR[1] += (ml ? R(0) : lsl) + (Ml ? R(0) : lsr);
    const R lcmax = lsr - lsl;
    R lcf[2] = {cl ? lcmax : R(0), cl ? R(0) : lcmax};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const R r = st[k][0], u = st[k][1], v = st[k][2], w = st[k][3], p = st[k][4], by = st[k][5], bz = st[k][6];
        R lr = R(0), lu = R(0), lv = R(0), lw = R(0), lp = R(0), lby = R(0), lbz = R(0);
        fast_speed_vjp(r, p, bn, by, bz, gamma, lcf[k], lr, lp, lbn, lby, lbz);
        const R* g = lFs[k];
        const R* h = lU[k];
        // U = (r, r u, r v, r w, e)
        lr += h[0] + h[1] * u + h[2] * v + h[3] * w;
        lu += h[1] * r;
        lv += h[2] * r;
        lw += h[3] * r;
        R le = h[4];
        // F0 = r u
        lr += g[0] * u;
        lu += g[0] * r;
        // F1 = r u^2 + pt - bn^2
        lr += g[1] * u * u;
        lu += g[1] * R(2) * r * u;
        R lpt = g[1];
        lbn -= g[1] * R(2) * bn;
        // F2 = r v u - by bn, F3 = r w u - bz bn
        lr += g[2] * v * u + g[3] * w * u;
        lv += g[2] * r * u;
        lw += g[3] * r * u;
        lu += g[2] * r * v + g[3] * r * w;
        lby -= g[2] * bn;
        lbz -= g[3] * bn;
        lbn -= g[2] * by + g[3] * bz;
        // F4 = (e + pt) u - bn vb, vb = u bn + v by + w bz
        le += g[4] * u;
        lpt += g[4] * u;
        lu += g[4] * (e[k] + pt[k]);
        lbn -= g[4] * vb[k];
        const R lvb = -g[4] * bn;
        lu += lvb * bn;
        lbn += lvb * u;
        lv += lvb * by;
        lby += lvb * v;
        lw += lvb * bz;
        lbz += lvb * w;
        // e = p/(gamma-1) + r (u^2 + v^2 + w^2)/2 + b2/2, pt = p + b2/2, b2 = bn^2 + by^2 + bz^2
        lp += le * gm1i + lpt;
        lr += le * R(0.5) * (u * u + v * v + w * w);
        lu += le * r * u;
        lv += le * r * v;
        lw += le * r * w;
        const R lb2 = R(0.5) * (le + lpt);
        lbn += lb2 * R(2) * bn;
        lby += lb2 * R(2) * by;
        lbz += lb2 * R(2) * bz;
        R* o = lst[k];
        o[0] += lr;
        o[1] += lu;
        o[2] += lv;
        o[3] += lw;
        o[4] += lp;
        o[5] += lby;
        o[6] += lbz;
    }
}

// d emf2d: lE -> cotangents of the four corner states (rho, p, ua, ub, Ba, Bb, Be each)
template <typename R>
MHD_HD void emf2d_vjp(const Corner<R>& SW, const Corner<R>& SE, const Corner<R>& NW, const Corner<R>& NE, R gamma,
                      R lE, Corner<R>& gSW, Corner<R>& gSE, Corner<R>& gNW, Corner<R>& gNE) {
    const Corner<R>* st[4] = {&SW, &SE, &NW, &NE};
    Corner<R>* gs[4] = {&gSW, &gSE, &gNW, &gNE};
    R ap[4], am[4], bp[4], bm[4], ca[4], cb[4], ra[4], rb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const Corner<R>& s = *st[k];
        corner_speeds(s, gamma, ca[k], cb[k], ra[k], rb[k]);
        ap[k] = s.ua + ca[k];
        am[k] = s.ua - ca[k];
        bp[k] = s.ub + cb[k];
        bm[k] = s.ub - cb[k];
    }
    // folds with the selected index (-1: the clip at zero won) and what the selected speed came from; a
    // NaN is passed over, as in max0_ and min0_
    struct Pick {
        int k;
        R c, root;
    };
    auto fold_max = [](const R* x, const R* c, const R* r, Pick& p) {
        R m = x[0];
        p = {0, c[0], r[0]};
#pragma unroll
        for (int j = 1; j < 4; ++j)
            if (greater_(x[j], m) || !number_(m)) {
                m = x[j];
                p = {j, c[j], r[j]};
            }
        if (!nonneg_(m)) {
            m = R(0);
            p.k = -1;
        }
        return m;
    };
    auto fold_min = [](const R* x, const R* c, const R* r, Pick& p) {
        R m = x[0];
        p = {0, c[0], r[0]};
#pragma unroll
        for (int j = 1; j < 4; ++j)
            if (greater_(m, x[j]) || !number_(m)) {
                m = x[j];
                p = {j, c[j], r[j]};
            }
        if (positive_(m)) {
            m = R(0);
            p.k = -1;
        }
        return m;
    };
    Pick kE, kW, kN, kS;
    const R sE = fold_max(ap, ca, ra, kE), sW = fold_min(am, ca, ra, kW), sN = fold_max(bp, cb, rb, kN),
            sS = fold_min(bm, cb, rb, kS);
    const R da = sE - sW, db = sN - sS;
    R e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) e[k] = st[k]->ua * st[k]->Bb - st[k]->ub * st[k]->Ba;
    // E = [sE X - sW Y] / da + sE sW / da jb - sN sS / db ja, X = (sN e0 - sS e2) / db and Y = (sN e1 -
    // sS e3) / db, and the same with a and b exchanged; so with 1 - sE / da = -sW / da, in which nothing
    // cancels, dE/dsE = -sW (X - Y + sW jb) / da^2, dE/dsW = sE (X - Y + sE jb) / da^2, and alike along b
    const R ida = rcp_near_(da), idb = rcp_near_(db), q = da * db;
    const R jb = SE.Bb - SW.Bb, ja = NW.Ba - SW.Ba;
    const R g_jb = lE * quot_(sE * sW, da, ida), g_ja = -lE * quot_(sN * sS, db, idb);
    gSE.Bb += g_jb;
    gSW.Bb -= g_jb;
    gNW.Ba += g_ja;
    gSW.Ba -= g_ja;
    const R xy = (sN * (e[0] - e[1]) - sS * (e[2] - e[3])) * idb, zt = (sE * (e[0] - e[2]) - sW * (e[1] - e[3])) * ida;
    const R ga = lE * ida * ida, gb = lE * idb * idb;
    const R g_sE = -ga * sW * (xy + sW * jb), g_sW = ga * sE * (xy + sE * jb);
    const R g_sN = -gb * sS * (zt - sS * ja), g_sS = gb * sN * (zt - sN * ja);
    const R g_num = quot_(lE, q, rcp_near_(q));
    const R g_e[4] = {g_num * sE * sN, -g_num * sW * sN, -g_num * sE * sS, g_num * sW * sS};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        gs[k]->ua += g_e[k] * st[k]->Bb;
        gs[k]->Bb += g_e[k] * st[k]->ua;
        gs[k]->ub -= g_e[k] * st[k]->Ba;
        gs[k]->Ba -= g_e[k] * st[k]->ub;
    }
    // Each of the four speeds comes from one corner: its velocity and fast speed there.  The corner
    // is selected by value, the result added by testing every corner, so that every index is a
    // compile-time constant and the corner cotangents stay in registers (four reverse fast speeds
    // instead of one per corner and direction).
    auto speed = [&](const Pick& pick, R g, bool alongb, R sgn) {
        const int k = pick.k;
        if (k < 0) return;
        Corner<R> s = *st[0];
#pragma unroll
        for (int j = 1; j < 4; ++j)
            if (j == k) s = *st[j];
        R lrho = R(0), lp = R(0), lbn = R(0), lbt = R(0), lbe = R(0);
        const R bn = alongb ? s.Bb : s.Ba, bt = alongb ? s.Ba : s.Bb;
        if constexpr (sizeof(R) == 8)
            fast_h_vjp(s.rho, s.p, bn, bt, s.Be, gamma, pick.c, pick.root, sgn * g, lrho, lp, lbn, lbt, lbe);
        else
            fast_speed_vjp(s.rho, s.p, bn, bt, s.Be, gamma, sgn * g, lrho, lp, lbn, lbt, lbe);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j != k) continue;
            (alongb ? gs[j]->ub : gs[j]->ua) += g;
            gs[j]->rho += lrho;
            gs[j]->p += lp;
            (alongb ? gs[j]->Bb : gs[j]->Ba) += lbn;
            (alongb ? gs[j]->Ba : gs[j]->Bb) += lbt;
            gs[j]->Be += lbe;
        }
    };
    speed(kE, g_sE, false, R(1));
    speed(kW, g_sW, false, R(-1));
    speed(kN, g_sN, true, R(1));
    speed(kS, g_sS, true, R(-1));
}

}  // namespace mhd
