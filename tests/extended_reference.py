"""The face flux and the edge EMF with their derivatives in extended precision (numpy's longdouble, 64
bits of significand or more), for measuring the rounding error of the double-precision code, and
random rows to measure it on."""
import numpy as np

LD = np.longdouble
GAMMA, GAMMA_M1_INV = LD(np.float64(5.0 / 3.0)), LD(1.5)


class Dual:
    """Values v (n,) and their derivatives d (m, n) with respect to m inputs."""

    def __init__(self, v, d=0):
        self.v, self.d = v, d

    @staticmethod
    def of(x):
        return x if isinstance(x, Dual) else Dual(x)

    def __add__(a, b):
        b = Dual.of(b)
        return Dual(a.v + b.v, a.d + b.d)

    def __neg__(a):
        return Dual(-a.v, -a.d)

    def __sub__(a, b):
        return a + -Dual.of(b)

    def __mul__(a, b):
        b = Dual.of(b)
        return Dual(a.v * b.v, a.d * b.v + a.v * b.d)

    def __truediv__(a, b):
        b = Dual.of(b)
        q = a.v / b.v
        return Dual(q, (a.d - q * b.d) / b.v)

    __radd__, __rmul__ = __add__, __mul__


def sqrt(a):
    r = np.sqrt(a.v)
    return Dual(r, a.d / (2 * r))


def where(m, a, b):
    return Dual(np.where(m, a.v, b.v), np.where(m, a.d, b.d))


def larger(a, b):
    return where(a.v >= b.v, a, b)


def smaller(a, b):
    return where(a.v <= b.v, a, b)


def inputs(x):
    """The columns of x (n, m), each its own input."""
    x = x.astype(LD)
    return [Dual(x[:, k], np.eye(x.shape[1], dtype=LD)[:, k:k + 1] * np.ones(len(x), LD)) for k in range(x.shape[1])]


def fast_speed(rho, p, bn, bt2):
    c, n, t = GAMMA * p / rho, bn * bn / rho, bt2 / rho
    return sqrt(LD(0.5) * (c + n + t + sqrt((c - n) * (c - n) + t * (2 * (c + n) + t))))


def face_flux(x, hll):
    """HLLD (or HLL) flux of the states x[:7], x[7:14] (rho, u, v, w, p, b1, b2) and the field x[14];
    no state of the rows is degenerate."""
    def side(S):
        rho, u, v, w, p, b1, b2 = S
        bb = bn * bn + b1 * b1 + b2 * b2
        pt = p + LD(0.5) * bb
        E = p * GAMMA_M1_INV + LD(0.5) * (rho * (u * u + v * v + w * w) + bb)
        vb = u * bn + v * b1 + w * b2
        F = [rho * u, rho * u * u + pt - bn * bn, rho * u * v - bn * b1, rho * u * w - bn * b2, (E + pt) * u - bn * vb]
        return pt, E, vb, F, fast_speed(rho, p, bn, b1 * b1 + b2 * b2), [rho, rho * u, rho * v, rho * w, E]

    def star(S, W, pt, E, vb):
        rho, u, v, w, _, b1, b2 = W
        rs, D = rho * (S - u) / (S - SM), rho * (S - u) * (S - SM) - bn * bn
        nu, nb = bn * (SM - u) / D, (rho * (S - u) * (S - u) - bn * bn) / D
        vs, ws, c1, c2 = v - b1 * nu, w - b2 * nu, b1 * nb, b2 * nb
        vbs = SM * bn + vs * c1 + ws * c2
        Es = ((S - u) * E - pt * u + ps * SM + bn * (vb - vbs)) / (S - SM)
        return rs, vs, ws, c1, c2, vbs, Es, [rs, rs * SM, rs * vs, rs * ws, Es]
    L, R, bn = x[:7], x[7:14], x[14]
    (pl, El, vbl, FL, cl, UL), (pr, Er, vbr, FR, cr, UR) = side(L), side(R)
    cm = larger(cl, cr)
    SL, SR = smaller(L[1], R[1]) - cm, larger(L[1], R[1]) + cm
    if hll:
        mid = [(SR * f - SL * g + SL * SR * (v - u)) / (SR - SL) for f, g, u, v in zip(FL, FR, UL, UR)]
        return [where(SL.v >= 0, f, where(SR.v >= 0, h, g)) for f, h, g in zip(FL, mid, FR)]
    dl, dr = (SL - L[1]) * L[0], (SR - R[1]) * R[0]
    SM = (dr * R[1] - dl * L[1] - pr + pl) / (dr - dl)
    ps = (dr * pl - dl * pr + dl * dr * (R[1] - L[1])) / (dr - dl)
    A, B = star(SL, L, pl, El, vbl), star(SR, R, pr, Er, vbr)
    ql, qr, sg = sqrt(A[0]), sqrt(B[0]), np.sign(bn.v)
    TL, TR = SM - bn * sg / ql, SM + bn * sg / qr
    vd = [(ql * A[k] + qr * B[k] + (B[k + 2] - A[k + 2]) * sg) / (ql + qr) for k in (1, 2)]
    bd = [(ql * B[k + 2] + qr * A[k + 2] + ql * qr * (B[k] - A[k]) * sg) / (ql + qr) for k in (1, 2)]
    vbd = SM * bn + vd[0] * bd[0] + vd[1] * bd[1]
    DL = [A[0], A[0] * SM, A[0] * vd[0], A[0] * vd[1], A[6] - ql * (A[5] - vbd) * sg]
    DR = [B[0], B[0] * SM, B[0] * vd[0], B[0] * vd[1], B[6] + qr * (B[5] - vbd) * sg]
    out = []
    for k in range(5):
        fl, fr = FL[k] + SL * (A[7][k] - UL[k]), FR[k] + SR * (B[7][k] - UR[k])
        f = where(SR.v >= 0, fr, FR[k])
        f = where(TR.v >= 0, fr + TR * (DR[k] - B[7][k]), f)
        f = where(SM.v >= 0, fl + TL * (DL[k] - A[7][k]), f)
        out.append(where(SL.v >= 0, FL[k], where(TL.v >= 0, fl, f)))
    return out


def edge_emf(corners):
    """Two-dimensional HLL EMF of four corners (rho, p, ua, ub, Ba, Bb, Be)."""
    ap, am, bp, bm, e = [], [], [], [], []
    for rho, p, ua, ub, Ba, Bb, Be in corners:
        ca, cb = fast_speed(rho, p, Ba, Bb * Bb + Be * Be), fast_speed(rho, p, Bb, Ba * Ba + Be * Be)
        for speeds, s in ((ap, ua + ca), (am, ua - ca), (bp, ub + cb), (bm, ub - cb), (e, ua * Bb - ub * Ba)):
            speeds.append(s)

    def fold(pick, speeds):
        m = speeds[0]
        for s in speeds[1:]:
            m = pick(m, s)
        return pick(m, 0 * m)
    sE, sW, sN, sS = fold(larger, ap), fold(smaller, am), fold(larger, bp), fold(smaller, bm)
    da, db = sE - sW, sN - sS
    num = sE * sN * e[0] - sE * sS * e[2] - sW * sN * e[1] + sW * sS * e[3]
    return num / (da * db) + sE * sW / da * (corners[1][5] - corners[0][5]) - sN * sS / db * (corners[2][4] - corners[0][4])


def related_states(rng, n, count):
    """`count` states (rho, u, v, w, p, b1, b2) per row that differ by 1e-4 to 0.3, as the states around a
    face or an edge do."""
    base = np.stack([np.exp(0.35 * rng.normal(size=n)), *(0.6 * rng.normal(size=(3, n))),
                     np.exp(0.35 * rng.normal(size=n)), *(0.25 * rng.normal(size=(2, n)))])
    d, out = 10 ** rng.uniform(-4, -0.5, n), []
    for _ in range(count):
        s = base.copy()
        s[[0, 4]] *= np.exp(d * rng.normal(size=(2, n)))
        s[[1, 2, 3, 5, 6]] += d * rng.normal(size=(5, n)) * np.array([1, 1, 1, 0.5, 0.5])[:, None]
        out.append(s.T)
    return out


def face_rows(n, seed):
    rng = np.random.default_rng(seed)
    return np.concatenate(related_states(rng, n, 2) + [0.25 * rng.normal(size=(n, 1)), rng.normal(size=(n, 5))], axis=1)


def edge_rows(n, seed):
    rng = np.random.default_rng(seed)
    corners = [s[:, [0, 4, 1, 2, 5, 6, 3]] * np.array([1, 1, 1, 1, 1, 1, 0.4]) for s in related_states(rng, n, 4)]
    return np.concatenate(corners + [rng.normal(size=(n, 1))], axis=1)
