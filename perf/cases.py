"""The calls a user of the MHD bunch library makes, as cases whose time is measured.

A case is a dict of plain values.  `kind` says which call it is:

  march    time steps of a device-resident bunch, at the CFL step of each state: a captured
           graph of `steps` steps (launch "graph") or as many eager steps (launch "eager")
  grad     one fixed-dt step and its adjoint through torch autograd (MHDStep)
  rollout  a checkpointed differentiable run of `steps` steps and its gradient (rollout)
  async    asynchronous per-patch time stepping over `span` CFL steps of the start state
  stream   `steps` steps of a state held in pinned host memory, streamed through the GPU

and the other keys give the box: cells per patch (nx, ny, nz), patches per axis (cx, cy, cz),
real (32 or 64 bits), riemann (0 HLLD, 1 HLL), limiter (0 minmod, 1 MC), outflow (1: the
ends of the last active axis are zero-gradient, 0: periodic).  layers > 0 makes a ragged
box instead: z-layers of 16^3, 24^3 and 32^3 patches under `side` x `side` cells.

Inputs are smooth seeded fields (a few random Fourier modes per variable): density and
pressure vary by some tens of per cent, the flow is subsonic to transonic and the face field
is the discrete curl of an edge potential plus a mean field, so it is divergence free.  A
march is fed its own result: passes on one state go on with the flow, as a run does.

`exact` restates the scheme on whole boxes in 64-bit torch arithmetic.
"""
import math

import numpy as np
import torch

from paper_2508_09568_gb300 import capi
from paper_2508_09568_gb300.autograd import MHDStep, rollout
from paper_2508_09568_gb300.bunch import MHDBunch
from paper_2508_09568_gb300.workloads import BC_OUTFLOW, BC_PERIODIC, Geometry, uniform_geometry

GAMMA, COURANT = 5.0 / 3.0, 0.8
DEV = "cuda:0"
RAGGED = (16, 24, 32)


def _case(name, kind, n, c, real=32, steps=1, launch="graph", riemann=0, limiter=0, outflow=0, span=0.0, layers=0,
          side=0):
    d = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], cx=c[0], cy=c[1], cz=c[2], real=real, steps=steps, launch=launch,
             riemann=riemann, limiter=limiter, outflow=outflow, span=span, layers=layers, side=side)
    return dict(d, name=name) if name else d


def listed():
    return [
        # a 1D shock-tube sized bunch (256 cells as 16 patches): the smallest call, where the
        # latency of a launch and of a tile counts
        _case("tube256_f64", "march", (16, 1, 1), (16, 1, 1), real=64, steps=8, outflow=1),
        # the 512^2 vortex box as 256 patches of 32^2 (the 2D test problem), in a graph
        _case("vortex512_f32", "march", (32, 32, 1), (16, 16, 1), steps=4),
        # the same box in double precision stepped eagerly, as the accuracy runs are
        _case("vortex512_f64", "march", (32, 32, 1), (16, 16, 1), real=64, steps=2, launch="eager"),
        # the benchmark: a 512^3 box as 4096 patches of 32^3
        _case("box512_f32", "march", (32, 32, 32), (16, 16, 16)),
        # the paper's own patch size (24^3 with three guard cells), 1000 patches
        _case("box240_p24_f32", "march", (24, 24, 24), (10, 10, 10), steps=2),
        # odd patch sizes whose planes are not 16-byte multiples, the other face-flux solver
        # and limiter, an open box
        _case("box_odd_hll_mc_f32", "march", (21, 28, 17), (5, 4, 6), steps=2, launch="eager", riemann=1, limiter=1,
              outflow=1),
        # a 3D box in double precision (check runs)
        _case("box128_f64", "march", (32, 32, 32), (4, 4, 4), real=64),
        # 1566 patches of three sizes in one bunch, each size with its own tile
        _case("ragged288_f32", "march", (0, 0, 0), (0, 0, 0), layers=11, side=288),
        # one differentiable step of the 64^3 adjoint box, forward and backward
        _case("grad64_f32", "grad", (32, 32, 32), (2, 2, 2)),
        # a checkpointed rollout in double precision, forward and backward
        _case("rollout64_f64", "rollout", (32, 32, 32), (2, 2, 2), real=64, steps=4),
        # patches at their own times (DISPATCH's mode)
        _case("async256_f32", "async", (32, 32, 32), (8, 8, 8), span=1.5),
        # a box kept in host memory and streamed through the GPU every step
        _case("stream256_f32", "stream", (32, 32, 32), (8, 8, 8), steps=2),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["march"] * 6 + ["grad", "rollout", "async", "stream"])
    real = rng.choice([32, 32, 64])
    opt = dict(riemann=rng.choice([0, 0, 1]), limiter=rng.choice([0, 0, 1]), outflow=rng.choice([0, 0, 1]))
    if kind != "march":
        n = [rng.randint(8, 36) for _ in range(3)]
        most = 40_000 if real == 64 else 4_000_000 if kind in ("async", "stream") else 400_000
        c = [1, 1, 1]
        for d in rng.sample(range(3), 3):
            c[d] = max(1, min(6, _loguniform(rng, 1, 8), most // (math.prod(n) * math.prod(c))))
        return _case("", kind, n, c, real=real, steps=rng.randint(2, 4) if kind in ("rollout", "stream") else 1,
                     span=rng.choice([0.75, 1.5, 2.0]) if kind == "async" else 0.0, **opt)
    dim = rng.choice([1, 2, 3, 3, 3, 3])
    steps, launch = rng.randint(1, 4), rng.choice(["graph", "graph", "eager"])
    if dim == 3 and rng.random() < 0.2:
        return _case("", kind, (0, 0, 0), (0, 0, 0), layers=rng.randint(3, 9), side=rng.choice([96, 192]), steps=steps,
                     launch=launch, riemann=opt["riemann"], limiter=opt["limiter"])
    n = [rng.randint(8, 40) if d < dim else 1 for d in range(3)]
    total = _loguniform(rng, *{1: (64, 4096), 2: (4096, 1 << 21), 3: (8192, 60_000_000)}[dim])
    if real == 64:
        total = min(total, 2_000_000)
    side = max(1.0, total / math.prod(n)) ** (1.0 / dim)
    c = [max(1, int(round(side * rng.uniform(0.7, 1.4)))) if d < dim else 1 for d in range(3)]
    return _case("", kind, n, c, real=real, steps=steps, launch=launch, **opt)


# ---------------------------------------------------------------------------------------------------
# boxes and inputs
# ---------------------------------------------------------------------------------------------------
def _geometry(case):
    if case["layers"]:
        side, sizes, origins, z = case["side"], [], [], 0
        for k in range(case["layers"]):
            s = RAGGED[(k * 2) % 3]
            for j in range(side // s):
                for i in range(side // s):
                    sizes.append([s, s, s])
                    origins.append([i * s, j * s, z])
            z += s
        return Geometry(np.array(sizes), np.array(origins), [side, side, z], [1.0 / side] * 3, [[BC_PERIODIC] * 2] * 3)
    n = [case["nx"], case["ny"], case["nz"]]
    N = [n[0] * case["cx"], n[1] * case["cy"], n[2] * case["cz"]]
    last = max(d for d in range(3) if n[d] > 1)
    bc = [[BC_OUTFLOW if case["outflow"] and d == last else BC_PERIODIC] * 2 for d in range(3)]
    return uniform_geometry(N, n, dx=[1.0 / v if v > 1 else 1.0 for v in N], bc=bc)


def _runs(geom):
    """Runs of equal patches: (first patch, count, first element, (X, Y, Z) padded)."""
    out, p, offs = [], 0, geom.offsets()
    while p < geom.npatch:
        q = p
        while q < geom.npatch and np.array_equal(geom.patch_n[q], geom.patch_n[p]) and (
                geom.uniform() or geom.origin[q][2] == geom.origin[p][2]):
            q += 1
        out.append((p, q - p, int(offs[p]), geom.padded(p)))
        p = q
    return out


def _owned(flat, geom):
    """The owned cells of a state as one view per run of equal patches: [P][8][nz][ny][nx]."""
    g, out = [int(v) for v in geom.gvec], []
    for p, count, off, (Z, Y, X) in _runs(geom):
        v = flat[off:off + count * 8 * Z * Y * X].view(count, 8, Z, Y, X)
        out.append(v[:, :, g[2]:Z - g[2], g[1]:Y - g[1], g[0]:X - g[0]])
    return out


def _cut(U, geom):
    """The owned cells of a global field (8, Nz, Ny, Nx), laid out as _owned gives them."""
    out = []
    for p, count, off, _ in _runs(geom):
        nx, ny, nz = (int(v) for v in geom.patch_n[p])
        oz = int(geom.origin[p][2])
        cx, cy = int(geom.domain[0]) // nx, int(geom.domain[1]) // ny
        cz = count // (cx * cy)
        v = U[:, oz:oz + cz * nz].reshape(8, cz, nz, cy, ny, cx, nx)
        out.append(v.permute(1, 3, 5, 0, 2, 4, 6).reshape(count, 8, nz, ny, nx))
    return out


def _smooth(rng, N, amp, modes=4, kmax=4):
    """A few random Fourier modes on an (Nz, Ny, Nx) grid, separably."""
    out = None
    for _ in range(modes):
        k = [int(rng.integers(-kmax, kmax + 1)) if N[d] > 1 else 0 for d in range(3)]
        ph, a = rng.uniform(0, 2 * math.pi), amp * rng.uniform(0.5, 1.0) / math.sqrt(modes)
        e = [torch.exp(2j * math.pi * k[d] * torch.arange(N[d], device=DEV, dtype=torch.float64) / N[d]) for d in range(3)]
        e = [v.to(torch.complex64) for v in e]
        plane = (e[1][:, None] * e[0][None, :]) * complex(a * math.cos(ph), a * math.sin(ph))
        f = e[2].real[:, None, None] * plane.imag + e[2].imag[:, None, None] * plane.real
        out = f if out is None else out.add_(f)
    return out


def _fields(case, geom, seed):
    """The start state (8, Nz, Ny, Nx) on the GPU in the case's precision."""
    N, dx, rng = [int(v) for v in geom.domain], geom.dx, np.random.default_rng([int(seed), 977])
    dt = torch.float32 if case["real"] == 32 else torch.float64
    U = torch.empty((8, N[2], N[1], N[0]), device=DEV, dtype=dt)
    rho = torch.exp(_smooth(rng, N, 0.35)).to(dt)
    E = torch.exp(_smooth(rng, N, 0.35)).to(dt).div_(GAMMA - 1.0)
    U[0] = rho
    for c in range(3):
        v = _smooth(rng, N, 0.6).to(dt)
        U[1 + c] = rho * v
        E += 0.5 * rho * v * v
    h = 0.25 / (2 * math.pi * 3)
    for c, mean in enumerate((0.2, 0.1, 0.05)):
        U[5 + c] = mean
    for a in range(3):   # edge potential along a: adds +d_b A to face field c, -d_c A to face field b
        b, c = (a + 1) % 3, (a + 2) % 3
        A = _smooth(rng, N, h).to(dt)
        if N[b] > 1:
            U[5 + c] += (torch.roll(A, -1, 2 - b) - A) / float(dx[b])
        if N[c] > 1:
            U[5 + b] -= (torch.roll(A, -1, 2 - c) - A) / float(dx[c])
    for c in range(3):
        m = 0.5 * (U[5 + c] + torch.roll(U[5 + c], -1, 2 - c))
        E += 0.5 * m * m
    U[4] = E
    return U


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.geom = case, _geometry(case)
    dtype = torch.float32 if case["real"] == 32 else torch.float64
    s.b = MHDBunch(s.geom, dtype=dtype, gamma=GAMMA, courant=COURANT, limiter=case["limiter"], riemann=case["riemann"],
                   device=DEV)
    U = _fields(case, s.geom, seed)
    torch.cuda.synchronize()
    for view, part in zip(_owned(s.b.buf[0], s.geom), _cut(U, s.geom)):
        view.copy_(part)
    kind = case["kind"]
    if kind == "stream":
        s.host = torch.cat([p.reshape(-1) for p in _cut(U, s.geom)]).cpu().pin_memory()
    del U
    torch.cuda.synchronize()
    s.views = [_owned(t, s.geom) for t in s.b.buf]
    if kind == "march":
        s.dts = torch.zeros(case["steps"], dtype=torch.float64, device=DEV)
        s.dt = [s.dts[k:k + 1] for k in range(case["steps"])]
        if case["layers"]:
            s.b.set_mode(capi.MHD_MODE_MIXED)
            s.b.autotune()
        if case["launch"] == "graph":
            s.b.graph_capture(case["steps"], s.dts)
    elif kind in ("grad", "rollout"):
        # the start state as a leaf (its ghost cells are filled by each step) and the gradient
        # of a loss with respect to the result (zero on the ghost cells)
        s.b.fill_guards()
        s.fixed_dt = 0.5 * s.b.cfl_dt()
        s.U = s.b.buf[0].clone().requires_grad_(True)
        s.lam = torch.zeros_like(s.b.buf[0])
        rng = torch.Generator(device=DEV).manual_seed(int(seed) + 5)
        for v in _owned(s.lam, s.geom):
            v.copy_(torch.randn(v.shape, generator=rng, device=DEV, dtype=dtype))
        if kind == "rollout":
            s.b.twin()
    elif kind == "async":
        s.b.fill_guards()
        s.span = case["span"] * s.b.cfl_dt()
    torch.cuda.synchronize()
    return s


def run(s):
    case, b = s.case, s.b
    kind = case["kind"]
    if kind == "march":
        if case["launch"] == "graph":
            b.graph_launch()
        else:
            for dt in s.dt:
                b.fill_cfl_device(dt)
                b.step_device_dt(dt)
        return {"state": s.views[0 if b.current() is b.buf[0] else 1], "dt": s.dts}
    if kind in ("grad", "rollout"):
        if kind == "grad":
            out = MHDStep.apply(s.U, b, s.fixed_dt)
        else:
            out = rollout(s.U, b, s.fixed_dt, case["steps"], 2)
        (grad,) = torch.autograd.grad(out, s.U, s.lam)
        return {"state": _owned(out.detach(), s.geom), "grad": _owned(grad, s.geom)}
    if kind == "async":
        b.advance_async(s.span)
        return {"state": s.views[0 if b.current() is b.buf[0] else 1]}
    t = b.advance_streamed_interior(s.host, case["steps"], 8)
    return {"state": s.host, "t": t}


def work(case):
    geom = _geometry(case)
    cells, rb = geom.interior_cells(), case["real"] // 8
    flops = (1100, 2000, 2703 if case["riemann"] else 3255)[int(sum(geom.active)) - 1]
    steps = case["span"] if case["kind"] == "async" else case["steps"]
    state = 8 * rb * cells
    if case["kind"] in ("grad", "rollout"):
        # every step forward once and its adjoint (state and cotangent in, cotangent out), at
        # the arithmetic of the recomputed step and its reverse
        return {"bytes": 5.0 * state * steps, "flops": 4.0 * flops * cells * steps}
    return {"bytes": 2.0 * state * steps, "flops": float(flops) * cells * steps}


# ---------------------------------------------------------------------------------------------------
# the scheme on a whole box in 64 bits
# ---------------------------------------------------------------------------------------------------
def _m(a, d):
    return torch.roll(a, 1, 2 - d)


def _p(a, d):
    return torch.roll(a, -1, 2 - d)


def _limited(q, d, limiter):
    a, b = q - _m(q, d), _p(q, d) - q
    pick = torch.where(a.abs() <= b.abs(), a, b)
    if limiter:
        c, pick = 0.5 * (a + b), 2 * pick
        pick = torch.where(c.abs() <= pick.abs(), c, pick)
    return torch.where(a * b > 0, pick, torch.zeros_like(a))


def _max(a, b):
    return torch.where(a >= b, a, b)


def _min(a, b):
    return torch.where(a <= b, a, b)


def _fast(rho, P, bn, bt2):
    """Fast speed, the discriminant as a sum of terms that are not negative."""
    c, n, t = GAMMA * P / rho, bn * bn / rho, bt2 / rho
    disc = (c - n) ** 2 + t * (2 * (c + n) + t)
    pos = disc > 0
    root = torch.where(pos, torch.sqrt(torch.where(pos, disc, torch.ones_like(disc))), torch.zeros_like(disc))
    return torch.sqrt(0.5 * (c + n + t + root))


def _prims(U):
    rho = U[0]
    vel = [U[1 + d] / rho for d in range(3)]
    B = [0.5 * (U[5 + d] + _p(U[5 + d], d)) for d in range(3)]
    P = (GAMMA - 1) * (U[4] - 0.5 * rho * sum(v * v for v in vel) - 0.5 * sum(b * b for b in B))
    return [rho, *vel, P, *B]


def _flux(L, R, bn, hll, eps):
    """HLLD (or HLL) flux of (rho, m_n, m_t1, m_t2, E) between the states (rho, u, v, w, P, b1, b2)."""
    def side(S):
        rho, u, v, w, P, b1, b2 = S
        bb = bn * bn + b1 * b1 + b2 * b2
        pt = P + 0.5 * bb
        E = P / (GAMMA - 1) + 0.5 * rho * (u * u + v * v + w * w) + 0.5 * bb
        vb = u * bn + v * b1 + w * b2
        F = [rho * u, rho * u * u + pt - bn * bn, rho * u * v - bn * b1, rho * u * w - bn * b2, (E + pt) * u - bn * vb]
        return pt, E, vb, F, _fast(rho, P, bn, b1 * b1 + b2 * b2), [rho, rho * u, rho * v, rho * w, E]
    (pl, El, vbl, FL, cl, UL), (pr, Er, vbr, FR, cr, UR) = side(L), side(R)
    cm = _max(cl, cr)
    SL, SR = _min(L[1], R[1]) - cm, _max(L[1], R[1]) + cm
    if hll:
        mid = [(SR * f - SL * g + SL * SR * (v - u)) / (SR - SL) for f, g, u, v in zip(FL, FR, UL, UR)]
        return [torch.where(SL >= 0, f, torch.where(SR >= 0, h, g)) for f, h, g in zip(FL, mid, FR)]
    dl, dr = (SL - L[1]) * L[0], (SR - R[1]) * R[0]
    SM = (dr * R[1] - dl * L[1] - pr + pl) / (dr - dl)
    ps = (dr * pl - dl * pr + dl * dr * (R[1] - L[1])) / (dr - dl)

    def star(S, W, pt, E, vb):
        rho, u, v, w, _, b1, b2 = W
        rs = rho * (S - u) / (S - SM)
        D = rho * (S - u) * (S - SM) - bn * bn
        deg = D.abs() <= eps * bn * bn
        Di = torch.where(deg, torch.zeros_like(D), 1 / torch.where(deg, torch.ones_like(D), D))
        nu, nb = bn * (SM - u) * Di, (rho * (S - u) ** 2 - bn * bn) * Di
        v1, w1 = v - b1 * nu, w - b2 * nu
        c1, c2 = torch.where(deg, b1, b1 * nb), torch.where(deg, b2, b2 * nb)
        vbs = SM * bn + v1 * c1 + w1 * c2
        Es = ((S - u) * E - pt * u + ps * SM + bn * (vb - vbs)) / (S - SM)
        return rs, v1, w1, c1, c2, vbs, Es, [rs, rs * SM, rs * v1, rs * w1, Es]
    A, B = star(SL, L, pl, El, vbl), star(SR, R, pr, Er, vbr)
    ql, qr = torch.sqrt(A[0]), torch.sqrt(B[0])
    sgn = torch.sign(bn)
    TL, TR = SM - bn.abs() / ql, SM + bn.abs() / qr
    vd = [(ql * A[k] + qr * B[k] + (B[k + 2] - A[k + 2]) * sgn) / (ql + qr) for k in (1, 2)]
    bd = [(ql * B[k + 2] + qr * A[k + 2] + ql * qr * (B[k] - A[k]) * sgn) / (ql + qr) for k in (1, 2)]
    vbd = SM * bn + vd[0] * bd[0] + vd[1] * bd[1]
    DL = [A[0], A[0] * SM, A[0] * vd[0], A[0] * vd[1], A[6] - ql * (A[5] - vbd) * sgn]
    DR = [B[0], B[0] * SM, B[0] * vd[0], B[0] * vd[1], B[6] + qr * (B[5] - vbd) * sgn]
    out = []
    for k in range(5):
        fl, fr = FL[k] + SL * (A[7][k] - UL[k]), FR[k] + SR * (B[7][k] - UR[k])
        f = torch.where(SR >= 0, fr, FR[k])
        f = torch.where(TR >= 0, fr + TR * (DR[k] - B[7][k]), f)
        f = torch.where(SM >= 0, fl + TL * (DL[k] - A[7][k]), f)
        f = torch.where(TL >= 0, fl, f)
        out.append(torch.where(SL >= 0, FL[k], f))
    return out


def _rate(U, dx, act):
    W = _prims(U)
    B2 = sum(b * b for b in W[5:])
    return sum((W[1 + d].abs() + _fast(W[0], W[4], W[5 + d], B2 - W[5 + d] ** 2)) / dx[d] for d in range(3) if act[d])


def _advance(U, dt, dx, act, limiter, hll, eps):
    """One step of a padded box; the outermost three layers of the result are not meaningful."""
    zero = torch.zeros_like(U[0])
    q, bf, h = _prims(U), [U[5], U[6], U[7]], 0.5 * dt
    S = [[_limited(w, d, limiter) if act[d] else zero for w in q] for d in range(3)]
    T = [[_limited(bf[c], d, limiter) if act[d] and d != c else zero for d in range(3)] for c in range(3)]

    def mean4(w, a, b):
        w = w + _m(w, a)
        return 0.25 * (w + _m(w, b))

    def curl(E, c):
        a, b = (c + 1) % 3, (c + 2) % 3
        t = zero
        if act[a]:
            t = t + (_p(E[b], a) - E[b]) / dx[a]
        if act[b]:
            t = t - (_p(E[a], b) - E[a]) / dx[b]
        return t
    E0 = []
    for e in range(3):
        a, b = (e + 1) % 3, (e + 2) % 3
        E0.append(mean4(q[1 + a], a, b) * 0.5 * (bf[b] + _m(bf[b], a)) - mean4(q[1 + b], a, b) * 0.5 * (bf[a] + _m(bf[a], b)))
    bh = [bf[c] + h * curl(E0, c) for c in range(3)]
    D = [[w / dx[d] for w in S[d]] for d in range(3)]
    div = D[0][1] + D[1][2] + D[2][3]

    def adv(k):
        return q[1] * D[0][k] + q[2] * D[1][k] + q[3] * D[2][k]
    Wh = [q[0] - h * (adv(0) + q[0] * div), None, None, None, q[4] - h * (adv(4) + GAMMA * q[4] * div)]
    for c in range(3):
        a, b = (c + 1) % 3, (c + 2) % 3
        force = D[c][4] + q[5 + a] * (D[c][5 + a] - D[a][5 + c]) + q[5 + b] * (D[c][5 + b] - D[b][5 + c])
        Wh[1 + c] = q[1 + c] - h * (adv(1 + c) + force / q[0])
    Wh += [0.5 * (bh[c] + _p(bh[c], c)) for c in range(3)]
    dU = [zero] * 5
    for d in range(3):
        if act[d]:
            t1, t2 = (d + 1) % 3, (d + 2) % 3
            ks = [0, 1 + d, 1 + t1, 1 + t2, 4, 5 + t1, 5 + t2]
            F = _flux([_m(Wh[k] + 0.5 * S[d][k], d) for k in ks], [Wh[k] - 0.5 * S[d][k] for k in ks], bh[d], hll, eps)
            for k, f in zip((0, 1 + d, 1 + t1, 1 + t2, 4), F):
                dU[k] = dU[k] - dt / dx[d] * (_p(f, d) - f)
    E1 = []
    for e in range(3):
        a, b = (e + 1) % 3, (e + 2) % 3
        if not (act[a] or act[b]):
            E1.append(zero)
            continue
        st = {}
        for sa in (1, -1):
            for sb in (1, -1):
                w = [Wh[k] + 0.5 * (sa * S[a][k] + sb * S[b][k]) for k in (0, 4, 1 + a, 1 + b, 5 + e)]
                fa, fb = bh[a] + 0.5 * sb * T[a][b], bh[b] + 0.5 * sa * T[b][a]
                fa = fa if sa < 0 else _p(bh[a], a) + 0.5 * sb * _p(T[a][b], a)
                fb = fb if sb < 0 else _p(bh[b], b) + 0.5 * sa * _p(T[b][a], b)
                w = w + [fa, fb]
                if sa > 0:
                    w = [_m(x, a) for x in w]
                if sb > 0:
                    w = [_m(x, b) for x in w]
                st[sa, sb] = w   # (1, 1): SW of the edge, (-1, 1): SE, (1, -1): NW, (-1, -1): NE
        order, lim = [(1, 1), (-1, 1), (1, -1), (-1, -1)], []
        for k, Bn, Bt in ((2, 5, 6), (3, 6, 5)):
            up = dn = None
            for key in order:
                w = st[key]
                cf = _fast(w[0], w[1], w[Bn], w[Bt] ** 2 + w[4] ** 2)
                up = w[k] + cf if up is None else _max(up, w[k] + cf)
                dn = w[k] - cf if dn is None else _min(dn, w[k] - cf)
            lim += [_max(up, zero), _min(dn, zero)]
        sE, sW, sN, sS = lim
        e4 = [st[key][2] * st[key][6] - st[key][3] * st[key][5] for key in order]
        num = sE * sN * e4[0] - sE * sS * e4[2] - sW * sN * e4[1] + sW * sS * e4[3]
        E1.append(num / ((sE - sW) * (sN - sS)) + sE * sW / (sE - sW) * (st[-1, 1][6] - st[1, 1][6])
                  - sN * sS / (sN - sS) * (st[1, -1][5] - st[1, 1][5]))
    return torch.stack([U[k] + dU[k] for k in range(5)] + [bf[c] + dt * curl(E1, c) for c in range(3)])


def _pad(U, geom, z0, z1):
    """The layers z0..z1-1 of the box with three more cells on each side of every active axis."""
    idx = []
    for d in range(3):
        N = int(geom.domain[d])
        lo, hi = (z0, z1) if d == 2 else (0, N)
        i = torch.arange(lo - 3, hi + 3, device=U.device) if N > 1 else torch.zeros(1, dtype=torch.int64, device=U.device)
        idx.append(i % N if int(geom.bc[d][0]) == BC_PERIODIC else i.clamp(0, N - 1))
    return U[:, idx[2][:, None, None], idx[1][None, :, None], idx[0][None, None, :]]


def _slabs(geom):
    nz, plane = int(geom.domain[2]), int(geom.domain[0] * geom.domain[1])
    h = max(1, min(nz, 8_000_000 // plane))
    return [(z, min(nz, z + h)) for z in range(0, nz, h)]


def _crop(V, geom):
    s = [slice(3, -3) if geom.domain[d] > 1 else slice(None) for d in range(3)]
    return V[..., s[2], s[1], s[0]]


def _dt(U, geom, dx, act):
    return COURANT / max(float(_crop(_rate(_pad(U, geom, *z), dx, act), geom).max()) for z in _slabs(geom))


def exact(case, seed):
    if case["kind"] == "async":
        return None   # the order in which patches come up for an update is not a formula
    geom = _geometry(case)
    U = _fields(case, geom, seed).double()
    dx, act = [float(v) for v in geom.dx], [bool(v) for v in geom.active]
    eps = 1e-6 if case["real"] == 32 else 1e-12

    def step(V, dt, slabs):
        return torch.cat([_crop(_advance(_pad(V, geom, *z), dt, dx, act, case["limiter"], case["riemann"], eps), geom)
                          for z in slabs], dim=1)
    if case["kind"] in ("grad", "rollout"):
        dt = 0.5 * _dt(U, geom, dx, act)
        whole = [(0, int(geom.domain[2]))]
        rng = torch.Generator(device=DEV).manual_seed(int(seed) + 5)
        dtype = torch.float32 if case["real"] == 32 else torch.float64
        V = U.clone().requires_grad_(True)
        out = V
        for _ in range(case["steps"]):
            out = step(out, dt, whole)
        parts = _cut(out, geom)
        lam = [torch.randn(p.shape, generator=rng, device=DEV, dtype=dtype).double() for p in parts]
        (grad,) = torch.autograd.grad(parts, V, lam)
        return {"state": [p.detach() for p in parts], "grad": _cut(grad, geom)}
    dts = []
    with torch.no_grad():
        for _ in range(case["steps"]):
            dts.append(_dt(U, geom, dx, act))
            U = step(U, dts[-1], _slabs(geom))
        parts = _cut(U, geom)
        if case["kind"] == "stream":
            return {"state": torch.cat([p.reshape(-1) for p in parts]), "t": sum(dts)}
        return {"state": parts, "dt": torch.tensor(dts, dtype=torch.float64)}
