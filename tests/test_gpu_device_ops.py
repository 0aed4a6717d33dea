"""The element operations of the scheme (mhd_ops.cuh, mhd_math.cuh, mhd_vjp.cuh) as the device
evaluates them, one operation per argument row, in both precisions and with the compiler flags of the
kernels."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest
import torch

import extended_reference as X

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
OPS = ["greater", "hlld_vjp", "compare", "max0", "emf2d", "emf2d_vjp", "roots", "hll_vjp"]
DTYPES = [torch.float64, torch.float32]
both = pytest.mark.parametrize("dtype", DTYPES, ids=["f64", "f32"])


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    """ops(name, rows, nout, dtype): rows (n, nin) through an operation, (n, nout) back."""
    from paper_2508_09568_gb300 import build as B
    tmp = tmp_path_factory.mktemp("device_ops")
    libs = {}
    for dtype, real, unit in ((torch.float64, "double", "kernels_f64.cu"), (torch.float32, "float", "kernels_f32.cu")):
        so = str(tmp / f"ops_{real}.so")
        flags = [f for f in B.UNITS[unit] if f.startswith("-prec") or f.startswith("-ftz")]
        subprocess.run([B._nvcc()] + B.ARCH + B.COMMON + flags + [f"-DREAL={real}", "-shared", "-o", so,
                                                                   os.path.join(HERE, "device_ops.cu")], check=True)
        libs[dtype] = ct.CDLL(so)
        libs[dtype].run_rows.argtypes = [ct.c_int, ct.c_int, ct.c_int, ct.c_void_p, ct.c_void_p, ct.c_int]

    def run(name, rows, nout, dtype):
        x = torch.as_tensor(np.ascontiguousarray(rows), dtype=dtype).cuda()
        y = torch.full((x.shape[0], nout), float("nan"), dtype=dtype, device="cuda")
        torch.cuda.synchronize()
        assert libs[dtype].run_rows(OPS.index(name), x.shape[1], nout, x.data_ptr(), y.data_ptr(), x.shape[0]) == 0
        return y.cpu().numpy()
    return run


def pairs(values):
    a, b = np.meshgrid(values, values, indexing="ij")
    return np.stack([a.ravel(), b.ravel()], axis=1)


@both
def test_greater_takes_the_two_zeros_as_equal(ops, dtype):
    x = pairs([0.0, -0.0, 1e-30, -1e-30, 1.0, -1.0, 1.5, -1.5, np.inf, -np.inf])
    assert np.array_equal(ops("greater", x, 1, dtype)[:, 0], (x[:, 0] > x[:, 1]).astype(float))


@both
def test_hlld_reverse_at_rest_does_not_depend_on_the_sign_of_zero(ops, dtype):
    """Gas at rest on both sides of a face, a velocity of +0 or -0: a tie of the two velocities, whose
    cotangent goes to the first in every case."""
    rng = np.random.default_rng(5)
    rows = []
    for ul in (0.0, -0.0):
        for ur in (0.0, -0.0):
            rows.append([1.0, ul, 0.1, -0.2, 0.9, 0.3, 0.2, 0.8, ur, 0.3, 0.1, 1.1, -0.1, 0.4, 0.5])
    rows = np.concatenate([np.array(rows), np.tile(rng.normal(size=5), (4, 1))], axis=1)
    y = ops("hlld_vjp", rows, 15, dtype)
    assert np.all(np.isfinite(y)) and np.any(y[:, [1, 8]] != 0)
    for k in range(1, 4):
        assert np.array_equal(y[k], y[0]), k


def special(dtype):
    """Values whose bits order in every way: zeros, normal numbers, infinities, NaN of both signs
    (double precision: subnormal numbers too)."""
    v = [0.0, -0.0, 1.0, -1.0, 1.5, -1.5, 1e-30, -1e-30, 3e30, -3e30, np.inf, -np.inf, np.nan, np.copysign(np.nan, -1.0)]
    return np.array(v + ([5e-324, -5e-324, 1e-310] if dtype == torch.float64 else []))


def same(got, ref):
    return np.all((got == ref) | (np.isnan(got) & np.isnan(ref)))


@both
def test_comparisons_are_those_of_the_values(ops, dtype):
    x = pairs(special(dtype))
    a, b = (x.astype(np.float32) if dtype == torch.float32 else x).T
    y = ops("compare", x, 8, dtype).T
    with np.errstate(invalid="ignore"):
        for k, ref in enumerate((a >= 0, a > 0, a != 0, a > b, ((a > 0) & (b > 0)) | ((a < 0) & (b < 0)))):
            assert same(y[k], ref.astype(float)), k
        assert same(y[5], np.fmax(a, b)) and same(y[6], np.fmin(a, b))
        both_ = ((a > 0) & (b > 0)) | ((a < 0) & (b < 0))
        ref = np.where(both_, np.where(np.abs(a) <= np.abs(b), a, b), 0)
        ok = slice(None) if dtype == torch.float64 else ~(np.isnan(a) | np.isnan(b))
        assert same(y[7][ok], ref[ok])


@both
def test_largest_and_smallest_of_four_pass_over_nan(ops, dtype):
    v = special(dtype)
    x = v[np.random.default_rng(3).integers(0, len(v), size=(4096, 4))]
    x = np.concatenate([x, [[s] * 4 for s in v]])
    y = ops("max0", x, 2, dtype)
    x = x.astype(y.dtype)
    assert same(y[:, 0], np.fmax(np.fmax.reduce(x, axis=1), 0)) and same(y[:, 1], np.fmin(np.fmin.reduce(x, axis=1), 0))


@both
@pytest.mark.parametrize("bad", range(4))
def test_edge_emf_beside_a_corner_without_speeds(ops, dtype, bad):
    """A corner whose extrapolated density is negative has no fast speed; the speeds of the other three
    decide, in the EMF and in its reverse: both equal, bit for bit, those with a corner so dense that its
    speeds are never the largest."""
    rng = np.random.default_rng(60 + bad)
    n = 256
    c = np.empty((n, 4, 7))
    c[:, :, 0] = rng.uniform(0.8, 1.2, (n, 4))
    c[:, :, 1] = rng.uniform(0.8, 1.2, (n, 4))
    c[:, :, 2:] = rng.uniform(-0.1, 0.1, (n, 4, 5))
    neg, dense = c.copy(), c.copy()
    neg[:, bad, 0], dense[:, bad, 0] = -0.3, 1e8
    l = rng.normal(size=(n, 1))
    e = [ops("emf2d", r.reshape(n, 28), 1, dtype) for r in (neg, dense)]
    assert np.all(np.isfinite(e[1])) and np.array_equal(e[0], e[1])
    g = [ops("emf2d_vjp", np.concatenate([r.reshape(n, 28), l], axis=1), 28, dtype) for r in (neg, dense)]
    assert np.all(np.isfinite(g[1])) and np.array_equal(g[0], g[1])


def test_fp64_square_root_and_reciprocal(ops):
    """Over every exponent with random significands, beside the powers of two (significands of few bits
    and of almost all), at the squares of points half way between two numbers and at reciprocals of
    numbers, where the rounding is closest; at and beside the ends of the range of the fast forms; and
    the special values.  rsqrt_ and rcp_: bit for bit the IEEE operations (numpy's).  The near forms:
    the same bits outside the range, at most the neighbour inside it, and within 0.51 units in the last
    place of the exact value (0.5 of the rounding and the two forms' remainders, at most 2^-60 and 2^-59
    of the value, 0.008 and 0.016 units, less than that where they add to 0.5)."""
    rng = np.random.default_rng(70)
    n = 1 << 19
    man = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    few = rng.integers(0, 1 << 12, n, dtype=np.uint64)
    one = np.uint64(1) << rng.integers(0, 52, n, dtype=np.uint64)
    top = np.uint64((1 << 52) - 1)
    ex = rng.integers(1, 2047, n, dtype=np.uint64) << np.uint64(52)
    m = ((np.uint64(1023) << np.uint64(52)) | man).view(np.float64)
    mid = np.ldexp(m * m + m * 2.0 ** -52, 2 * rng.integers(-400, 400, n))
    inv = np.ldexp(1.0 / m, rng.integers(-800, 800, n))
    ends = np.array([s for e in (-900, 900, -1022, 0, 1) for s in (2.0 ** e, np.nextafter(2.0 ** e, 0), np.nextafter(2.0 ** e, 9e300))])
    x = np.concatenate([(ex | v).view(np.float64) for v in (man, few, top - few, one, top - one, np.full(n, top))]
                       + [mid, inv, ends, np.finfo(float).max * np.ones(1), special(torch.float64)])
    x = np.concatenate([x, -x])
    y = ops("roots", x[:, None], 4, torch.float64)
    with np.errstate(invalid="ignore", divide="ignore", over="ignore"):
        ref = np.stack([np.sqrt(x), 1.0 / x], axis=1)
        assert same(y[:, :2], ref)
        assert np.array_equal(np.signbit(y[:, 1][np.isinf(x)]), np.signbit(x[np.isinf(x)]))
        inside = (np.abs(x) >= 2.0 ** -900) & (np.abs(x) < 2.0 ** 900)
        assert same(y[~inside, 2:], ref[~inside])
        k = inside & (x > 0)
        assert np.all(np.abs(y[k, 2] - ref[k, 0]) <= np.spacing(ref[k, 0]))
        assert np.all(np.abs(y[inside, 3] - ref[inside, 1]) <= np.spacing(np.abs(ref[inside, 1])))
    x, y = x[:n][k[:n]][:100000], y[:n][k[:n]][:100000]
    xl = x.astype(np.longdouble)   # (64 bits of significand or more)
    assert np.finfo(np.longdouble).nmant >= 63
    for c, exact in ((2, np.sqrt(xl)), (3, 1 / xl)):
        assert np.max(np.abs(y[:, c] - exact) / np.spacing(y[:, c])) <= 0.51


@pytest.mark.parametrize("name,bound", [("hlld_vjp", 1.21), ("hll_vjp", 0.664), ("emf2d_vjp", 0.415)])
def test_fp64_rounding_error_of_the_reverses(ops, name, bound):
    """Root mean square error of the cotangents, in units of 2^-53 of the row's largest, against the
    derivative in extended precision.  The bounds are what the reverses with IEEE divisions and square
    roots throughout give on the same rows (1.208, 0.6626, 0.4143), rounded up."""
    n = 3000
    if name == "emf2d_vjp":
        x = X.edge_rows(n, 81)
        v = X.inputs(x[:, :28])
        ref = (x[:, 28].astype(X.LD) * X.edge_emf([v[7 * k:7 * k + 7] for k in range(4)]).d).T
    else:
        x = X.face_rows(n, 82)
        F = X.face_flux(X.inputs(x[:, :15]), name == "hll_vjp")
        ref = sum(x[:, 15 + k].astype(X.LD) * F[k].d for k in range(5)).T
    y = ops(name, x, ref.shape[1], torch.float64)
    err = (np.abs(y - ref) / np.max(np.abs(ref), axis=1, keepdims=True)).astype(float) * 2.0 ** 53
    assert np.sqrt(np.mean(err ** 2)) <= bound
