"""Launch sizes chosen on the host."""
import ctypes as ct
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    from paper_2508_09568_gb300 import build as B
    so = str(tmp_path_factory.mktemp("rules") / "rules.so")
    subprocess.run([B._nvcc()] + B.ARCH + B.COMMON + ["-shared", "-o", so, os.path.join(HERE, "launch_rules.cu")], check=True)
    lib = ct.CDLL(so)
    lib.interp_grid_of.restype = ct.c_uint
    return lib


@pytest.mark.parametrize("Zp", [1, 11, 38, 70, 4102])
def test_asynchronous_fill_has_a_cta_per_plane_or_fills_the_chip(rules, Zp):
    """On any bunch: no more CTAs than planes nor than sixteen per SM, and fewer than planes only with at
    least four per SM and eight per patch (or sixteen per SM)."""
    sms = 152
    for patches in (1, 2, 3, 8, 15, 64, 76, 303, 304, 305, 512, 4096, 100000):
        n, planes = rules.interp_grid_of(patches, Zp, 2 * sms), patches * Zp
        assert 0 < n <= min(planes, 16 * sms)
        assert n == planes or (n >= 4 * sms and n >= min(8 * patches, 16 * sms)), (patches, n)
    assert rules.interp_grid_of(7, Zp, 0) == 7 * Zp
