"""The 3D step on patches at the edges of its plane staging and of its lane maps: rows too wide for
the bulk copies (element copies then), rows and volumes that are not multiples of 16 bytes (every
offset of a staged block), tiles with ragged tails, patches of the smallest extents, bunches of few
tiles (marched as z-blocks by the persistent launch, as whole columns by the other); every tile
configuration against the oracle, with the parity bounds of one step, and bitwise the same."""
import numpy as np
import pytest
import torch

from helpers import assert_parity, gpu_bunch, gpu_steps, interior_global, oracle_bunch, oracle_steps, rounded
from paper_2508_09568_gb300 import capi
from paper_2508_09568_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (box, patch): 38 padded columns are the widest row staged in bulk
SHAPES = {
    "rows_38": ((32, 9, 4), (32, 9, 4)),
    "rows_39": ((33, 9, 8), (33, 9, 4)),
    "wide": ((70, 8, 5), (70, 8, 5)),
    "odd_volume": ((42, 13, 9), (21, 13, 9)),
    "odd_rows": ((31, 20, 10), (31, 10, 5)),
    "smallest": ((6, 6, 6), (3, 3, 3)),
    "flat_tiles": ((25, 17, 3), (25, 17, 3)),
    "z_blocks": ((12, 10, 37), (12, 10, 37)),
}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("limiter", [0, 1], ids=["minmod", "mc"])
def test_step_matches_oracle_in_every_configuration(shape, dtype, limiter):
    ncell, patch = SHAPES[shape]
    geom, U, meta = W.small_box(ncell=ncell, patch=patch, seed=31)
    flat = rounded(W.to_patches(U, geom), dtype)
    ob = oracle_bunch(geom, meta["gamma"], limiter=limiter, dtype=dtype)
    dt = ob.cfl_dt(ob.fill_guards(ob.split(flat)))
    ref = interior_global(oracle_steps(geom, flat, meta["gamma"], [dt], limiter=limiter, dtype=dtype), geom)
    b = gpu_bunch(geom, flat, meta["gamma"], dtype, limiter=limiter)
    first = None
    for cfg in range(-1, b.num_configs()):   # -1: the configuration chosen by the patch sizes
        for mode in (capi.MHD_MODE_PERSISTENT, capi.MHD_MODE_BUNCHED):
            b.set_mode(mode, cfg)
            b.upload(flat)
            got = interior_global(gpu_steps(b, [dt]), geom)
            if first is None:
                first = got
                assert_parity(got, ref, dtype, what=shape)
            assert np.array_equal(got, first), (shape, cfg, mode)
    assert b.error()[0] == 0


@pytest.mark.parametrize("n", [3, 27, 63, 64, 65, 100])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
def test_1d_tiles_that_reach_past_their_patch(n, dtype):
    """1D patches from a few cells to more than a tile: the chunks past the patch are left out."""
    geom, U, meta = W.sod(ncell=4 * n, npatch=4)
    flat = rounded(W.to_patches(U, geom), dtype)
    ob = oracle_bunch(geom, meta["gamma"], dtype=dtype)
    dt = ob.cfl_dt(ob.fill_guards(ob.split(flat)))
    ref = interior_global(oracle_steps(geom, flat, meta["gamma"], [dt, dt], dtype=dtype), geom)
    b = gpu_bunch(geom, flat, meta["gamma"], dtype)
    assert_parity(interior_global(gpu_steps(b, [dt, dt]), geom), ref, dtype)
    assert b.error()[0] == 0


# 1D and 2D boxes with all field components: edges along and across the collapsed axes
COLLAPSED = {
    "1d": ((37, 1, 1), (37, 1, 1)),
    "1d_patches": ((72, 1, 1), (24, 1, 1)),
    "2d_odd": ((33, 17, 1), (33, 17, 1)),
    "2d_patches": ((40, 24, 1), (20, 12, 1)),
    "2d_smallest": ((6, 6, 1), (3, 3, 1)),
}


@pytest.mark.parametrize("shape", list(COLLAPSED))
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("riemann,limiter", [(0, 0), (1, 1)], ids=["hlld_minmod", "hll_mc"])
def test_edges_of_collapsed_axes(shape, dtype, riemann, limiter):
    ncell, patch = COLLAPSED[shape]
    geom, U, meta = W.small_box(ncell=ncell, patch=patch, seed=47)
    flat = rounded(W.to_patches(U, geom), dtype)
    ob = oracle_bunch(geom, meta["gamma"], limiter=limiter, dtype=dtype, riemann=riemann)
    dt = ob.cfl_dt(ob.fill_guards(ob.split(flat)))
    ref = oracle_steps(geom, flat, meta["gamma"], [dt], limiter=limiter, dtype=dtype, riemann=riemann)
    b = gpu_bunch(geom, flat, meta["gamma"], dtype, limiter=limiter, riemann=riemann)
    for cfg in range(-1, b.num_configs()):
        b.set_mode(capi.MHD_MODE_PERSISTENT, cfg)
        b.upload(flat)
        assert_parity(interior_global(gpu_steps(b, [dt]), geom), interior_global(ref, geom), dtype, what=shape, b_vector=True)
    assert b.error()[0] == 0
