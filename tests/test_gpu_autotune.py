"""The autotuner's saved choices."""
import pytest
import torch

from helpers import gpu_bunch, rounded
from paper_2508_09568_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
def test_saved_choice_holds_for_the_tiles_it_was_made_among(dtype, tmp_path):
    """What is saved is an index: its key names the tile of every configuration, a file with the same key
    is taken as it is, and one whose list of tiles is another (that of another version of the library)
    is not."""
    geom, U, meta = W.small_box(ncell=(16, 16, 16), patch=(8, 8, 8), seed=23)
    flat = rounded(W.to_patches(U, geom), dtype)
    b = gpu_bunch(geom, flat, meta["gamma"], dtype)
    n = b.num_configs()
    path = str(tmp_path / "choices")
    chosen = b.autotune(path)
    (line,) = open(path).read().splitlines()
    key, index = line.split()
    tiles = ",".join("%dx%dx%d" % b.config_info(k) for k in range(n))
    assert int(index) == chosen and key.endswith("|c" + tiles)
    # the same list: the saved index is taken, without measuring again
    other = (chosen + 1) % n
    open(path, "w").write(f"{key} {other}\n")
    assert b.autotune(path) == other
    assert len(open(path).read().splitlines()) == 1
    # another list, or none (files written before the key had one): measured again and added
    for stale in (key[: key.rindex("|c")] + "|c" + ",".join(["8x8x64"] * n), key[: key.rindex("|c")]):
        open(path, "w").write(f"{stale} {other}\n")
        b.autotune(path)
        lines = open(path).read().splitlines()
        assert len(lines) == 2 and lines[1].split()[0] == key
    b.close()
