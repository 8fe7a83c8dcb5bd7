"""Tile lists built by counting (per-tile segments, each sorted on its own) and by the global radix sorts, against
oracle/binning.py: the sizes and depth distributions at which the per-tile sort changes its method -- lists that
one warp sorts, lists of one CTA, lists longer than its shared memory; depths all different, in a few groups,
and all equal. Keys, values and ranges are exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import binning  # noqa: E402
from paper_2603_02887_gb300 import synth  # noqa: E402
from paper_2603_02887_gb300.render import Renderer  # noqa: E402
from tests.gpu_util import frame_arrays, upload  # noqa: E402


def _scene(n, depths, seed):
    """n splats in front of an identity camera, most of them over several 16x16 tiles, at the given depths."""
    rng = np.random.default_rng(seed)
    s = synth.tiny_scene(seed, n=n)
    if depths == "all":
        z = rng.uniform(2.0, 6.0, n)
    elif depths == "one":
        z = np.full(n, 3.0)
    elif depths == "most":  # three quarters of the splats at one depth
        z = np.where(rng.random(n) < 0.75, 3.0, rng.uniform(2.0, 6.0, n))
    else:
        z = 2.0 + rng.integers(0, int(depths), n) / 7.0
    s["means"] = np.stack([rng.uniform(-0.2, 0.2, n) * z, rng.uniform(-0.2, 0.2, n) * z, z], 1).astype(np.float32)
    s["log_scales"] = rng.normal(-2.2, 0.3, (n, 3)).astype(np.float32)
    return s


@pytest.mark.parametrize("n", [1, 31, 256, 700, 4000, 9000])
@pytest.mark.parametrize("depths", ["all", "one", "most", "9"])
@pytest.mark.parametrize("schedule", ["tiles", "persistent"])
def test_tile_lists_match_the_oracle(n, depths, schedule):
    scene = _scene(n, depths, seed=n)
    cam = synth.pinhole(np.concatenate([np.eye(3), np.zeros((3, 1))], 1), 37, 45, 80.0, 80.0)
    r = Renderer("cuda:0")
    img, od, frame = r.render(upload(scene), cam, "sup", dict(schedule=schedule))
    fa = frame_arrays(frame)
    keys, vals, ranges = binning.sorted_pairs(fa["records"], fa["view"]["log2_alpha_min"], 16, 16, 37, 45)
    assert np.array_equal(fa["keys"], keys)
    assert np.array_equal(fa["values"], vals)
    assert np.array_equal(fa["ranges"].astype(np.int64), ranges)
    r.close()


@pytest.mark.parametrize("n", [9000, 24576, 24577])  # 384 records per tile: the last counted, and the first radix-sorted, size
@pytest.mark.parametrize("depths", ["all", "most", "9"])
def test_long_lists_and_the_limit_of_counting(n, depths):
    """Lists longer than a CTA's shared memory in a frame of 64 tiles, most of them empty."""
    scene = _scene(n, depths, seed=n)
    cam = synth.pinhole(np.concatenate([np.eye(3), np.zeros((3, 1))], 1), 128, 128, 80.0, 80.0)
    r = Renderer("cuda:0")
    img, od, frame = r.render(upload(scene), cam, "sup")
    fa = frame_arrays(frame)
    keys, vals, ranges = binning.sorted_pairs(fa["records"], fa["view"]["log2_alpha_min"], 16, 16, 128, 128)
    assert int((ranges[:, 1] - ranges[:, 0]).max()) > 2048
    assert np.array_equal(fa["keys"], keys)
    assert np.array_equal(fa["values"], vals)
    assert np.array_equal(fa["ranges"].astype(np.int64), ranges)
    r.close()
