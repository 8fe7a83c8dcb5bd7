"""The replay's sums over a warp's pixels: eight entries are gathered and summed together, so the numbers of entries at
which a group is full, or has one entry, against the oracle; and an upstream gradient that is not finite, which reaches
the Gaussians that its pixel composites and no other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2603_02887_gb300 import _abi, synth  # noqa: E402
from paper_2603_02887_gb300.render import Renderer  # noqa: E402
from tests.gpu_util import upload  # noqa: E402
from tests.test_gpu_parity import _backward_check  # noqa: E402


MODELS = ["exp", "sub", (_abi.NGS_MODEL_BLEND, 0.5), (_abi.NGS_MODEL_VICINI, 0.5)]
IDS = ["exp", "sub", "blend", "vicini"]


@pytest.fixture(scope="module")
def rnd():
    r = Renderer("cuda:0")
    yield r
    r.close()


@pytest.mark.parametrize("tile", [(8, 8, 32), (16, 16, 0), (16, 32, 1024)])  # one-pixel staging in the last
@pytest.mark.parametrize("model", MODELS, ids=IDS)
def test_group_remainders_match_oracle(rnd, model, tile):
    opts = dict(tile_w=tile[0], tile_h=tile[1], chunk=tile[2])
    for n in (1, 8, 9, 41):
        scene = synth.tiny_scene(n, n=n)
        scene["log_scales"] = (scene["log_scales"] + np.float32(1.0)).astype(np.float32)  # over several tiles
        _backward_check(rnd, scene, synth.tiny_camera(), model, options=opts)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("model", MODELS, ids=IDS)
@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (16, 32)])
def test_non_finite_upstream_stays_with_its_pixel(rnd, model, tile, value):
    params, cam = upload(synth.tiny_scene(5)), synth.tiny_camera()
    img, _, f = rnd.render(params, cam, model, dict(tile_w=tile[0], tile_h=tile[1]))
    gen = torch.Generator(device="cuda").manual_seed(7)
    dl = torch.randn(img.shape, generator=gen, device="cuda")
    y, x = img.shape[0] // 2 + 3, img.shape[1] // 2 + 1

    def grads(g):
        return {k: v.clone() for k, v in rnd.backward(f, params, g.contiguous()).items()}

    lone = torch.zeros_like(dl)
    lone[y, x] = dl[y, x]
    reached = torch.zeros(params["means"].shape[0], dtype=torch.bool, device="cuda")
    for v in grads(lone).values():
        reached |= (v.reshape(len(reached), -1) != 0).any(1)
    assert 0 < int(reached.sum()) < len(reached)
    without, bad = dl.clone(), dl.clone()
    without[y, x] = 0
    bad[y, x, 1] = value
    want, got = grads(without), grads(bad)
    wrong = torch.zeros_like(reached)
    for k, v in got.items():
        wrong |= ~torch.isfinite(v.reshape(len(reached), -1)).all(1)
        # FP32 sums of the other pixels in another order
        assert torch.allclose(v[~reached], want[k][~reached], rtol=1e-4, atol=1e-5 * float(want[k].abs().max())), k
    assert wrong.any() and not (wrong & ~reached).any()
    rnd.recycle(f)
