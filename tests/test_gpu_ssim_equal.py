"""The photometric objective where image and target agree bit for bit: an SSIM
of 1 and a gradient of no more than the rounding of its last sum."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

W, H = 203, 117


def _image(kind):
    yy, xx = np.mgrid[0:H, 0:W] / W
    one = {"smooth": 0.5 + 0.3 * np.sin(9 * xx) + 0.15 * np.cos(13 * yy), "flat": np.full((H, W), 0.7),
           "dark": np.full((H, W), 0.03), "noise": np.random.default_rng(3).random((H, W))}[kind]
    return np.tile(one.astype(np.float32).reshape(-1), 3)


@pytest.mark.parametrize("kind", ["smooth", "flat", "dark", "noise"])
def test_equal_images(kind):
    import paper_2602_23040_gb300 as pk
    sc = synth.make_scene([(16, 16, 0, 0, 0)], (16, 16), 0.5, [synth.scenes.pinhole((0, 0, -3), W, H)], sh_degree=0,
                          seed=1)
    p = pk.Plan.for_scene(sc)
    ws = pk.make_workspace(p)
    pk.workspace_init(p, ws)
    x = torch.from_numpy(_image(kind)).cuda()
    g = torch.empty_like(x)
    pk.photo_loss_grad(p, x, x.clone(), g, ws, 1.0)
    st = pk.read_status(p, ws)
    assert abs(st["ssim"] - 1.0) < 1e-9 and abs(st["loss"]) < 1e-9
    # the gradient is 2 (G*d1 + x G*d11 + x G*d12) / 3P with d1 = 0 and d11 = -d12, at most 1 / 9e-4 < 2^11: what
    # is left is the rounding of x G*d11 < 2^11, half a unit of 2^-13 at most
    assert float(g.abs().max()) * 3 * W * H <= 2.0 ** -13 * 1.001
