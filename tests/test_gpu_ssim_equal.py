"""The photometric objective where image and target agree bit for bit -- an SSIM
of 1 and a gradient of no more than the rounding of its last sum -- and where
they have nothing in common, against the oracle."""

import numpy as np
import pytest

import synth
from tests import helpers as H_

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

W, H = 203, 117


def _image(kind):
    yy, xx = np.mgrid[0:H, 0:W] / W
    one = {"smooth": 0.5 + 0.3 * np.sin(9 * xx) + 0.15 * np.cos(13 * yy), "flat": np.full((H, W), 0.7),
           "dark": np.full((H, W), 0.03), "noise": np.random.default_rng(3).random((H, W))}[kind]
    return np.tile(one.astype(np.float32).reshape(-1), 3)


def _loss(x, y):
    import paper_2602_23040_gb300 as pk
    sc = synth.make_scene([(16, 16, 0, 0, 0)], (16, 16), 0.5, [synth.scenes.pinhole((0, 0, -3), W, H)], sh_degree=0,
                          seed=1)
    p = pk.Plan.for_scene(sc)
    ws = pk.make_workspace(p)
    pk.workspace_init(p, ws)
    g = torch.empty(3 * W * H, dtype=torch.float32, device="cuda")
    pk.photo_loss_grad(p, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), g, ws, 1.0)
    return pk.read_status(p, ws), g.cpu().numpy().astype(np.float64), sc


@pytest.mark.parametrize("kind", ["smooth", "flat", "dark", "noise"])
def test_equal_images(kind):
    x = _image(kind)
    st, g, _ = _loss(x, x.copy())
    assert abs(st["ssim"] - 1.0) < 1e-9 and abs(st["loss"]) < 1e-9
    # the gradient is 2 (G*d1 + x G*d11 + x G*d12) / 3P with d1 = 0 and d11 = -d12, at most 1 / 9e-4 < 2^11: what
    # is left is the rounding of x G*d11 < 2^11, half a unit of 2^-13 at most
    assert np.abs(g).max() * 3 * W * H <= 2.0 ** -13 * 1.001


@pytest.mark.parametrize("scale_x,scale_y", [(0.0, 1.0), (1.0, 0.0), (0.01, 1.0), (1.0, 0.01), (0.01, 0.01), (1.0, 1.0)])
def test_unlike_images(orc, scale_x, scale_y):
    """Factors of the SSIM value from 1 down to C1 / (m^2 + C1): a few units in
    the last place of every term, five times the 2e-7 that FP32 leaves here."""
    r = np.random.default_rng(8)
    x, y = ((s * r.random(3 * W * H)).astype(np.float32) for s in (scale_x, scale_y))
    st, g, sc = _loss(x, y)
    o = orc.photo_loss(x.astype(np.float64), y.astype(np.float64), orc.views_array(sc.views), lam=1.0)
    assert abs(st["ssim"] - o["ssim"]) <= 1e-7
    assert H_.rel_err(g, o["grad"]) <= 1e-6
