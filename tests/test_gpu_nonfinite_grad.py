"""A NaN or infinite dL/dimage at one pixel: the mean, conic and opacity
gradients of the splats that do not blend there, and of one whose alpha is
clamped there, are those of the same image gradient with that pixel at zero."""

import numpy as np
import pytest

from tests import helpers as H

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PX, PY = 10, 12   # in the left half of the tile: its warp holds a 16 x 8 block


def _records(n, side):
    rng = np.random.default_rng(n)
    rec = np.zeros((n, 12), np.float32)
    rec[:, 0:2] = rng.uniform(0.5, side - 0.5, (n, 2))
    rec[:, 2] = rng.uniform(0.4, 1.2, n)
    rec[:, 3] = rng.uniform(-0.2, 0.2, n)
    rec[:, 4] = rng.uniform(0.4, 1.2, n)
    rec[:, 5] = rng.uniform(0.02, 0.3, n)
    rec[:, 6] = rng.permutation(n) / n * 4.0 + 1.0
    rec[:, 7] = 5.0
    rec[:, 8:11] = rng.uniform(0, 1, (n, 3))
    rec[0, :7] = (PX + 0.5, PY + 0.5, 1.0, 0.0, 1.0, 0.999, 1.0)   # clamped at the pixel, in front of the others
    return rec


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("n,count,stage", [(100, False, "loads"), (100, True, "bulk"), (700, False, "loads")])
def test_gradients_of_the_splats_elsewhere_are_unchanged(value, n, count, stage):
    import paper_2602_23040_gb300 as pk
    import synth
    side = 32
    rec = _records(n, side)
    d = np.array([PX + 0.5, PY + 0.5]) - rec[:, :2].astype(np.float64)
    q = rec[:, 2] * d[:, 0] ** 2 + 2.0 * rec[:, 3] * d[:, 0] * d[:, 1] + rec[:, 4] * d[:, 1] ** 2
    away = (q > 9.1) | (rec[:, 5] * np.exp(-0.5 * q) < 0.99 / 255.0)
    away[0] = True
    near = (np.abs(d[:, 0]) < 16) & (np.abs(d[:, 1]) < 8)
    assert (away & near).sum() > 10 and (~away).sum() > 3
    plan = pk.Plan([(32, 32, 0, 0, 0)], (32, 32), 0, 1, "f32", [synth.scenes.pinhole((0, 0, -3), side, side)], n,
                   max_dups=2 * n + 1024, stage_bwd=stage, count_evals=count)
    ws = pk.make_workspace(plan)
    pk.workspace_init(plan, ws)
    drec = torch.from_numpy(rec.reshape(-1)).cuda()
    vals = torch.empty(plan.max_dups + 64, dtype=torch.int32, device="cuda")
    ranges = torch.empty(2 * plan.n_tiles, dtype=torch.int64, device="cuda")
    img = torch.empty(3 * plan.P, dtype=torch.float32, device="cuda")
    T = torch.empty(plan.P, dtype=torch.float32, device="cuda")
    nc = torch.empty(plan.P, dtype=torch.int32, device="cuda")
    pk.bin_and_sort(plan, drec, vals, ranges, ws)
    pk.rasterize_fwd(plan, drec, vals, ranges, img, T, nc, ws)
    w = torch.from_numpy(np.random.default_rng(5).standard_normal(3 * plan.P).astype(np.float32)).cuda()

    def grads(x):
        w.view(3, side, side)[:, PY, PX] = x
        g2 = torch.empty(12 * plan.pairs, dtype=torch.float32, device="cuda")
        pk.rasterize_bwd(plan, drec, vals, ranges, T, nc, w, g2, ws)
        return g2.view(-1, 12).cpu().numpy().astype(np.float64)[:, :6]

    want, got = grads(0.0), grads(value)
    assert pk.read_status(plan, ws)["flags"] == 0
    assert np.isfinite(want).all() and np.isfinite(got[away]).all()
    assert not np.isfinite(got[~away]).all()
    # the two differ by the order of the atomic additions alone
    assert H.rel_err(got[away], want[away]) < 1e-5
