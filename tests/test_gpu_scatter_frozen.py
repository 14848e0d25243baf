"""The texel gradients with a freeze mask (thawed Gaussians listed by block and
taken in turn) at the edges of the blocks' chunks, thawed none, few and all:
thawed texels equal, bit for bit, to the call without a mask, frozen ones zero,
or untouched where the call accumulates."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 127, 128, 129, 5000, 155_647, 155_648, 155_905])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_frozen_gaussians(n, share):
    import paper_2602_23040_gb300 as pk
    import synth
    rng = np.random.default_rng(n)
    side = int(np.ceil(np.sqrt(1.3 * n))) + 1
    views = [synth.scenes.pinhole((0.4, 0.3, -3.2), 64, 48), synth.scenes.pinhole((-2.6, -0.5, -1.8), 48, 64)]
    plan = pk.Plan([(side, side, 0, 0, 0)], (side, side), 1, 1, "f32", views, n, max_dups=1024)
    ws = pk.make_workspace(plan)
    pk.workspace_init(plan, ws)
    soa = rng.standard_normal((plan.D, n)).astype(np.float32) * 0.3
    soa[6] += 1.0
    soa[3:6] -= 3.0
    texel = np.sort(rng.choice(side * side, n, replace=False)).astype(np.int32)
    flag = (rng.random(n) < share).astype(np.uint8)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    dsoa, dtexel, dflag = dev(soa.reshape(-1)), dev(texel), dev(flag)
    g2d = dev(rng.standard_normal((plan.pairs, 12)).astype(np.float32).reshape(-1))
    every = torch.zeros(plan.D * side * side, device="cuda")
    pk.atlas_scatter_grad(plan, dsoa, g2d, None, dtexel, every, False, ws)
    every = every.view(plan.D, -1)[:, dtexel.long()]
    for accumulate in (False, True):
        out = torch.full((plan.D * side * side,), 2.0, device="cuda")
        pk.atlas_scatter_grad(plan, dsoa, g2d, dflag, dtexel, out, accumulate, ws)
        got = out.view(plan.D, -1)
        want = torch.full_like(got, 2.0)
        thawed = dflag.bool()[None]
        want[:, dtexel.long()] = torch.where(thawed, every + 2.0, 2.0) if accumulate else torch.where(thawed, every, 0.0)
        assert torch.equal(got, want)
