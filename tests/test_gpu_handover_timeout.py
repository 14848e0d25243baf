"""A bulk-staged walk whose wait gives up while few CTAs are left takes no
long-list slot: its block is left as it was, not finished by the kernel of
the handed-over lists from whatever its scratch holds."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_a_timed_out_walk_is_not_handed_over():
    import paper_2602_23040_gb300 as pk
    import synth
    # 2,704 blocks, all empty but the last: the other CTAs have left by the time its first batch of 256 -- the
    # first point at which a list of twice that may be handed over -- has landed
    side, n, batch = 832, 700, 256
    rng = np.random.default_rng(1)
    rec = np.zeros((n, 12), np.float32)
    rec[:, 0:2] = rng.uniform(side - 10, side - 6, (n, 2))
    rec[:, 2] = rec[:, 4] = 1.5
    rec[:, 5] = 0.02
    rec[:, 6] = rng.permutation(n) / n + 1.0
    rec[:, 7] = 3.0
    rec[:, 8:11] = rng.uniform(0, 1, (n, 3))
    views = [synth.scenes.pinhole((0, 0, -3), side, side)]
    args = dict(levels=[(32, 32, 0, 0, 0)], atlas_wh=(32, 32), sh_degree=0, frames=1, texel_type="f32", views=views,
                n_live=n, max_dups=2 * n + 1024, tile=16)
    sorter = pk.Plan(**args)
    plan = pk.Plan(**args, batch=batch, stage_fwd="bulk", first_wait_polls=-1)
    ws0, ws = pk.make_workspace(sorter), pk.make_workspace(plan)
    pk.workspace_init(sorter, ws0)
    drec = torch.from_numpy(rec.reshape(-1)).cuda()
    vals = torch.empty(plan.max_dups + 64, dtype=torch.int32, device="cuda")
    ranges = torch.empty(2 * plan.n_tiles, dtype=torch.int64, device="cuda")
    pk.bin_and_sort(sorter, drec, vals, ranges, ws0)
    assert pk.read_status(sorter, ws0)["dups"] == n
    r = ranges.view(-1, 2).cpu().numpy()
    assert r[-1, 1] - r[-1, 0] == n and not (r[:-1, 1] - r[:-1, 0]).any()
    for _ in range(20):
        pk.workspace_init(plan, ws)
        img = torch.full((3 * plan.P,), -7.0, device="cuda")
        T = torch.full((plan.P,), -7.0, device="cuda")
        nc = torch.full((plan.P,), -7, dtype=torch.int32, device="cuda")
        pk.rasterize_fwd(plan, drec, vals, ranges, img, T, nc, ws)
        st = pk.read_status(plan, ws)
        assert st["rc"] == 4 and st["flags"] == 4
        for x in (img.view(3, side, side), T.view(1, side, side), nc.view(1, side, side)):
            assert bool((x[:, -16:, -16:] == -7).all())
