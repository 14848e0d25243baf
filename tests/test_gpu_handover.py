"""Walks handed over part way: a launch of many blocks of which all but a few
are empty, so that the long lists are still being walked when few CTAs are
left.  The forward bit for bit as the counting variant, which walks every
list whole, the gradients against the oracle; blocks whose left half has
stopped, and blocks that stop within the very batch that decides."""

import numpy as np
import pytest

from tests import helpers as H

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _thin(rng, x0, y0, n, dense):
    """n splats inside the 16 px block at (x0, y0), too thin to stop a pixel but (dense) in its left half."""
    rec = np.zeros((n, 12), np.float32)
    rec[:, 0] = x0 + rng.uniform(3.5, 12.5, n)
    rec[:, 1] = y0 + rng.uniform(3.5, 12.5, n)
    rec[:, 2] = rec[:, 4] = rng.uniform(1.2, 1.6, n)
    rec[:, 3] = rng.uniform(-0.1, 0.1, n)
    rec[:, 5] = np.where(dense & (rec[:, 0] < x0 + 8), rng.uniform(0.1, 0.9, n), rng.uniform(0.004, 0.02, n))
    rec[:, 7] = 3.0
    return rec


def _wall(x0, y0):
    """125 splats that stop every pixel of the 16 px block at (x0, y0)."""
    at = np.stack(np.meshgrid(np.arange(0, 17, 4), np.arange(0, 17, 4)), -1).reshape(-1, 2)
    rec = np.zeros((125, 12), np.float32)
    rec[:, 0:2] = np.tile(at, (5, 1)) + (x0, y0)
    rec[:, 2] = rec[:, 4] = 0.2
    rec[:, 5] = 0.99
    rec[:, 7] = 7.0
    return rec


def _records(side, blocks, seed):
    """Every third of `blocks` (16 px) is walled up between its entries 128 and 256."""
    rng = np.random.default_rng(seed)
    out = []
    for i, (bx, by, n) in enumerate(blocks):
        if i % 3 == 2:
            r = np.concatenate([_thin(rng, 16 * bx, 16 * by, 128, False), _wall(16 * bx, 16 * by),
                                _thin(rng, 16 * bx, 16 * by, n - 253, False)])
        else:
            r = _thin(rng, 16 * bx, 16 * by, n, i % 3 == 1)
        r[:, 6] = 1.0 + np.arange(n) / 1024.0   # in list order
        out.append(r)
    rec = np.concatenate(out)
    rec[:, 8:11] = rng.uniform(0, 1, (len(rec), 3))
    return rec


def _blocks(side, count, lens):
    """The last `count` blocks of every other block column and row, list lengths from `lens` in turn."""
    nb = side // 16
    at = [(x, y) for y in range(1, nb, 2) for x in range(1, nb, 2)][-count:]
    return [(x, y, lens[i % len(lens)]) for i, (x, y) in enumerate(at)]


# 900 blocks: fewer than the resident CTAs, a walk may go on elsewhere after 256 entries; 6,400: more than four
# times as many, after 1,024, and over 128 lists to split in the backward
@pytest.mark.parametrize("side,tile,stage,batch,count,lens", [
    (480, 16, "loads", 128, 24, (3000, 513, 2049)), (480, 16, "bulk", 64, 24, (3000, 512, 777)),
    (480, 16, "bulk", 256, 24, (1025, 5000, 900)), (480, 16, "loads", 256, 24, (4100, 640, 2500)),
    (480, 32, "loads", 128, 12, (2777, 1500, 600)), (480, 32, "bulk", 128, 12, (2560, 700, 3100)),
    (1280, 16, "loads", 128, 150, (2500, 2048, 2300)), (1280, 16, "bulk", 128, 150, (2048, 3100, 2400))])
def test_walks_handed_over_part_way(orc, side, tile, stage, batch, count, lens):
    import paper_2602_23040_gb300 as pk
    import synth
    rec = _records(side, _blocks(side, count, lens), side + count)
    n = len(rec)
    views = [synth.scenes.pinhole((0, 0, -3), side, side)]
    s = int(np.ceil(np.sqrt(n)))
    plan = pk.Plan([(s, s, 0, 0, 0)], (s, s), 0, 1, "f32", views, n, max_dups=4 * n, tile=tile, batch=batch,
                   stage_fwd=stage, stage_bwd=stage)
    ws = pk.make_workspace(plan)
    pk.workspace_init(plan, ws)
    drec = torch.from_numpy(rec.reshape(-1)).cuda()
    vals = torch.empty(plan.max_dups + 64, dtype=torch.int32, device="cuda")
    ranges = torch.empty(2 * plan.n_tiles, dtype=torch.int64, device="cuda")
    pk.bin_and_sort(plan, drec, vals, ranges, ws)
    out = {}
    whole = plan.with_options(count_evals=True)
    ws1 = pk.make_workspace(whole)
    pk.workspace_init(whole, ws1)
    for p, w_ in ((plan, ws), (whole, ws1)):
        img = torch.empty(3 * plan.P, dtype=torch.float32, device="cuda")
        T = torch.empty(plan.P, dtype=torch.float32, device="cuda")
        nc = torch.empty(plan.P, dtype=torch.int32, device="cuda")
        pk.rasterize_fwd(p, drec, vals, ranges, img, T, nc, w_)
        out[p is plan] = img, T, nc
    # lists handed over, by the workspace's counters (the RasterQueue of each pass behind two 64-bit counts):
    # in launches of so many CTAs only part way
    items = lambda k: int(ws.view(torch.int32)[(256 + 16 + 32 * k) // 4 + 2])
    assert items(0) > 0
    for a, b in zip(out[True], out[False]):
        assert torch.equal(a, b)
    img, T, nc = out[True]
    rec64 = rec.reshape(1, n, 12).astype(np.float64)
    va = orc.views_array(views)
    rvals, rranges = orc.bin_sort(rec64, va, tile)
    ref = orc.render(rec64, va, tile, rvals, rranges, m_tol=0.0)
    ref["view_pixels"] = [side * side]
    ref["border"] = ref["border"] & ~np.uint8(H.B_DEPTH)
    w = np.random.default_rng(n).standard_normal(3 * plan.P).astype(np.float32)
    w = H.zero_on_borderline(w, ref)
    g2 = torch.empty(12 * plan.pairs, dtype=torch.float32, device="cuda")
    pk.rasterize_bwd(plan, drec, vals, ranges, T, nc, torch.from_numpy(w).cuda(), g2, ws)
    assert items(1) > 0
    assert pk.read_status(plan, ws)["flags"] == 0
    got = g2.view(-1, 12).cpu().numpy().astype(np.float64)[:, :9]
    want = orc.render_bwd(rec64, va, tile, rvals, rranges, w.astype(np.float64)).reshape(-1, 9)
    for name, sl in {"mean": slice(0, 2), "conic": slice(2, 5), "opacity": slice(5, 6),
                     "colour": slice(6, 9)}.items():
        assert H.rel_err(got[:, sl], want[:, sl]) < H.GRAD_RTOL, name
