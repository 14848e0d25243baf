"""Lists long enough to be spread over several CTAs (128 entries and up in a
small launch): forward and backward against the oracle on the same FP32
records, around the shortest such list, at remainders of the batches and
segments, and with longer segments; the forward bit for bit as the counting
variant, which walks every list whole.  Saturated, rim and untouched pixels
share the blocks."""

import numpy as np
import pytest

from tests import helpers as H

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _records(n, side, seed):
    """n splats of about 1.5 px, all in a view's one tile: 7 in 8 within its
    dense left half (opaque: its pixels pass the cutoff), the others thin and
    spread, none near the right edge."""
    rng = np.random.default_rng(seed)
    rec = np.zeros((n, 12), np.float32)
    dense = rng.random(n) < 0.875
    rec[:, 0] = np.where(dense, rng.normal(0.25 * side, 0.09 * side, n), rng.uniform(2.0, 0.85 * side, n))
    rec[:, 1] = rng.uniform(2.0, side - 2.0, n)
    np.clip(rec[:, 0], 1.0, 0.85 * side, out=rec[:, 0])
    rec[:, 2] = rng.uniform(0.5, 1.5, n)
    rec[:, 3] = rng.uniform(-0.3, 0.3, n)
    rec[:, 4] = rng.uniform(0.5, 1.5, n)
    rec[:, 5] = np.where(dense, rng.uniform(0.01, 0.9, n), rng.uniform(0.004, 0.05, n))
    rec[:, 6] = rng.permutation(n) / n * 4.0 + 1.0
    rec[:, 7] = 5.0
    rec[:, 8:11] = rng.uniform(0, 1, (n, 3))
    return rec


@pytest.mark.parametrize("n,tile,stage", [(127, 32, "loads"), (128, 32, "loads"), (129, 32, "bulk"), (640, 16, "loads"),
                                          (3333, 16, "bulk"), (20011, 32, "loads"), (70001, 32, "loads")])
def test_long_lists_match_the_oracle(orc, n, tile, stage):
    import paper_2602_23040_gb300 as pk
    import synth
    side = tile
    views = [synth.scenes.pinhole((0, 0, -3), side, side)]
    rec = _records(n, side, n)
    s = int(np.ceil(np.sqrt(n)))
    plan = pk.Plan([(s, s, 0, 0, 0)], (s, s), 0, 1, "f32", views, n, max_dups=2 * n + 1024, tile=tile,
                   stage_fwd=stage, stage_bwd=stage)
    ws = pk.make_workspace(plan)
    pk.workspace_init(plan, ws)
    drec = torch.from_numpy(rec.reshape(-1)).cuda()
    vals = torch.empty(plan.max_dups + 64, dtype=torch.int32, device="cuda")
    ranges = torch.empty(2 * plan.n_tiles, dtype=torch.int64, device="cuda")
    img, img1 = (torch.empty(3 * plan.P, dtype=torch.float32, device="cuda") for _ in range(2))
    T = torch.empty(plan.P, dtype=torch.float32, device="cuda")
    nc = torch.empty(plan.P, dtype=torch.int32, device="cuda")
    pk.bin_and_sort(plan, drec, vals, ranges, ws)
    pk.rasterize_fwd(plan, drec, vals, ranges, img1, T, nc, ws)
    pk.rasterize_fwd(plan, drec, vals, ranges, img, T, nc, ws)
    assert torch.equal(img, img1)   # the same bits from run to run
    st = pk.read_status(plan, ws)
    assert st["flags"] == 0 and st["dups"] == n
    rec64 = rec.reshape(1, n, 12).astype(np.float64)
    rec64[..., 11] = 0
    va = orc.views_array(views)
    rvals, rranges = orc.bin_sort(rec64, va, tile)
    ref = orc.render(rec64, va, tile, rvals, rranges, m_tol=0.0)
    ref["view_pixels"] = [side * side]
    ref["border"] = ref["border"] & ~np.uint8(H.B_DEPTH)
    H.check_images(img.cpu().numpy(), T.cpu().numpy(), ref, tol=2e-5, max_border_frac=0.05, max_threshold_frac=0.05,
                   label=f"{n} entries, tile {tile}")
    ok = (ref["border"] & H.IMAGE_BORDER) == 0
    assert np.array_equal(H.u32(nc)[ok], ref["last"][ok])
    assert (ref["last"] > 64).any()
    q = plan.with_options(count_evals=True)
    ws1 = pk.make_workspace(q)
    pk.workspace_init(q, ws1)
    T1, nc1 = torch.empty_like(T), torch.empty_like(nc)
    pk.rasterize_fwd(q, drec, vals, ranges, img1, T1, nc1, ws1)
    assert torch.equal(img, img1) and torch.equal(T, T1) and torch.equal(nc, nc1)
    w = np.random.default_rng(n + 1).standard_normal(3 * plan.P).astype(np.float32)
    w = H.zero_on_borderline(w, ref)
    g2 = torch.empty(12 * plan.pairs, dtype=torch.float32, device="cuda")
    pk.rasterize_bwd(plan, drec, vals, ranges, T, nc, torch.from_numpy(w).cuda(), g2, ws)
    got = g2.view(-1, 12).cpu().numpy().astype(np.float64)[:, :9]
    want = orc.render_bwd(rec64, va, tile, rvals, rranges, w.astype(np.float64)).reshape(-1, 9)
    for name, sl in {"mean": slice(0, 2), "conic": slice(2, 5), "opacity": slice(5, 6),
                     "colour": slice(6, 9)}.items():
        assert H.rel_err(got[:, sl], want[:, sl]) < 1e-3, name
    assert pk.read_status(plan, ws)["flags"] == 0
