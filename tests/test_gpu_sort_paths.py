"""bin_and_sort on every way its radix passes find their digits' positions
(one block's own count, the parts' counts added up, the scanned counters) and
with depths that span 1 float to the whole range (a pass whose digit is 0 in
every key is left out): every tile's list equal to the oracle's, called twice
on one workspace."""

import numpy as np
import pytest

from tests import helpers as H
from tests.test_gpu_parity import _records_plan, _synthetic_records, assert_same_tile_lists

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# (views, pairs per view): one block of 1 and 2 tiles of pairs and one pair
# more (3,072 pairs a tile); parts added up; and scanned (over 64 parts)
SIZES = [(1, 6), (1, 3072), (1, 6144), (1, 6145), (3, 4000), (1, 30000), (1, 230000), (7, 9001)]


@pytest.mark.parametrize("V,N", SIZES)
@pytest.mark.parametrize("bits", [8, 11])
def test_positions_of_digits(orc, V, N, bits):
    _check(orc, V, N, bits, None)


@pytest.mark.parametrize("span", [0, 1, 255, 256, 65535, 65536, (1 << 24) - 1, 1 << 24, (1 << 22) - 1, 1 << 22, 1 << 11])
@pytest.mark.parametrize("bits", [8, 11])
def test_depth_spans(orc, span, bits):
    _check(orc, 2, 3500, bits, span)


def _check(orc, V, N, bits, span):
    import paper_2602_23040_gb300 as pk
    import synth
    views = [synth.scenes.pinhole((0, 0, -3), 150 - 16 * v, 100 + 9 * v) for v in range(V)]
    rec = _synthetic_records(views, N, 31 * V + N + bits, huge=N < 10000)
    rec[..., 7] = np.minimum(rec[..., 7], 4000 if N < 10000 else 12)
    if N == 6:
        rec[..., 0:2], rec[..., 7] = 20.0, 6.0
    if span is not None:
        # the nearest and the farthest pair `span` floats apart, the others between
        rng = np.random.default_rng(span)
        z = np.float32(1.5).view(np.uint32) + rng.integers(0, span + 1, (V, N)).astype(np.uint32)
        rec[..., 6] = z.view(np.float32)
        for k, at in ((1, 0), (2, span)):
            rec[0, k, :8] = (30.0, 30.0, 0.5, 0.0, 0.5, 0.5, (np.float32(1.5).view(np.uint32) + np.uint32(at)).view(np.float32), 6.0)
    for tile in (16, 32):
        plan = _records_plan(views, N, "ellipse", tile, sort_bits_depth=bits, sort_bits_tile=bits)
        ws = pk.make_workspace(plan)
        pk.workspace_init(plan, ws)
        drec = torch.from_numpy(rec.reshape(-1)).cuda()
        r = rec.reshape(V * N, 12)
        ref_vals, ref_ranges = orc.bin_sort32(r[:, 0], r[:, 1], r[:, 7], r[:, 6], orc.views_array(views), N, tile,
                                              r[:, 2], r[:, 3], r[:, 4], mode=orc.BIN_ELLIPSE)
        for _ in range(2):
            vals = torch.empty(plan.max_dups + 64, dtype=torch.int32, device="cuda")
            ranges = torch.full((2 * plan.n_tiles,), 5, dtype=torch.int64, device="cuda")
            pk.bin_and_sort(plan, drec, vals, ranges, ws)
            st = pk.read_status(plan, ws)
            assert st["dups"] == len(ref_vals) and st["flags"] == 0
            assert_same_tile_lists(H.u32(vals[:len(ref_vals)]), H.i64(ranges).reshape(-1, 2), ref_vals, ref_ranges)
