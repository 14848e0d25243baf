"""UV cells where FP32 cannot tell neighbouring cells apart (cell edges, the
poles, values whose squares leave FP32's range) and at the sizes around one
block's share of Gaussians: cells, ranks, keep flags and counts equal to the
FP64 oracle's."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pk():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_23040_gb300 as pk
    pk.build.build()
    return pk


def _run(pk, soa, M, N, K):
    n = soa.shape[1]
    cell, rank = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    keep = torch.empty(n, dtype=torch.uint8, device="cuda")
    count = torch.empty(M * N, dtype=torch.int32, device="cuda")
    pk.uv_max_k(torch.from_numpy(soa).cuda(), n, M, N, K, cell, rank, keep, count)
    torch.cuda.synchronize()
    u32 = lambda t: t.cpu().numpy().view(np.uint32)
    return dict(cell=u32(cell), rank=u32(rank), keep=keep.cpu().numpy(), count=u32(count))


@pytest.mark.parametrize("n,M,N", [(1, 8, 4), (2047, 64, 32), (2048, 1024, 1024), (2049, 5000, 3000), (6151, 37, 19)])
def test_uv_cells_at_cell_edges(pk, orc, n, M, N):
    rng = np.random.default_rng(n)
    # half on cell edges to FP32 rounding, half anywhere
    u = rng.integers(0, M, n) + np.where(rng.random(n) < 0.5, 0.0, rng.random(n))
    v = rng.integers(0, N, n) + np.where(rng.random(n) < 0.5, 0.0, rng.random(n))
    theta, phi = u / M * 2 * np.pi - np.pi, v / N * np.pi
    rho = 10.0 ** rng.choice([-18.0, -3.0, 0.0, 3.0, 18.0], n)   # squares below, inside and above FP32's range
    soa = np.zeros((14, n), np.float32)
    soa[0], soa[1], soa[2] = rho * np.sin(phi) * np.cos(theta), rho * np.sin(phi) * np.sin(theta), rho * np.cos(phi)
    pole = rng.random(n) < 0.05                                   # within FP32 rounding of the poles
    soa[:2, pole] *= np.float32(1e-7)
    soa[10] = np.round(rng.normal(0.0, 1.0, n), 1)
    got = _run(pk, soa, M, N, 2)
    want = orc.uv_max_k(soa.astype(np.float64), M, N, 2)
    for k in ("cell", "rank", "keep"):
        ok = want["border"] == 0
        if k != "cell":   # a borderline Gaussian may change its neighbours' ranks
            ok &= ~np.isin(want["cell"], np.r_[want["cell"][want["border"] != 0], got["cell"][want["border"] != 0]])
        np.testing.assert_array_equal(got[k][ok], want[k][ok], err_msg=k)
    assert got["count"].sum() == (got["cell"] != orc.INVALID).sum()
