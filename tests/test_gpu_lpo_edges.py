"""Codes of the low-precision proxy at the edges of its steps: values at and
within a few ulps of the rounding boundaries, where a product with the
step's reciprocal and the quotient may round apart, over ranges from
denormal to huge steps, full and partly live groups of four.  Bit for bit
the oracle's codes, and the same codes through the gather of the masters."""

import numpy as np
import pytest

from tests.test_gpu_lpo import Lpo, _scene, pk  # noqa: F401

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


@pytest.mark.parametrize("W", [128, 125])
@pytest.mark.parametrize("scale", [1.0, 1e-36, 3e33])
def test_codes_at_step_boundaries(pk, orc, W, scale):  # noqa: F811
    sc = _scene(W, seed=905)
    a = sc.atlas
    F, D, Ha, Wa = a.shape
    rng = np.random.default_rng(906)
    f32 = np.float32
    for c in range(D):
        steps = 65535 if c < 3 else 255
        lo, hi = f32(-0.7 * scale * (1 + c)), f32(1.3 * scale * (1 + c))
        delta = f32((hi - lo) / f32(steps))
        k = rng.integers(0, steps, (F, Ha, Wa))
        x = (np.float64(lo) + (k + 0.5) * np.float64(delta)).astype(f32)   # on a boundary
        bits = x.view(np.int32) + rng.integers(-3, 4, x.shape, dtype=np.int32)   # and a few ulps off
        x = np.clip(bits.view(f32), lo, hi)
        pick = rng.random(x.shape)
        x[pick < 0.05] = lo
        x[pick > 0.95] = hi
        a[:, c] = x
    run = Lpo(pk, sc)
    lohi, codes = run.run()
    np.testing.assert_array_equal(lohi.view(np.uint32), orc.lpo_minmax(a, sc.occ).view(np.uint32))
    np.testing.assert_array_equal(codes, orc.lpo_encode(a, sc.occ, lohi))
    from_codes = run.gather(pk.api.LPO_CODES)
    np.testing.assert_array_equal(run.gather(pk.api.LPO_MASTERS).view(np.uint32), from_codes.view(np.uint32))
