"""Master sky of more than 64 frames with star masks and without, in shared
memory and beyond it (more than 8192 frames): the oracle's bits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [65, 300, 8192, 8193])
@pytest.mark.parametrize("stars", [False, True])
def test_sky_median_long_stacks(T, stars):
    from paper_1510_04331_gb300 import graphic as g
    n = 64
    rng = np.random.default_rng(T)
    c = rng.standard_normal((T, n, n)).astype(np.float32)
    c[rng.random(c.shape) < 0.05] = np.nan
    c[:, 5, 9] = np.inf
    c[:, 7] = np.where(rng.random((T, n)) < 0.5, -0.0, 0.0)
    c[:, 11] = rng.integers(-1, 2, (T, n))
    args = (rng.uniform(5, 60, T), rng.uniform(5, 60, T), 8.0) if stars else ()
    got = g.context().graphic_sky_median(torch.from_numpy(c).cuda(), *args).cpu().numpy()
    want = oracle.sky_median(c, *args)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[~np.isnan(got)].view(np.uint32), want[~np.isnan(want)].view(np.uint32))
