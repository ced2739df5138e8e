"""Master sky of up to 64 frames at every width of its register network and the
lengths beside it, with masks, non-finite values, ties and signed zeros: the
oracle's bits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [2, 3, 4, 5, 6, 7, 8, 10, 11, 12, 13, 20, 21, 24, 25, 40, 41, 63])
def test_sky_median_widths(T):
    from paper_1510_04331_gb300 import graphic as g
    n = 64
    rng = np.random.default_rng(100 + T)
    c = rng.normal(0.0, 1.0, (T, n, n)).astype(np.float32)
    c[rng.random(c.shape) < 0.1] = np.nan
    c[:, 5, 9] = -np.inf
    c[:, 20:24] = rng.integers(-1, 2, (T, 4, n))
    c[:, 7] = np.where(rng.random((T, n)) < 0.5, -0.0, 0.0)
    mx, my = rng.integers(5, 60, T).astype(float), rng.integers(5, 60, T).astype(float)
    x = torch.from_numpy(c).cuda()
    for args in ((), (mx, my, 9.5)):
        got, want = g.context().graphic_sky_median(x, *args).cpu().numpy(), oracle.sky_median(c, *args)
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(got[~np.isnan(got)].view(np.uint32), want[~np.isnan(want)].view(np.uint32))
