"""General median PSF path with few units, whose sweep goes in chunks of a few
queries: bit-exact against the oracle on every pixel of the annuli, for lengths
that leave short last chunks and warps without one."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 3, 4, 5, 7, 63, 130, 301, 1029])
@pytest.mark.parametrize("edges", [[5.0, 6.0], [3.0, 9.0, 13.0]])
def test_few_units(T, edges):
    from paper_1510_04331_gb300 import graphic as g
    n = 64
    rng = np.random.default_rng(T)
    c = rng.standard_normal((T, n, n)).astype(np.float32)
    c[:, :, ::3] = rng.integers(-2, 3, c[:, :, ::3].shape)
    pa, times = np.linspace(-65, 65, T), np.linspace(0.0, 3.0, T)
    yy, xx = np.mgrid[-n // 2:n // 2, -n // 2:n // 2]
    rho2 = (xx * xx + yy * yy).ravel()
    pix = np.flatnonzero((rho2 >= edges[0] ** 2) & (rho2 < edges[-1] ** 2))[::1 if T < 1000 else 7]
    for t_max in (0.4, 50.0):
        got = g.graphic_adi_subtract(torch.from_numpy(c).cuda(), pa, 4.0, 1.5, edges, times=times, t_max=t_max)
        ref = oracle.adi_subtract(c, pa, 4.0, 1.5, edges, pixels=pix, times=times, t_max=t_max)
        assert np.array_equal(got.cpu().numpy().reshape(T, -1)[:, pix].T, ref)
