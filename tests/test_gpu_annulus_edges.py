"""Annulus membership in integers: edges whose squares are whole, a rounding
away from whole, between the same two whole numbers (an annulus without a
pixel), beyond every pixel and overflowing when squared, on the band path and
on the general path (time gate), against the FP32 oracle bit for bit (medians
and one FP32 difference)."""
import numpy as np
import pytest

import oracle
from paper_1510_04331_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [
    [0.0, 5.0, np.nextafter(13.0, 0), 25.0, 46.0],
    [np.nextafter(5.0, 9), np.sqrt(50.0), np.nextafter(np.sqrt(50.0), 9), 20.01, 20.02, 31.0],
    [3.0, 1e200],
    [0.5, 7.2, 60.0, 1e9],
    [70.0, 80.0],
]


@pytest.mark.parametrize("edges", EDGES)
@pytest.mark.parametrize("gate", [False, True])
def test_edges_at_and_between_whole_squares(edges, gate):
    from paper_1510_04331_gb300 import graphic as g
    T, n = 40, 64
    d = synth.make_cube(T, n, seed=5, parang=np.linspace(-60, 60, T), edges=np.array([4.0, 46.0]))
    e = np.array(edges)
    kw = dict(times=np.arange(T, dtype=float), t_max=7.5) if gate else {}
    args = (d.parang, d.fwhm, d.n_fwhm, e)
    got = g.graphic_adi_subtract(torch.from_numpy(d.cube).cuda(), *args, **kw).cpu().numpy()
    want = oracle.adi_subtract(d.cube, *args, **kw)
    assert np.array_equal(got, want.astype(np.float32))
