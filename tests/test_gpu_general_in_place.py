"""General median PSF path in place: what a call refuses and what it returns
are those of the call out of place, where a segment of 8 pixels holds pixels of
no annulus or of several annuli, and where the units' tables go through the
scratch in several chunks, the last one ragged."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1510_04331_gb300 import graphic
    return graphic


@pytest.mark.parametrize("row,col", [(32, 33), (32, 31), (32, 54), (13, 24)])
def test_non_finite_pixel_of_no_annulus(g, row, col):
    """Pixels inside the first and outside the last edge, 8-pixel segments that also hold pixels of the annulus."""
    T, n = 40, 64
    c = np.random.default_rng(3).standard_normal((T, n, n)).astype(np.float32)
    c[3, row, col] = np.nan
    pa = np.linspace(-60, 60, T)
    x = torch.from_numpy(c).cuda()
    for out in (torch.empty_like(x), x):
        with pytest.raises(g.GraphicError, match="NONFINITE"):
            g.graphic_adi_subtract(x, pa, 4.0, 1.5, [5.0, 20.0], out=out, times=np.arange(T), t_max=20.0)


@pytest.mark.parametrize("sorted_frames", [True, False])
def test_several_chunks_of_units(g, sorted_frames):
    T, n = 2048, 256
    edges = [0.0, 30.0, 60.0, 90.0, 130.0, 190.0]
    yy, xx = np.mgrid[-n // 2:n // 2, -n // 2:n // 2]
    rho2 = xx * xx + yy * yy
    # a unit of 32 pixels has 32 x 6 bytes of tables per frame, the scratch is 256 MiB: three chunks if every unit
    # were full, and segments with pixels of two annuli are in a unit of each
    assert n * n // 32 * T * 32 * 6 >= 3 * (256 << 20)
    gen = torch.Generator(device="cuda").manual_seed(11)
    x = torch.randn((T, n, n), device="cuda", generator=gen)
    # pixels on the inner side of the edge at 60, in segments that also hold
    # pixels beyond it: finite values whose residuals overflow
    seg = np.arange(n * n) // 8
    inner, outer = ((rho2 >= 900) & (rho2 < 3600)).ravel(), ((rho2 >= 3600) & (rho2 < 8100)).ravel()
    shared = np.flatnonzero(inner & np.isin(seg, seg[outer]))
    flat = x.view(T, -1)
    flat[:, torch.from_numpy(shared).cuda()] = -3.0e38
    flat[T // 2, torch.from_numpy(shared).cuda()] = 3.0e38
    pa, times = np.linspace(-75, 75, T), np.linspace(0.0, 3.0, T)
    if not sorted_frames:
        p = np.random.default_rng(5).permutation(T)
        x = x[torch.from_numpy(p).cuda()].contiguous()
        pa, times = pa[p], times[p]
    out = g.graphic_adi_subtract(x, pa, 4.0, 1.5, edges, times=times, t_max=0.3)
    c = x.cpu().numpy()
    g.graphic_adi_subtract(x, pa, 4.0, 1.5, edges, out=x, times=times, t_max=0.3)
    assert torch.equal(x, out)
    # pixels all over every annulus' units, the last ones of each among them
    pix = []
    for lo, hi in zip(edges[:-1], edges[1:]):
        a = np.flatnonzero(((rho2 >= lo * lo) & (rho2 < hi * hi)).ravel())
        pix += list(a[np.linspace(0, a.size - 1, 9).astype(int)])
    pix = np.unique(pix + [int(shared[0]), int(shared[-1])])
    ref = oracle.adi_subtract(c, pa, 4.0, 1.5, edges, pixels=pix, times=times, t_max=0.3)
    assert np.array_equal(out.view(T, -1)[:, torch.from_numpy(pix).cuda()].cpu().numpy().T, ref)
