"""General path of the median PSF subtraction (every frame ranked, one lane per
pixel): bit-exact against the oracle around the lengths where its ranking, its
maps and its chunks change (a map word, 256 counters or 1024, chunks of 32
queries), on values that defeat linear bins (ties, outliers, constants), in and
out of angle order, with a time gate and without, and where one 4-pixel group
has pixels of annuli with and without a rank band."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1510_04331_gb300 import graphic
    return graphic


def _values(T, n, rng):
    """Rows of the frame hold different kinds of values."""
    c = (rng.standard_normal((T, n, n)) * 30).astype(np.float32)
    c[:, 4:12] = rng.integers(-1, 2, (T, 8, n)).astype(np.float32)          # ties
    c[:, 12] = 7.25                                                         # constant
    out = rng.random((T, 6, n)) < 0.02
    c[:, 14:20][out] = np.where(rng.random(out.sum()) < 0.5, -1e30, 1e30)   # stretched range
    c[:, 20] = np.where(rng.random((T, n)) < 0.5, -0.0, 0.0)
    return c


@pytest.mark.parametrize("T", [1, 2, 31, 32, 33, 65, 256, 257, 600])
@pytest.mark.parametrize("sorted_frames", [True, False])
def test_general_path_bit_exact(g, T, sorted_frames):
    n = 64
    rng = np.random.default_rng(T)
    c = _values(T, n, rng)
    pa = np.sort(rng.uniform(-70, 70, T))
    times = np.linspace(0.0, 3.0, T)
    if not sorted_frames:
        p = rng.permutation(T)
        c, pa, times = c[p].copy(), pa[p].copy(), times[p].copy()
    edges = [0.0, 3.0, 9.0, 20.0, 40.0]
    pix = np.unique(np.concatenate([rng.choice(n * n, 60), np.arange(4 * n + 20, 21 * n, 37)]))
    for t_max in (0.25, 1.1, 50.0):
        got = g.graphic_adi_subtract(torch.from_numpy(c).cuda(), pa, 4.0, 1.5, edges, times=times,
                                     t_max=t_max).cpu().numpy()
        ref = oracle.adi_subtract(c, pa, 4.0, 1.5, edges, pixels=pix, times=times, t_max=t_max)
        assert np.array_equal(got.reshape(T, -1)[:, pix].T, ref)


@pytest.mark.parametrize("T", [1300, 2048])
def test_groups_shared_with_band_annuli(g, T):
    """Long sequence whose inner annuli have bands wider than 1024 ranks: their
    4-pixel groups also hold pixels of annuli with a band and of none."""
    n = 64
    rng = np.random.default_rng(T)
    c = _values(T, n, rng)
    pa = np.linspace(-75, 75, T) + rng.uniform(-0.02, 0.02, T)
    edges = [2.0, 3.5, 5.0, 6.5, 18.0, 29.0]
    x = torch.from_numpy(c).cuda()
    got = g.graphic_adi_subtract(x, pa, 4.0, 1.5, edges).cpu().numpy()
    yy, xx = np.mgrid[-32:32, -32:32]
    near = np.flatnonzero((xx * xx + yy * yy).ravel() <= 64)
    pix = np.unique(np.concatenate([near[::3], rng.choice(n * n, 20)]))
    ref = oracle.adi_subtract(c, pa, 4.0, 1.5, edges, pixels=pix)
    assert np.array_equal(got.reshape(T, -1)[:, pix].T, ref)
    g.graphic_adi_subtract(x, pa, 4.0, 1.5, edges, out=x)   # in place
    assert np.array_equal(x.cpu().numpy(), got)


def test_non_finite_input_is_reported_and_stays_in_bounds(g):
    T, n = 300, 64
    c = np.random.default_rng(1).standard_normal((T, n, n)).astype(np.float32)
    c[5, 30, 10:50] = np.nan
    c[:, 31, 20] = np.inf
    c[7, 32, 33] = -np.inf
    for kw in (dict(times=np.arange(T), t_max=40.0), {}):
        with pytest.raises(g.GraphicError, match="NONFINITE"):
            g.graphic_adi_subtract(torch.from_numpy(c).cuda(), np.linspace(-60, 60, T), 4.0, 1.5, [0.0, 9.0, 40.0], **kw)
