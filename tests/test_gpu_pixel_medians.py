"""Register-network medians (binning, master sky), the device-side bad pixel
map and the listed bad pixel correction at the sizes where they switch form:
every network width and its neighbours, masks whose rim passes through pixel
centres or that lie far off, frames more than half bad, odd sides and
unaligned cubes.  All selections or exact arithmetic: compared bit for bit
with the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1510_04331_gb300 import graphic
    return graphic


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _same(a, b):
    return np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(a[~np.isnan(a)].view(np.uint32),
                                                                       b[~np.isnan(b)].view(np.uint32))


@pytest.mark.parametrize("B", [3, 4, 5, 6, 7, 8, 9, 11, 12, 13, 15, 19, 20, 21, 23, 24, 25, 31, 33, 39, 40, 41, 49, 51,
                               63])
def test_bin_median_every_network(g, B):
    rng = np.random.default_rng(B)
    c = rng.standard_normal((2 * B + B // 2 + 1, 64, 64)).astype(np.float32)   # ragged last bin
    c[:, :8] = rng.integers(-1, 2, c[:, :8].shape) * np.float32(0.5)           # ties
    c[:, 8][rng.random(c[:, 8].shape) < 0.7] = -0.0
    c[:, 9] = np.where(rng.random(c[:, 9].shape) < 0.5, -0.0, 0.0)
    assert _same(g.context().graphic_bin_median(_dev(c), B).cpu().numpy(), oracle.bin_median(c, B))


@pytest.mark.parametrize("T", [1, 2, 8, 9, 16, 17, 32, 33, 50, 51, 64, 65])
def test_sky_median_every_network(g, T):
    rng = np.random.default_rng(T)
    n = 64
    c = rng.normal(0.0, 1.0, (T, n, n)).astype(np.float32)
    c[rng.random(c.shape) < 0.1] = np.nan
    c[rng.random(c.shape) < 0.02] = np.inf
    c[:, 5, 9] = np.nan
    c[:, 7] = np.where(rng.random((T, n)) < 0.5, -0.0, 0.0)
    # integer centres and radius 5: rim pixels at exactly 25 stay; then a mask
    # over the whole frame, masks far off, one not a number
    mx, my = rng.integers(5, 60, T).astype(float), rng.integers(5, 60, T).astype(float)
    mx[1::7] += 1e-13
    my[2::7] = 1e9
    mx[3::7] = np.nan
    mx[4::7] = 3.0e6
    for r in (5.0, 0.0, 13.7, 2000.0):
        got = g.context().graphic_sky_median(_dev(c), mx, my, r).cpu().numpy()
        assert _same(got, oracle.sky_median(c, mx, my, r))
    assert _same(g.context().graphic_sky_median(_dev(c)).cpu().numpy(), oracle.sky_median(c))


@pytest.mark.parametrize("n", [1, 2, 7, 33, 100, 256])
def test_bad_pixel_map_sizes(g, n):
    rng = np.random.default_rng(n)
    for ref in (rng.normal(-3.0, 2.0, (n, n)), rng.integers(0, 3, (n, n)), np.full((n, n), 2.5),
                rng.normal(0, 1, (n, n)) * 10.0 ** rng.integers(-30, 30, (n, n))):
        ref = ref.astype(np.float32)
        got = g.context().graphic_bad_pixel_map(_dev(ref), 2.0).cpu().numpy().astype(bool)
        assert np.array_equal(got, oracle.bad_pixel_map(ref, 2.0))
    ref = np.ones((n, n), np.float32)
    ref[-1, -1] = np.inf
    with pytest.raises(g.GraphicError, match="NONFINITE"):
        g.context().graphic_bad_pixel_map(_dev(ref), 2.0)


@pytest.mark.parametrize("n,offset", [(64, 0), (65, 0), (64, 1), (130, 2)])
def test_bad_pixel_fix_sparse_and_dense_frames(g, n, offset):
    """Frames a few, just half, more than half and almost all bad, in one
    cube; odd sides and cubes that start off a 16-byte boundary."""
    rng = np.random.default_rng(n + offset)
    c = rng.normal(0, 1, (6, n, n)).astype(np.float32)
    c[0, 3:9, 4:10] = np.nan
    c[1][rng.random((n, n)) < 0.3] = np.inf
    c[2].ravel()[rng.choice(n * n, n * n // 2, replace=False)] = np.nan
    c[3, : n // 2 + 3] = np.nan
    c[4] = np.nan
    c[4, n // 3, n - 1] = 4.0
    bad = np.zeros((n, n), np.uint8)
    bad[-1, -1] = 7
    for cube in (c, c[:3] * np.float32(1.0), c[:2].copy()):
        want, st = oracle.bad_pixel_fix(cube, bad.astype(bool))
        assert st == 0
        buf = torch.empty(cube.size + offset, dtype=torch.float32, device="cuda")
        x = buf[offset:].view(cube.shape)
        x.copy_(torch.from_numpy(cube))
        g.context().graphic_bad_pixel_fix(x, _dev(bad))
        assert np.array_equal(x.cpu().numpy(), want)
