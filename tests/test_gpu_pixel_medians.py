"""Register-network medians of the binning at every network width and its
neighbours, compared bit for bit with the oracle."""
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
