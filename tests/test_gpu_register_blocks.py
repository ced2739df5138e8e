"""The registration fit with a block per frame: fit windows around a tile of
model values (512 pixels) and patches around the 32 x 128 pixels that one step
of the flood fill marks, against the FP64 oracle; a threshold below zero,
where the patch's centroid may lie far outside the frame.

Bounds: both sides stop within a drop of 1e-14 of the squared error of the
same minimum, which leaves 1e-6 px in the centre and 1e-5 relative in the
strongly correlated parameters (see the curvature argument of the
registration parity tests)."""
import math

import numpy as np
import pytest

import oracle
from paper_1510_04331_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1510_04331_gb300 import graphic
    return graphic


def _check(g, cube, thresh, R, mn, mx, w):
    got = g.context().graphic_register(torch.from_numpy(cube).cuda(), thresh, R, mn, mx, w).cpu().numpy()
    found = 0
    for t in range(cube.shape[0]):
        ok, cx, cy, sz = oracle.centroid(cube[t], thresh, R, mn, mx)
        assert (got[t, 0] == 1.0) == ok
        if not ok:
            assert not got[t].any()
            continue
        found += 1
        p, _ = oracle.moffat_fit(cube[t], cx, cy, max(1.0, math.sqrt(sz / math.pi)), w)
        want = np.array([p[1], p[2], oracle.moffat_fwhm(p[3], p[4]), p[0], p[3], p[4]])
        assert np.abs(got[t, 1:3] - want[:2]).max() <= 1e-6
        assert (np.abs(got[t, 3:7] - want[2:]) <= 1e-5 * np.abs(want[2:])).all()
    return found


@pytest.mark.parametrize("T,w", [(1, 10), (5, 11), (3, 15), (3, 16), (2, 32), (40, 5)])
def test_fit_windows_around_a_tile(g, T, w):
    """441 and 529 pixels (one tile, one and a remainder), 961 and 1089 (two,
    two and a remainder), 4225, 121 (fewer than the block's threads)."""
    d = synth.star_frames(T, 160, seed=300 + w, jitter=20.0, fwhm=4.0)
    assert _check(g, d.cube, 0.1 * d.peak, 16, 3, 600, w) == T


def test_serpentine_patch_of_the_whole_box(g):
    """R = 32 in a 65 x 65 frame: a box of 4225 pixels (more than one step
    marks) whose patch is one path winding through every other row, joined at
    alternating ends, so the labels travel backwards through the steps."""
    n = 65
    y, x = np.mgrid[0:n, 0:n]
    star = 1e4 / (1.0 + ((x - 32.2) ** 2 + (y - 31.9) ** 2) / 9.0) ** 2.5
    f = 10.0 + star + np.random.default_rng(7).normal(0.0, 0.1, (n, n))
    wall = (y % 2 == 1) & (x != np.where(y % 4 == 1, n - 1, 0))
    f[wall & (np.hypot(x - 32, y - 32) > 13)] = 0.0
    cube = np.stack([f, f[::-1, ::-1]]).astype(np.float32)
    seed = np.argmax(cube.reshape(2, -1), axis=1)
    assert (seed == 32 * n + 32).all()
    assert _check(g, cube, 5.0, 32, 1000, 5000, 8) == 2


def test_threshold_below_zero(g):
    """A patch of nearly balanced values: its centroid may be anywhere, the
    window may be empty; the call returns and the other frames are as alone."""
    rng = np.random.default_rng(8)
    cube = rng.normal(0.0, 1.0, (6, 48, 48)).astype(np.float32)
    cube[1] -= cube[1].mean()
    d = synth.star_frames(1, 48, seed=9, jitter=0.0)
    cube = np.concatenate([cube, d.cube])
    args = (-50.0, 24, 1, 5000, 6)
    got = g.context().graphic_register(torch.from_numpy(cube).cuda(), *args).cpu().numpy()
    alone = g.context().graphic_register(torch.from_numpy(d.cube).cuda(), *args).cpu().numpy()
    assert np.array_equal(got[6:], alone, equal_nan=True)
