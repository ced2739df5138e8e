"""Shift and rotation passes at every line length and quarter turn (rows,
staged columns, columns read backwards, frames in and out of place), against
the FP64 oracle to 1e-5 of the frame peak; and frames that start 8 but not 16
bytes into a buffer through the allocation-free rotation."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ANGLES = np.array([0.0, 33.0, 90.0, 101.5, 180.0, 171.25, 270.0, 291.0, -44.9, 44.9])


@pytest.fixture(scope="module")
def g():
    from paper_1510_04331_gb300 import graphic
    return graphic


def _frames(n, seed):
    """Noise with a bright off-centre pixel, and a bright border: every row and column counts."""
    c = np.random.default_rng(seed).standard_normal((len(ANGLES), n, n)).astype(np.float32)
    c[:, n // 3, n - 2] = 50.0
    c[:, 0] += 10.0
    c[:, :, 0] -= 10.0
    return c


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024])
def test_every_quarter_turn_and_size(g, n):
    c = _frames(n, n)
    x = torch.from_numpy(c).cuda()
    tol = 1e-5 * np.abs(c).max()
    got = g.graphic_rotate(x, ANGLES).cpu().numpy()
    assert np.abs(got - oracle.rotate(c.astype(np.float64), ANGLES)).max() <= tol
    d = np.linspace(-3.3, 2.9, len(ANGLES))
    got = g.graphic_shift(x, d, d[::-1].copy(), out=x).cpu().numpy()
    assert np.abs(got - oracle.shift(c.astype(np.float64), d, d[::-1].copy())).max() <= tol


@pytest.mark.parametrize("n", [64, 128, 256])
def test_frames_off_a_16_byte_boundary(g, n):
    c = torch.from_numpy(_frames(n, n + 1)).cuda()
    buf = torch.empty(c.numel() + 2, device="cuda")
    x = buf[2:].view(c.shape)
    x.copy_(c)
    want = g.graphic_rotate_noalloc(c, ANGLES, torch.empty_like(c))
    assert torch.equal(g.graphic_rotate_noalloc(x, ANGLES, x), want)
