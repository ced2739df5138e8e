"""The allocation-free rotation on frames that start 4, 8 or 12 bytes past a
16-byte boundary: the same bits as on aligned frames, for every frame side and
quarter turn (exact quarter turns included), in place and out of place."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ANGLES = np.array([0.0, 33.0, 90.0, 101.5, 180.0, 171.25, 270.0, 291.0, -44.9, 44.9])


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_frames_at_any_float_address(n, offset):
    from paper_1510_04331_gb300 import graphic as g
    c = np.random.default_rng(n + offset).standard_normal((len(ANGLES), n, n)).astype(np.float32)
    c[:, 0] += 10.0
    c[:, :, 0] -= 10.0
    x = torch.from_numpy(c).cuda()
    want = g.graphic_rotate_noalloc(x, ANGLES, torch.empty_like(x))

    def shifted():
        return torch.zeros(x.numel() + offset, device="cuda")[offset:].view(x.shape)

    y, out = shifted().copy_(x), shifted()
    assert y.data_ptr() % 16 == 4 * offset
    assert torch.equal(g.graphic_rotate_noalloc(y, ANGLES, out), want)
    assert torch.equal(y, x)
    assert torch.equal(g.graphic_rotate_noalloc(y, ANGLES, y), want)
