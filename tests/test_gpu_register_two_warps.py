"""Registration of many frames on small windows (two warps a frame) returns the
bits of the same frames in short calls (four warps a frame), for windows within
one tile and patch boxes larger than one step of the flood fill."""
import numpy as np
import pytest

from paper_1510_04331_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,w,T", [(6, 3, 977), (8, 5, 533), (16, 10, 977), (16, 10, 1611), (32, 8, 977), (32, 11, 977)])
def test_same_bits_as_short_calls(R, w, T):
    from paper_1510_04331_gb300 import graphic as g
    d = synth.star_frames(70, 96, seed=40 + w, jitter=10.0, fwhm=4.0, lost=0.15)
    few = torch.from_numpy(d.cube).cuda()
    x = few.repeat(-(-T // 70), 1, 1)[:T].contiguous()
    args = (0.1 * d.peak, R, 3, 600, w)
    it, it_few = (torch.zeros(len(c), dtype=torch.int32, device="cuda") for c in (x, few))
    got = g.graphic_register(x, *args, iters=it)
    want = g.graphic_register(few, *args, iters=it_few)
    idx = torch.arange(len(x), device="cuda") % len(few)
    assert want[:, 0].sum() > 40 and want[:, 0].sum() < 70
    assert torch.equal(got, want[idx]) and torch.equal(it, it_few[idx])
