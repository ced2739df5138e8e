"""Median collapse of up to 64 frames (register network) and just above: every
network width and its neighbours, strided frames, an output that is not
8-byte aligned (the warp-per-pixel kernels), non-finite input.  A selection
and one FP32 average: compared bit for bit with the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1510_04331_gb300 import graphic
    return graphic.context()


def _cube(T, n=64):
    rng = np.random.default_rng(T)
    c = rng.standard_normal((T, n, n)).astype(np.float32)
    c[:, :8] = rng.integers(-1, 2, c[:, :8].shape) * np.float32(0.5)
    c[:, 9] = np.where(rng.random(c[:, 9].shape) < 0.5, -0.0, 0.0)
    c[:, 10] = np.float32(3.4e38) * np.sign(c[:, 10])
    return c


@pytest.mark.parametrize("T", [1, 2, 3, 5, 7, 9, 11, 13, 16, 17, 21, 24, 25, 32, 33, 40, 41, 50, 51, 63, 64, 65])
def test_collapse_around_every_network(ctx, T):
    c = _cube(T)
    want = oracle.collapse_median(c).astype(np.float32)
    x = torch.from_numpy(c).cuda()
    assert np.array_equal(ctx.graphic_collapse_median(x).cpu().numpy().view(np.uint32), want.view(np.uint32))
    # a row of the frame between frames, so that the stride is not n^2
    y = torch.zeros((T, 65, 64), device="cuda")
    y[:, :64] = x
    s = y[:, :64]
    assert T == 1 or not s.is_contiguous()
    assert np.array_equal(ctx.graphic_collapse_median_cube(s).cpu().numpy().view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("T", [4, 33, 64, 65])
def test_collapse_refuses_what_is_not_finite(ctx, T):
    from paper_1510_04331_gb300 import graphic
    for v in (np.nan, np.inf, -np.inf):
        c = _cube(T)
        c[T // 2, 63, 63] = v
        with pytest.raises(graphic.GraphicError, match="NONFINITE"):
            ctx.graphic_collapse_median(torch.from_numpy(c).cuda())


@pytest.mark.parametrize("T", [20, 65])
def test_reduction_into_an_image_of_any_alignment(ctx, T):
    from paper_1510_04331_gb300 import synth
    d = synth.make_cube(T, 64, seed=T, parang=np.linspace(-40, 40, T), edges=synth.default_edges(64))
    x = torch.from_numpy(d.cube).cuda()
    args = (d.dx, d.dy, d.parang, d.fwhm, d.n_fwhm, d.edges)
    want = ctx.graphic_reduce(x, *args).cpu().numpy()
    out = torch.full((64 * 64 + 2,), 7.0, device="cuda")
    got = ctx.graphic_reduce(x, *args, out=out[1:-1].view(64, 64)).cpu().numpy()
    assert np.array_equal(got, want)
    assert out[0] == 7.0 and out[-1] == 7.0
