"""Bad pixel map and correction where a call is refused, where a frame holds
more than 2^32 pixels, and where frames change from the listed fill to the
dense passes."""
import ctypes

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1510_04331_gb300 import graphic
    return graphic


@pytest.mark.parametrize("n", [7, 256])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_map_of_a_refused_frame_is_left_alone(g, n, value):
    ref = torch.randn((n, n), device="cuda")
    ref[n // 2, n - 1] = float(value)
    bad = torch.full((n, n), 7, dtype=torch.uint8, device="cuda")
    ctx = g.context()
    ctx._stream()
    rc = g.lib().graphic_bad_pixel_map(ctx.h, ctypes.c_void_p(ref.data_ptr()), n, 2.0, ctypes.c_void_p(bad.data_ptr()))
    assert rc == -5, rc
    assert bool((bad == 7).all())


def _room(gib):
    if torch.cuda.mem_get_info()[0] < gib * 2 ** 30:
        pytest.skip(f"needs {gib} GiB of device memory")


@pytest.mark.parametrize("case", ["one bin", "ramp"])
def test_map_of_frames_beyond_32_bit_counts(g, case):
    """One bin that holds more than 2^32 pixels; a ramp with more than 2^32 pixels in the bins below the middle's."""
    _room(60)
    if case == "one bin":
        n = 65600
        ref = torch.full((n, n), 2.5, device="cuda")
        ref[5] = 3.5
        want = np.arange(n) == 5
    else:
        n = 100000
        ref = torch.arange(n, dtype=torch.float32, device="cuda")[:, None].expand(n, n).contiguous()
        # n values of each row number: median (n - 1) / 2, sigma sqrt((n^2 - 1) / 12)
        want = np.abs(np.arange(n) - (n - 1) / 2) > np.sqrt((n * n - 1.0) / 12.0)
    got = g.context().graphic_bad_pixel_map(ref, 1.0)
    lo, hi = got.amin(dim=1).cpu().numpy(), got.amax(dim=1).cpu().numpy()
    assert np.array_equal(lo, want) and np.array_equal(hi, want)
    del ref, got
    torch.cuda.empty_cache()


def test_correction_of_a_frame_of_2_32_bad_pixels(g):
    _room(60)
    n = 65536
    ctx = g.Context(torch.cuda.current_device())   # its scratch, as large as the frame, goes with it
    try:
        x = torch.full((1, n, n), float("nan"), device="cuda")
        ctx._stream()
        rc = g.lib().graphic_bad_pixel_fix(ctx.h, ctypes.c_void_p(x.data_ptr()), 1, n, None)
        assert rc == -5, rc
        x.fill_(2.0)
        x[0, 7, 9] = float("inf")
        rc = g.lib().graphic_bad_pixel_fix(ctx.h, ctypes.c_void_p(x.data_ptr()), 1, n, None)
        assert rc == 0, rc
        assert bool((x == 2.0).all())
        del x
    finally:
        ctx.close()
    torch.cuda.empty_cache()


@pytest.mark.parametrize("T,n,counts", [
    # lists of up to 4096 + D n^2 / 320 pixels, D frames with more than 4096 + n^2 / 320
    (3, 256, [4300, 4301, 5]), (3, 256, [4505, 4506, 5]),
    (1, 512, [4915]), (1, 512, [4916]),
    # half a frame; the fills of more than 304 and of more than 608 frames
    (305, 64, [0, 1, 40, 2047, 2048, 2049, 3000, 4095]), (609, 64, [0, 1, 40, 2047, 2048, 2049, 3000, 4095]),
])
def test_correction_around_the_longest_list(g, T, n, counts):
    rng = np.random.default_rng(T + n)
    c = rng.normal(0, 1, (T, n, n)).astype(np.float32)
    for t in range(T):
        k = counts[t % len(counts)]
        where = np.arange(k) if t % 2 else rng.choice(n * n, k, replace=False)   # a block of rows, or anywhere
        c[t].ravel()[where] = np.nan
    want, st = oracle.bad_pixel_fix(c, None)
    assert st == 0
    x = torch.from_numpy(c).cuda()
    g.context().graphic_bad_pixel_fix(x)
    assert np.array_equal(x.cpu().numpy(), want)


def test_correction_of_a_frame_with_many_bad_pixels_uses_the_whole_chip(g):
    """40 % bad pixels may take a few times as long as 0.1 % (more pixels, some more passes); a frame filled by one
    block takes a hundred times as long."""
    n = 1024
    src = torch.randn((1, n, n), device="cuda")
    u = torch.rand((1, n, n), device="cuda")
    ms = []
    for share in (0.001, 0.4):
        bad = torch.where(u < share, torch.full_like(src, float("nan")), src)
        best = 1e9
        for _ in range(6):
            x = bad.clone()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.context().graphic_bad_pixel_fix(x)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    assert ms[1] < 10 * ms[0], ms
