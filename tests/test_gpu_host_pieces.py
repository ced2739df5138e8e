"""graphic_reduce_host copies and shifts the cube in pieces of an eighth of it
(16 to 256 MiB): one piece, whole pieces, a ragged last piece, and pieces cut
again by the scratch chunks, equal to the device path bit for bit (the same
kernels on the same frames)."""
import numpy as np
import pytest

from paper_1510_04331_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,n,chunk_mb", [(12, 64, None), (32, 512, None), (41, 512, None), (9, 1024, None),
                                          (41, 512, "5")])
def test_pieces_equal_the_device_path(T, n, chunk_mb, monkeypatch):
    from paper_1510_04331_gb300 import graphic as g
    d = synth.make_cube(T, n, seed=T, parang=np.linspace(-40, 40, T), edges=synth.default_edges(n))
    x = torch.from_numpy(d.cube).cuda()
    a = g.graphic_reduce(x, d.dx, d.dy, d.parang, d.fwhm, d.n_fwhm, d.edges).cpu().numpy()
    if chunk_mb:
        monkeypatch.setenv("GRAPHIC_CHUNK_MB", chunk_mb)
    b = g.graphic_reduce_host(d.cube, d.dx, d.dy, d.parang, d.fwhm, d.n_fwhm, d.edges)
    assert np.array_equal(a, b)
