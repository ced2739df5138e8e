"""A recorded batch graph names the plan buffers it was recorded with: a call
that makes the context replace them (a longer plan) must not leave the graph to
be replayed, also when the new buffers take the old ones' addresses."""
import numpy as np
import pytest

from paper_1510_04331_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["PERSISTENT", "GROUPED"])
def test_batch_after_the_plan_grew(mode):
    from paper_1510_04331_gb300 import graphic as g
    batch = synth.uneven_batch(seed=3, n_cubes=5, sides=(64, 128), t_range=(1, 9))
    cubes = [torch.from_numpy(b[0]).cuda() for b in batch]
    args = [b[1] for b in batch], [b[2] for b in batch], [b[3] for b in batch]
    ctx = g.Context(0)
    want = [o.cpu().numpy() for o in ctx.graphic_batch_geom(cubes, *args, mode=getattr(g, "BATCH_" + mode))]
    for T, n in ((40, 64), (300, 64), (1500, 128)):   # each with a longer plan than the last
        x = torch.randn((T, n, n), device="cuda")
        ctx.graphic_adi_subtract(x, np.linspace(-60, 60, T), 4.0, 1.5, synth.default_edges(n))
        for o, w in zip(ctx.graphic_batch_geom(cubes, *args, mode=getattr(g, "BATCH_" + mode)), want):
            assert np.array_equal(o.cpu().numpy(), w)
    ctx.close()
