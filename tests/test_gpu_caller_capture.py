"""Steps captured into a graph of the caller's own: every replay goes on from the state the last one left."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("steps", [1, 2, 3])
def test_replays_of_captured_steps(precision, steps):
    import torch
    from paper_1707_04333_gb300 import fetdpic
    w = inputs.pair_plasma(14, 8, kT=0.2, wc_over_wp=0.5, seed=4)
    sims = [fetdpic.Simulation(w, precision=precision, sort_interval=-1, stream=torch.cuda.Stream(), use_torch=True).load()
            for _ in range(2)]
    a, b = sims
    for s in sims:
        s.step(1, "vay").sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=a.stream, capture_error_mode="thread_local"):
        a.step(steps, "vay")
    with torch.cuda.stream(a.stream):
        for _ in range(4):
            g.replay()
    b.step(4 * steps, "vay")
    for s in sims:
        s.sync()
    for x, y in zip(sims[0].species, sims[1].species):
        p, q = a.read_species(x[1]), b.read_species(y[1])
        assert all(np.array_equal(p[n], q[n]) for n in ("x", "u", "cell"))
    f, h = a.read_fields(), b.read_fields()
    assert all(np.array_equal(f[n], h[n]) for n in ("e", "b", "j"))
    del g
    for s in sims:
        s.close()
