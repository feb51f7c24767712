"""Sorted contexts equal never-sorted ones bit for bit on both sides of the size from which contexts are
sorted (2,048 slots), with several species, beside the checks and with graphs."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


# particles per species and triangles per side: 2 x 1024 slots, one more species' worth, many
@pytest.mark.parametrize("n,nx,species", [(1024, 6, 2), (1025, 6, 2), (300, 6, 3), (40000, 40, 2), (9000, 90, 2)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("check,graphs", [(0, True), (0, False), (2, False)])
def test_sort_changes_nothing(n, nx, species, precision, check, graphs):
    from paper_1707_04333_gb300 import fetdpic
    m = inputs.jittered_delaunay(nx, nx, 1.0, 1.0, 0.3, seed=2)
    rng = np.random.default_rng(n)
    sp = []
    for k in range(species):
        tri = rng.integers(0, len(m.triangles), n).astype(np.int32)
        sp.append(inputs.Species((-1) ** k * 1e-13, 1e-24, inputs.sample_in_triangles(m, tri, rng),
                                 rng.normal(0, 2e8, (n, 2)), tri))
    w = inputs.Workload("sort", m, sp, 0.1 / nx / 3e8, b0=1e-3)
    sims = [fetdpic.Simulation(w, precision=precision, sort_interval=s, use_graphs=graphs, check_interval=check).load()
            for s in (3, -1)]
    for steps in (3, 4, 6, 1):
        for s in sims:
            s.step(steps, "boris").sync()
        for k in range(species):
            a, b = (s.read_species(k) for s in sims)
            assert all(np.array_equal(a[i], b[i]) for i in ("x", "u", "cell"))
        a, b = (s.read_fields() for s in sims)
        assert all(np.array_equal(a[i], b[i]) for i in ("e", "b", "j"))
        if check:
            a, b = (fetdpic.fetdpic_check(s.h, 0) for s in sims)
            assert a["dce"] == b["dce"] and a["dgl"] == b["dgl"] and a["energy"] == b["energy"]
    for s in sims:
        s.close()
