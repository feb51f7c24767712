"""Nodal charge of species whose charges differ by hundreds of orders of magnitude: the small one's rounds
to nothing."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("ratio", [1e-120, 1e-240, 1e-300, 1e-308, 0.0])
def test_charge_of_a_vanishing_species(precision, ratio):
    from paper_1707_04333_gb300 import fetdpic
    m = inputs.jittered_delaunay(4, 4, 1.0, 1.0, 0.2, seed=1)
    tri = np.arange(len(m.triangles), dtype=np.int32)
    corner = m.nodes[m.triangles]
    # on the first corner but for rounding: barycentric coordinates down to 1e-17 and below
    x = corner[:, 0] + 1e-30 * (corner[:, 1] - corner[:, 0])
    mid = corner.mean(1)
    u = np.zeros_like(x)
    big = inputs.Species(-1e-9, 1e-20, mid, u, tri)
    out = []
    for species in ([big], [big, inputs.Species(-1e-9 * ratio, 1e-20, x, u, tri), inputs.Species(1e-9 * ratio, 1e-20, mid, u, tri)]):
        s = fetdpic.Simulation(inputs.Workload("q", m, species, 1e-11), precision=precision).load()
        out.append(fetdpic.fetdpic_read_charge(s.h, 0)[0])
        s.close()
    assert np.array_equal(*out)
