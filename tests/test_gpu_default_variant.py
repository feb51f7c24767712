"""The particle kernels that variant 0 chooses by size, density and pusher: the same bits as a named one."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


# at most a chunk per SM; few particles per triangle; early and late kernels at both late choices
@pytest.mark.parametrize("nx,ppc", [(4, 1), (70, 2), (24, 20), (190, 16)])
@pytest.mark.parametrize("pusher", ["boris", "vay"])
@pytest.mark.parametrize("steps", [(1, 4, 11, 3), (19,)])
def test_default_equals_named_variant(nx, ppc, pusher, steps):
    from paper_1707_04333_gb300 import fetdpic
    w = inputs.pair_plasma(nx, ppc, kT=0.2, wc_over_wp=0.5, seed=3, pusher=pusher)
    sims = [fetdpic.Simulation(w, precision="fp32", sort_interval=8, use_graphs=g, kernel_variant=v).load()
            for v, g in ((0, True), (10, False))]
    for n in steps:
        for s in sims:
            s.step(n, pusher).sync()
    for k in range(2):
        a, b = (s.read_species(k) for s in sims)
        assert all(np.array_equal(a[n], b[n]) for n in ("x", "u", "cell"))
    a, b = (s.read_fields() for s in sims)
    assert all(np.array_equal(a[n], b[n]) for n in ("e", "b", "j"))
    for s in sims:
        s.close()
