"""FP64 path at |beta| = |q B dt / 2m| where the quartic's gamma cancels: the oracle's bits as long as it
is above zero, and ENONFINITE, not a finite momentum, where sigma + sqrt(sigma^2 + 4 beta^2) is exactly 0."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu
C, QE, ME = inputs.C_LIGHT, inputs.Q_E, inputs.M_E


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("pusher,log2_beta", [(p, b) for p in ("boris", "vay", "hc") for b in (10.0, 25.5, 26.0, 28.0, 40.3)])
def test_strong_field_push(pusher, log2_beta, sign):
    from oracle import oracle
    from paper_1707_04333_gb300 import fetdpic
    rng = np.random.default_rng(5)
    n, dt = 300, 1e-10
    m = inputs.jittered_delaunay(6, 5, 1.0, 0.8, 0.3, seed=2)
    tri = np.sort(rng.integers(0, len(m.triangles), n)).astype(np.int32)
    x, u = inputs.sample_in_triangles(m, tri, rng), rng.normal(0, 0.5 * C, (n, 2))
    bz = sign * 2.0 ** log2_beta / (QE * dt / (2.0 * ME))
    w = inputs.Workload("strong", m, [inputs.Species(QE, ME, x, u, tri)], dt, ext=(0.0, 0.0, bz))
    sim = fetdpic.Simulation(w, precision="fp64", spai_level=1, sort_interval=-1).load()
    lost = pusher != "boris" and log2_beta >= 28.0
    if lost:
        with pytest.raises(fetdpic.FetdpicError) as ei:
            sim.step(1, pusher).sync()
        assert ei.value.code == fetdpic.ENONFINITE
    else:
        ora = oracle.OracleSim(m.nodes, m.triangles, dt, eps0=inputs.EPS0, mu0=inputs.MU0, c=C, spai_level=1,
                               b0=w.b0, e0=w.e0, ext=w.ext, max_cross=64)
        ora.load(QE, ME, x, u, tri)
        sim.step(1, pusher).sync()
        ora.step(pusher)
        got, o = sim.read_species(0), ora.species[0]
        assert np.array_equal(got["cell"], o["cell"])
        assert np.array_equal(got["x"], np.stack([o["x"], o["y"]], 1))
        assert np.array_equal(got["u"], np.stack([o["ux"], o["uy"]], 1))
    sim.close()
