"""FP32 path above gamma = 10: on both sides of each line between the double-float push and the one in FP64
(gamma^2 = 1e17, kick and |beta| of gamma / 8, |beta| of gamma / 31.6 for Boris-tan), against FP64 numpy."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs
from test_gpu_high_gamma_push import _push

pytestmark = pytest.mark.gpu
C = inputs.C_LIGHT


@pytest.mark.parametrize("pusher", ["boris", "boris_tan", "vay", "hc"])
@pytest.mark.parametrize("line,lo,hi,bz,ex", [("gamma", 2e8, 5e8, 0.3, 0.2), ("beta", 400.0, 1600.0, 100.0, 0.0),
                                              ("kick", 400.0, 1600.0, 1.0, 100.0), ("angle", 1600.0, 6400.0, 100.0, 0.5)])
def test_push_beside_a_switch(pusher, line, lo, hi, bz, ex):
    from paper_1707_04333_gb300 import fetdpic
    rng = np.random.default_rng(11)
    n = 4096
    g = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    th = rng.uniform(0, 2 * np.pi, n)
    p = np.sqrt(g * g - 1.0)
    u = np.stack([p * np.cos(th), p * np.sin(th)], 1).astype(np.float32).astype(np.float64)
    mesh = inputs.jittered_delaunay(8, 8, 1.0, 1.0, 0.2, seed=3)
    x = rng.uniform(0.3, 0.7, (n, 2))
    dt, kappa = 1e-12, -inputs.Q_E / inputs.M_E
    w = inputs.Workload("hg", mesh, [inputs.Species(-inputs.Q_E, inputs.M_E, x, u * C, np.full(n, -1, np.int32))], dt,
                        b0=2 * bz / (kappa * dt), ext=(2 * C * ex / (kappa * dt), 0.0, 0.0), pusher=pusher)
    sim = fetdpic.Simulation(w, precision="fp32", spai_level=1).load()
    u0 = (u * C * (1.0 / C)).astype(np.float32).astype(np.float64)
    sim.step(1, pusher).sync()
    got = sim.read_species(0)["u"] / C
    sim.close()
    want = np.stack(_push(pusher, u0[:, 0], u0[:, 1], ex, bz), 1)
    # half a unit of the last place; 4 roundings of eps (twice) and of beta; 2^-44 of |u| for the push's own
    eps = 2.0 ** -24
    mag = np.hypot(want[:, 0], want[:, 1])[:, None]
    tol = eps * np.abs(want) * (1 + 1e-6) + 8 * eps * abs(ex) + 4 * eps * abs(bz) + 2.0 ** -44 * mag
    bad = np.abs(got - want) > tol
    assert not bad.any(), (g[bad.any(1)][:5], (np.abs(got - want) / tol).max())
