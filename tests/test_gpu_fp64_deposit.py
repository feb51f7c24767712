"""FP64 path, particles of odd scales beside ordinary ones (integer and FP64 instructions in one warp): the
deposited current against the oracle's, and the Boris-tan pusher, whose tan is not correctly rounded."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu
C, QE, ME = inputs.C_LIGHT, inputs.Q_E, inputs.M_E


@pytest.mark.parametrize("pusher", ["boris", "boris_tan", "vay", "hc"])
@pytest.mark.parametrize("n,scale_e", [(1, 5e4), (33, 1e-140), (2049, 5e4), (2500, 0.0)])
def test_current_of_mixed_scales(pusher, n, scale_e):
    from oracle import oracle
    from paper_1707_04333_gb300 import fetdpic
    rng = np.random.default_rng(n)
    m = inputs.jittered_delaunay(9, 7, 1.0, 0.8, 0.3, seed=n)
    tri = np.sort(rng.integers(0, len(m.triangles), n)).astype(np.int32)
    x = inputs.sample_in_triangles(m, tri, rng)
    u = rng.normal(0, 0.8 * C, (n, 2))
    u[1::3] *= 1e-200                                      # the FP64 instructions; every third one at rest
    u[2::3] = 0.0
    w = inputs.Workload("mixed", m, [inputs.Species(-QE, ME, x, u, tri)], 2e-10)
    sim = fetdpic.Simulation(w, precision="fp64", spai_level=1, sort_interval=2).load()
    ora = oracle.OracleSim(m.nodes, m.triangles, w.dt, eps0=inputs.EPS0, mu0=inputs.MU0, c=C, spai_level=1,
                           b0=w.b0, e0=w.e0, ext=w.ext, max_cross=64)
    ora.load(-QE, ME, x, u, tri)
    om = ora.mesh
    e = rng.normal(0, scale_e, om.ne) * (om.edge_bnd == 0)
    b = rng.uniform(-0.01, 0.01, om.nf) * 0.5 * om.d2A
    fetdpic.fetdpic_write_fields(sim.h, 0, e, b)
    ora.e, ora.b = e.copy(), b.copy()
    for _ in range(3):
        sim.step(1, pusher).sync()
        ora.step(pusher)
        f, p, o = sim.read_fields(0), sim.read_species(0), ora.species[0]
        # half a quantum (q/dt 2^-52) a contribution, at most 8 contributions a particle on an edge, and the
        # oracle's FP64 sums; tan: 4 ulp of it, at most 1e-15 of u and of the step's length
        tan = 1e-13 if pusher == "boris_tan" else 0.0
        tol = 4 * n * QE / w.dt * 2.0 ** -52 + (1e-13 + 10 * tan) * np.abs(ora.i_abs).max()
        assert np.abs(f["j"] - ora.i).max() <= tol
        assert np.array_equal(p["cell"], o["cell"])
        assert np.abs(p["x"] - np.stack([o["x"], o["y"]], 1)).max() <= tan
        assert np.abs(p["u"] - np.stack([o["ux"], o["uy"]], 1)).max() <= tan * C
        # the oracle goes on from the library's state
        ora.e, ora.b = f["e"].copy(), f["b"].copy()
        o["x"], o["y"], o["ux"], o["uy"] = (np.ascontiguousarray(v) for v in (*p["x"].T, *p["u"].T))
    sim.close()
