"""FP64 path: the particles whose push runs in integer arithmetic and those that fall back to the FP64
instructions both match the oracle bit for bit."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu
C, QE, ME = inputs.C_LIGHT, inputs.Q_E, inputs.M_E


def _setup(n, jitter, q, ext, seed):
    rng = np.random.default_rng(seed)
    m = inputs.jittered_delaunay(9, 7, 1.0, 0.8, jitter, seed=seed)
    tri = np.sort(rng.integers(0, len(m.triangles), n)).astype(np.int32)
    x = inputs.sample_in_triangles(m, tri, rng)
    u = rng.normal(0, 0.8 * C, (n, 2))
    u[::5] = 0.0                                       # at rest
    u[1::7, 1] = 0.0
    u[2::11] *= 1e-40                                  # below the integer form's range
    u[3::13] *= 1e-200
    w = inputs.Workload("arith", m, [inputs.Species(q, ME, x, u, tri)], 2e-10, ext=ext)
    return w, rng


# the second field set mixes scales: zero, far below and inside the integer form's range
@pytest.mark.parametrize("scale_e", [5e4, 1e-30, 1e-140, 0.0])
@pytest.mark.parametrize("n,jitter,q,ext", [(1, 0.3, -QE, (0.0, 0.0, 0.0)), (33, 0.0, -QE, (0.0, 0.0, 0.0)),
                                            (2049, 0.3, 0.0, (0.0, 0.0, 0.0)), (2050, 0.0, QE, (1e4, -3e3, 0.01)),
                                            (1500, 0.3, QE, (1e-130, 0.0, 0.0))])
@pytest.mark.parametrize("pusher", ["boris", "vay", "hc"])
@pytest.mark.parametrize("block", [32, 256])
def test_fp64_push_bits(scale_e, n, jitter, q, ext, pusher, block):
    from oracle import oracle
    from paper_1707_04333_gb300 import build_lib, fetdpic
    build_lib.build()
    oracle.build()
    w, rng = _setup(n, jitter, q, ext, n + 1)
    sim = fetdpic.Simulation(w, precision="fp64", spai_level=1, record_walk=16, sort_interval=2, block_size=block).load()
    ora = oracle.OracleSim(w.mesh.nodes, w.mesh.triangles, w.dt, eps0=inputs.EPS0, mu0=inputs.MU0, c=C, spai_level=1,
                           b0=w.b0, e0=w.e0, ext=w.ext, max_cross=64)
    s = w.species[0]
    ora.load(s.q, s.m, s.x, s.u, s.hint)
    om = ora.mesh
    e = rng.normal(0, scale_e, om.ne) * (om.edge_bnd == 0)
    e[::3] *= 1e-20
    b = rng.uniform(-0.01, 0.01, om.nf) * 0.5 * om.d2A
    fetdpic.fetdpic_write_fields(sim.h, 0, e, b)
    ora.e, ora.b = e.copy(), b.copy()
    for _ in range(3):
        sim.step(1, pusher).sync()
        ora.step(pusher)
        # the oracle goes on from the library's fields: only the particle arithmetic is compared
        f = sim.read_fields(0)
        ora.e, ora.b = f["e"].copy(), f["b"].copy()
        got = sim.read_species(0)
        o = ora.species[0]
        assert np.array_equal(got["cell"], o["cell"])
        assert np.array_equal(got["x"], np.stack([o["x"], o["y"]], 1))
        assert np.array_equal(got["u"], np.stack([o["ux"], o["uy"]], 1))
    sim.close()
