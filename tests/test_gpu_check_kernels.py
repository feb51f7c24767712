"""Check kernels where warps straddle triangles, species, instances and the padding: nodal charge and
field energy against plain sums."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


def _workload(n, seed, ppt):
    """n triangles a side; ppt particles per triangle in two species of different weights."""
    m = inputs.jittered_delaunay(n, n, 1.0, 1.0, 0.3, seed=seed)
    rng = np.random.default_rng(seed)
    sp = []
    for q, k in ((-1.0, ppt), (0.37, max(1, ppt // 3))):
        tri = np.repeat(np.arange(len(m.triangles), dtype=np.int32), k)
        x = inputs.sample_in_triangles(m, tri, rng)
        sp.append(inputs.Species(q * 1e-12, 1e-20, x, rng.normal(0, 1e7, (len(x), 2)), tri))
    return inputs.Workload("check", m, sp, 1e-11, b0=0.01)


def _charge(m, x, cell, q):
    """sum Q lambda_i(r) per node, FP64."""
    p = m.nodes[m.triangles[cell]]
    d = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1])
    out = np.zeros(len(m.nodes))
    for k in range(3):
        a, b = p[:, (k + 1) % 3], p[:, (k + 2) % 3]
        lam = ((a[:, 0] - x[:, 0]) * (b[:, 1] - x[:, 1]) - (b[:, 0] - x[:, 0]) * (a[:, 1] - x[:, 1])) / d
        np.add.at(out, m.triangles[cell][:, k], q * lam)
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("ppt", [1, 7, 33, 100])
def test_charge_and_energy(precision, ppt):
    """Charge within 1e-6 (FP32: rounding of lambda and of the quantum) or 1e-12 of a node's total, and
    the energy of each instance, over instances of different sizes in one context.  (The residuals
    themselves are held to the exact integer sums in test_gpu_conservation.py.)"""
    from paper_1707_04333_gb300 import fetdpic
    ws = [_workload(9, 1, ppt), _workload(4, 2, ppt), _workload(13, 3, 2)]
    sim = fetdpic.Simulation(ws, precision=precision, check_interval=2, sort_interval=3).load()
    sim.step(6, "boris").sync()
    for k, w in enumerate(ws):
        got, _ = fetdpic.fetdpic_read_charge(sim.h, k)
        want, total = np.zeros(len(w.mesh.nodes)), np.zeros(len(w.mesh.nodes))
        for (inst, sid, _), s in zip(sim.species, [s for v in ws for s in v.species]):
            if inst == k:
                p = sim.read_species(sid)
                want += _charge(w.mesh, p["x"], p["cell"], s.q)
                total += _charge(w.mesh, p["x"], p["cell"], abs(s.q))
        assert (np.abs(got - want) <= (1e-6 if precision == "fp32" else 1e-12) * total.max()).all()
        c, f = fetdpic.fetdpic_check(sim.h, k), sim.read_fields(k)
        # the magnetic part of the energy from the faces: b^2 / (2 mu0 A), and the electric part is positive
        t = w.mesh.nodes[w.mesh.triangles]
        area = 0.5 * np.abs((t[:, 1, 0] - t[:, 0, 0]) * (t[:, 2, 1] - t[:, 0, 1]) -
                            (t[:, 2, 0] - t[:, 0, 0]) * (t[:, 1, 1] - t[:, 0, 1]))
        mag = (f["b"] ** 2 / (2 * inputs.MU0 * area)).sum()
        assert c["energy"] > mag * (1 - 1e-12)
        single = fetdpic.Simulation(w, precision=precision, check_interval=6, sort_interval=-1).load()
        single.step(6, "boris").sync()
        # the same instance alone: the same state, the same energy but for the order of its sum
        assert abs(fetdpic.fetdpic_check(single.h, 0)["energy"] - c["energy"]) <= 1e-13 * c["energy"]
        single.close()
    sim.close()
