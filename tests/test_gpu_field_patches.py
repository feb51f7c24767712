"""Field update by patches, with the next step's Faraday in the same launch, against the one
cooperative launch over the whole mesh (fuse_field_update): bit for bit, over the meshes, inverses and
ways of stepping a context takes."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu
C = inputs.C_LIGHT


def _plasma(nx, ny, ppc, seed, **kw):
    return inputs.pair_plasma(nx, ppc, kT=0.2, wc_over_wp=0.5, seed=seed, ny=ny, **kw)


def _single(nx):
    """One particle on a mesh of 2 nx^2 triangles (nx = 1: two triangles, one free edge)."""
    m = inputs.jittered_delaunay(nx, nx, 1.0, 1.0, 0.2, seed=4)
    x, u = np.array([[0.41, 0.37]]), np.array([[0.3 * C, -0.5 * C]])
    return inputs.Workload("one", m, [inputs.Species(-1e-9, 1e-9 * inputs.M_E / inputs.Q_E, x, u, np.full(1, -1, np.int32))],
                           1e-10, b0=0.01)


def _beam():
    w = inputs.high_gamma_beam(n_tri_side=20, n_particles=3000, seed=3, side=1.0)
    rng = np.random.default_rng(1)
    w.ext_profile = rng.uniform(0, 2, (len(w.mesh.triangles), 2))
    return w


CASES = {
    "two_triangles": lambda: [_single(1)],
    "one_patch": lambda: [_single(5)],
    "patch_edge": lambda: [_plasma(8, 8, 3, 1)],               # 128 triangles: two patches of 64
    "ragged": lambda: [_plasma(23, 17, 2, 2)],
    "strip": lambda: [_plasma(40, 4, 4, 3, periodic_y=True)],
    "applied": lambda: [_beam()],
    "batch": lambda: [_plasma(9, 7, 3, 5), _single(3), _plasma(14, 11, 1, 6), _plasma(31, 30, 2, 7)],
    "large_patch": lambda: [_plasma(190, 170, 1, 8)],          # 64,600 triangles: patches above 128
}


def _state(sim):
    out = []
    for k in range(len(sim.workloads)):
        f = sim.read_fields(k)
        out += [f["e"], f["b"], f["j"]]
    for s in range(len(sim.species)):
        p = sim.read_species(s)
        out += [p["x"], p["u"], p["cell"]]
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("graphs,sort", [(False, 3), (True, 4), (True, 3), (True, -1)])
@pytest.mark.parametrize("name,level", [(n, 2) for n in CASES] + [("ragged", 1), ("ragged", 3), ("batch", 4), ("patch_edge", -1)])
def test_patches_equal_the_whole_mesh_update(precision, graphs, sort, name, level):
    from paper_1707_04333_gb300 import fetdpic
    sims = [fetdpic.Simulation(CASES[name](), precision=precision, spai_level=level, sort_interval=sort,
                               use_graphs=graphs and not whole, fuse_field_update=whole).load() for whole in (False, True)]
    rng = np.random.default_rng(0)
    for n in (1, 5, 8, 2):
        for s in sims:
            s.step(n, "vay").sync()
        a, b = _state(sims[0]), _state(sims[1])
        assert all(np.array_equal(x, y) for x, y in zip(a, b)), (name, n)
        e, bb = rng.normal(0, 1e3, len(a[0])), rng.normal(0, 1e-6, len(a[1]))
        for s in sims:                                         # the buffers may have changed places
            fetdpic.fetdpic_write_fields(s.h, 0, e, bb)
    for s in sims:
        s.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_fields_without_particles(precision):
    """No particle kernel between the field kernels: the curl waits for Faraday's result."""
    from paper_1707_04333_gb300 import fetdpic
    w = _plasma(30, 28, 1, 9)
    w.species = []
    out = []
    for whole in (False, True):
        s = fetdpic.Simulation(w, precision=precision, fuse_field_update=whole).load()
        rng = np.random.default_rng(2)
        f = s.read_fields()
        fetdpic.fetdpic_write_fields(s.h, 0, rng.normal(0, 1, len(f["e"])), rng.normal(0, 1e-9, len(f["b"])))
        s.step(37, "boris").sync()
        f = s.read_fields()
        out.append((f["e"], f["b"], f["j"]))
        s.close()
    assert all(np.array_equal(x, y) for x, y in zip(*out)) and np.abs(out[0][0]).max() > 0
