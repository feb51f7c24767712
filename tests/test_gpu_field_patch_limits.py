"""Patches of the field update whose tables need more shared memory than every kernel may use, and more
than any block gets (there the separate kernels run): bit for bit the whole-mesh update, with contexts of
different needs alive together."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


def _scattered(nx, seed):
    """A fine square whose triangles, in no order, share one cell of the space-filling curve because two
    more triangles lie far away: a patch's triangles are no neighbours, so it needs many other edges."""
    m = inputs.jittered_delaunay(nx, nx, 1e-10, 1e-10, 0.2, seed=seed)
    rng = np.random.default_rng(seed)
    n = len(m.nodes)
    nodes = np.concatenate([m.nodes, np.array([[1.0, 1.0], [1.001, 1.0], [1.001, 1.001], [1.0, 1.001]])])
    tri = np.concatenate([m.triangles[rng.permutation(len(m.triangles))], [[n, n + 1, n + 2], [n, n + 2, n + 3]]]).astype(np.int32)
    mesh = inputs.Mesh(nodes, tri, m.lx, m.ly)
    x = rng.uniform(2e-11, 8e-11, (500, 2))
    u = rng.normal(0, 0.3 * inputs.C_LIGHT, (500, 2))
    h = 1e-10 / nx
    s = inputs.Species(-1e-18, 1e-18 * inputs.M_E / inputs.Q_E, x, u, np.full(500, -1, np.int32))
    return inputs.Workload("scattered", mesh, [s], 0.02 * h / inputs.C_LIGHT, b0=0.01)


def _state(sim):
    f, p = sim.read_fields(), sim.read_species(0)
    return [f["e"], f["b"], f["j"], p["x"], p["u"], p["cell"]]


def _equal(a, b):
    return all(np.array_equal(x, y) for x, y in zip(_state(a), _state(b)))


# shared memory a block, host build of the tables: 80 KB, 60 KB, 139 KB (the three separate kernels)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("graphs", [False, True])
def test_contexts_with_large_patches_live_together(precision, graphs):
    from paper_1707_04333_gb300 import fetdpic

    def sim(nx, level, whole=False):
        return fetdpic.Simulation(_scattered(nx, nx), precision=precision, spai_level=level, sort_interval=4,
                                  use_graphs=graphs and not whole, fuse_field_update=whole).load()
    shapes = [(60, 7), (45, 7), (90, 9)]
    sims = [sim(*s) for s in shapes]
    for s, shape in zip(sims, shapes):                     # the first one steps after all were created
        whole = sim(*shape, whole=True)
        for n in (1, 8, 3):
            s.step(n, "boris").sync()
            whole.step(n, "boris").sync()
            assert _equal(s, whole), (shape, n)
        assert np.abs(_state(s)[0]).max() > 0
        whole.close()
    for s in sims:
        s.close()


def _clustered(nx, level, side=112):
    """The square in no order of nx x nx cells beside an ordinary one: the patches pay on the whole, and
    those of the cluster are large."""
    w = _scattered(nx, nx)
    m = inputs.jittered_delaunay(side, side, 1.0, 1.0, 0.2, seed=7)
    n = len(w.mesh.nodes)
    nodes = np.concatenate([w.mesh.nodes, m.nodes + 1.5])
    w.mesh = inputs.Mesh(nodes, np.concatenate([w.mesh.triangles, m.triangles + n]).astype(np.int32), 3.0, 3.0)
    return w


@pytest.mark.parametrize("graphs", [False, True])
def test_large_patches_among_small_ones(graphs):
    """55 and 50 KB a block (host build of the tables); the first context steps after the second exists."""
    from paper_1707_04333_gb300 import fetdpic

    def sim(level, whole=False):
        return fetdpic.Simulation(_clustered(42, level), precision="fp32", spai_level=level, sort_interval=-1,
                                  use_graphs=graphs and not whole, fuse_field_update=whole).load()
    sims = [sim(7), sim(6)]
    for s, level in zip(sims, (7, 6)):
        whole = sim(level, True)
        s.step(1, "boris").sync()
        whole.step(1, "boris").sync()
        fetdpic.fetdpic_stage_times(s.h)
        s.step(8, "boris").sync()
        whole.step(8, "boris").sync()
        # Faraday, then particles and one field launch a step: the patches are in use
        assert fetdpic.fetdpic_stage_times(s.h)[1] == 17
        assert _equal(s, whole)
        whole.close()
    for s in sims:
        s.close()
