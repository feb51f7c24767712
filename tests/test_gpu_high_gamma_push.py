"""FP32 path, gamma > 10: the double-float push against plain FP64 numpy on the same FP32 inputs."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu
C = inputs.C_LIGHT


def _push(pusher, ux, uy, ex, bz):
    """Momentum (units of c) after one push, FP64; eps = (ex, 0), beta = bz."""
    def gam(a, b):
        return np.sqrt(1.0 + a * a + b * b)
    if pusher == "vay":
        g0 = gam(ux, uy)
        px, py = ux + 2 * ex + uy / g0 * bz, uy - ux / g0 * bz
        sig = 1.0 + px * px + py * py - bz * bz
        t = bz / np.sqrt(0.5 * (sig + np.sqrt(sig * sig + 4 * bz * bz)))
        return (px + py * t) / (1 + t * t), (py - px * t) / (1 + t * t)
    mx, my = ux + ex, uy
    g = gam(mx, my)
    if pusher == "hc":
        sig = g * g - bz * bz
        t = bz / np.sqrt(0.5 * (sig + np.sqrt(sig * sig + 4 * bz * bz)))
    else:
        t = np.tan(bz / g) if pusher == "boris_tan" else bz / g
    s = 2 * t / (1 + t * t)
    rx, ry = mx + my * t, my - mx * t
    return mx + ry * s + ex, my - rx * s


@pytest.mark.parametrize("pusher", ["boris", "boris_tan", "vay", "hc"])
@pytest.mark.parametrize("bz,ex", [(0.05, 0.0), (0.3, 0.2), (20.0, -3.0)])
def test_high_gamma_push_rounds_like_fp64(pusher, bz, ex):
    """gamma from just above 10 to 1e9 (beyond 1e9, and at |beta| > gamma / 2, the FP64 form runs).
    A component may differ by half a unit in its last FP32 place, plus what the FP32 fields carry:
    4 roundings of eps (twice), 4 of beta times |u| / gamma <= 1, and 2^-41 of |u| for the
    double-float arithmetic."""
    from paper_1707_04333_gb300 import fetdpic
    rng = np.random.default_rng(7)
    n = 4096
    g = np.exp(rng.uniform(np.log(10.2), np.log(3e9), n))
    th = rng.uniform(0, 2 * np.pi, n)
    p = np.sqrt(g * g - 1.0)
    u = np.stack([p * np.cos(th), p * np.sin(th)], 1).astype(np.float32).astype(np.float64)
    mesh = inputs.jittered_delaunay(8, 8, 1.0, 1.0, 0.2, seed=3)
    x = rng.uniform(0.3, 0.7, (n, 2))
    dt, kappa = 1e-12, -inputs.Q_E / inputs.M_E
    b0, e_ext = 2 * bz / (kappa * dt), 2 * C * ex / (kappa * dt)
    w = inputs.Workload("hg", mesh, [inputs.Species(-inputs.Q_E, inputs.M_E, x, u * C, np.full(n, -1, np.int32))], dt,
                        b0=b0, ext=(e_ext, 0.0, 0.0), pusher=pusher)
    sim = fetdpic.Simulation(w, precision="fp32", spai_level=1).load()
    u0 = (u * C * (1.0 / C)).astype(np.float32).astype(np.float64)
    sim.step(1, pusher).sync()
    got = sim.read_species(0)["u"] / C
    sim.close()
    want = np.stack(_push(pusher, u0[:, 0], u0[:, 1], ex, bz), 1)
    eps = 2.0 ** -24
    mag = np.hypot(want[:, 0], want[:, 1])[:, None]
    tol = eps * np.abs(want) * (1 + 1e-6) + 8 * eps * abs(ex) + 4 * eps * abs(bz) + 2.0 ** -41 * mag
    bad = np.abs(got - want) > tol
    assert not bad.any(), (g[bad.any(1)][:5], (np.abs(got - want) / tol).max())
