"""The autotuner also tries the default where that is a pair of kernels without a number of its own
(above 2 M particles, pushers other than Vay); the state is left as it was."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_autotune_with_an_unnumbered_default():
    from paper_1707_04333_gb300 import fetdpic
    w = inputs.pair_plasma(190, 16, kT=0.2, wc_over_wp=0.5, seed=3, pusher="hc")      # 2.3 M particles
    a, b = (fetdpic.Simulation(w, precision="fp32", use_graphs=True).load() for _ in range(2))
    for s in (a, b):
        s.step(3, "hc").sync()
    v, interval = a.autotune("hc", trial_steps=8)
    assert v in (0, *range(2, 23)) and v != 1 and interval in (8, 12, 16, 32)
    fetdpic.fetdpic_set_tuning(a.h, v, interval)                                       # 0 is taken back too
    for s in (a, b):
        s.step(20, "hc").sync()
    for k in range(2):
        p, q = a.read_species(k), b.read_species(k)
        assert all(np.array_equal(p[n], q[n]) for n in ("x", "u", "cell"))
    f, g = a.read_fields(), b.read_fields()
    assert all(np.array_equal(f[n], g[n]) for n in ("e", "b", "j"))
    a.close()
    b.close()
