"""fetdpic_check clears the maxima and take_status the status word in the context stream's order: steps
enqueued right behind keep what they find."""
import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_maxima_of_the_step_behind_a_check_survive():
    from paper_1707_04333_gb300 import fetdpic
    w = inputs.pair_plasma(6, 20, kT=0.2, wc_over_wp=0.5, seed=2)
    s = fetdpic.Simulation(w, precision="fp32", check_interval=1).load()
    s.step(1, "vay").sync()
    fetdpic.fetdpic_check(s.h, 0)
    for k in range(300):
        s.step(1, "vay")                       # nothing between the last check's clear and this step's maxima
        c = fetdpic.fetdpic_check(s.h, 0)
        assert c["dce"] > 0 and c["dgl"] > 0, k
    s.close()


def test_fault_behind_a_reported_fault_is_reported():
    from paper_1707_04333_gb300 import fetdpic
    m = inputs.jittered_delaunay(4, 4, 1.0, 1.0, 0.2, seed=1)
    w = inputs.Workload("f", m, [inputs.Species(-1e-18, 1e-18 * inputs.M_E / inputs.Q_E, np.array([[0.4, 0.45]]),
                                                np.zeros((1, 2)), np.full(1, -1, np.int32))], 1e-11)
    s = fetdpic.Simulation(w, precision="fp64").load()
    good = s.read_species(0)
    for k in range(100):
        fetdpic.fetdpic_write_particles(s.h, 0, good["x"], good["u"], np.array([len(m.triangles) + 3], np.int32))
        with pytest.raises(fetdpic.FetdpicError) as ei:
            s.sync()
        assert ei.value.code == fetdpic.EINVAL, k
    s.close()
