"""Fields come back in the caller's order whichever of them are asked for, small (one copy through the
context's buffer) and large (a copy each)."""
import ctypes as C

import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


# 2 edges + 1 triangle values of 8 bytes on both sides of 384 KB (12,288 triangles)
@pytest.mark.parametrize("nx", [3, 77, 80])
def test_any_subset_equals_the_whole(nx):
    from paper_1707_04333_gb300 import fetdpic
    ws = [inputs.pair_plasma(n, 1, kT=0.1, wc_over_wp=0.5, seed=n) for n in (4, nx)]
    sim = fetdpic.Simulation(ws, precision="fp32").load()
    sim.step(3, "boris").sync()
    for inst in (0, 1):
        whole = sim.read_fields(inst)
        for names in ("e", "b", "j", "eb", "ej", "bj"):
            got = {n: np.full_like(whole[n], np.nan) for n in names}
            p = [got[n].ctypes.data_as(C.c_void_p) if n in got else None for n in "ebj"]
            assert fetdpic.lib().fetdpic_read(sim.h, inst, *p, 0, None, None, None) == 0
            assert all(np.array_equal(got[n], whole[n]) for n in names)
    sim.close()
