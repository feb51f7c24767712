"""A read of fields and particles that fails for want of memory has finished its field copies."""
import ctypes as C

import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_failed_read_leaves_no_copy_in_flight(monkeypatch):
    import torch
    from paper_1707_04333_gb300 import fetdpic
    allocator, fail = fetdpic._torch_allocator, []

    def limited():
        alloc, free = allocator()

        @fetdpic._ALLOC
        def some(nbytes, user):
            return None if fail else alloc(nbytes, user)
        keep.append(alloc)
        return some, free
    keep = []
    monkeypatch.setattr(fetdpic, "_torch_allocator", limited)
    w = inputs.pair_plasma(160, 2, kT=0.2, wc_over_wp=0.5, seed=4)
    s = fetdpic.Simulation(w, precision="fp32").load()
    s.step(1, "vay").sync()
    n, ne = s.species[0][2], len(s.read_fields()["e"])     # fields too large for the context's own buffer
    e = torch.full((ne,), float("nan"), dtype=torch.float64, pin_memory=True).numpy()
    x = np.zeros((n, 2))
    fail.append(True)                                      # no staging for the particles
    s.step(600, "vay")                                     # some 10 ms of work ahead of the copy
    rc = fetdpic.lib().fetdpic_read(s.h, 0, e.ctypes.data_as(C.c_void_p), None, None, 0, x.ctypes.data_as(C.c_void_p), None, None)
    got = e.copy()
    assert rc == fetdpic.ENOMEM
    fail.clear()
    assert np.array_equal(got, s.read_fields()["e"])
    s.close()
