"""Contexts of different block sizes and precisions stepped by several host threads at once: the state
each reaches alone."""
import threading

import numpy as np
import pytest

from paper_1707_04333_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_no_launch_state_is_shared_between_threads():
    """Occupancy and SM counts are kept per thread: no function-local static of the launch code is
    shared (read from the source), and contexts on eight threads step as they do alone."""
    import os
    import re
    from paper_1707_04333_gb300 import build_lib, fetdpic
    for name in build_lib.CU_SOURCES:
        text = open(os.path.join(build_lib.SRC, name)).read()
        assert not re.search(r"^\s+static\s+(?!thread_local|const|__device__|inline|_)\w+\s+\w+\s*=", text, re.M), name
    w = inputs.pair_plasma(12, 6, kT=0.2, wc_over_wp=0.5, seed=5)
    kinds = [("fp64", 32), ("fp64", 256), ("fp32", 32), ("fp64", 64)] * 2

    def run(kind, out):
        s = fetdpic.Simulation(w, precision=kind[0], block_size=kind[1], use_torch=False, sort_interval=3).load()
        for k in range(25):
            s.step(1 + k % 3, "vay")
        s.sync()
        p, f = s.read_species(0), s.read_fields()
        out.append([p["x"], p["u"], p["cell"], f["e"], f["b"]])
        s.close()
    alone, together = [], [[] for _ in kinds]
    for k in kinds[:4]:
        run(k, alone)
    threads = [threading.Thread(target=run, args=(k, o)) for k, o in zip(kinds, together)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, o in enumerate(together):
        assert all(np.array_equal(a, b) for a, b in zip(alone[i % 4], o[0])), kinds[i]
