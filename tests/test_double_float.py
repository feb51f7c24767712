"""Double-float push of the FP32 path above gamma = 10: on the host, against extended precision."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1707_04333_gb300 import build_lib
    exe = str(tmp_path_factory.mktemp("df") / "double_float_host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", build_lib.INCLUDE, "-I", build_lib.SRC,
                    os.path.join(ROOT, "tests", "double_float_host.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("ulps", [1, 2])
def test_errors_no_larger_than_in_fp64_with_newton_roots(program, ulps):
    """u, 1/gamma and v before the rounding to FP32, over gamma 10 to 3e8 and kicks and |beta| up to
    gamma / 8: rms and largest error of the double-float push against those of the push in FP64 whose
    roots take one Newton step from the same seeds (the device's are within 2 ulp)."""
    out = subprocess.run([program, "100000", str(ulps)], capture_output=True, text=True, check=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 4 * 4 * 3
    for pusher, rng, what, *v in rows:
        rms64, rms, max64, top = map(float, v)
        assert rms <= rms64 and top <= max64, (pusher, rng, what, v)
