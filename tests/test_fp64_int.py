"""Integer IEEE arithmetic of the FP64 particle kernel: on the host, bit for bit against the processor."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fp64int") / "fp64_int_host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1707_04333_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fp64_int_host.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("ulps", [0, 1, 2, 6])
def test_integer_arithmetic_gives_the_processors_bits(program, ulps):
    """The device's approximate reciprocal and root seeds are within 1 and 2 units of the last place."""
    out = subprocess.run([program, "4000000", str(ulps)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
