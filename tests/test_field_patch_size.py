"""Triangles of a patch: whole waves of blocks up to one measured patch size, at every mesh size."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_patch_sizes(tmp_path):
    from paper_1707_04333_gb300 import build_lib
    exe = str(tmp_path / "field_patch_size_host")
    cuda = os.path.join(build_lib._cuda_home(build_lib._nvcc()), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", build_lib.INCLUDE, "-I", build_lib.SRC, "-I", cuda,
                    os.path.join(ROOT, "tests", "field_patch_size_host.cpp"),
                    os.path.join(build_lib.SRC, "field_patches.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nx", [404, 440, 445])               # 716 and 850 triangles a patch, and 434 in two waves
def test_largest_patches_equal_the_whole_mesh_update(precision, nx):
    from paper_1707_04333_gb300 import fetdpic, inputs
    m = inputs.jittered_delaunay(nx, nx, 1.0, 1.0, 0.2, seed=3)
    rng = np.random.default_rng(1)
    tri = np.sort(rng.integers(0, len(m.triangles), 5000)).astype(np.int32)
    x, u = inputs.sample_in_triangles(m, tri, rng), rng.normal(0, 0.3 * inputs.C_LIGHT, (len(tri), 2))
    sp = inputs.Species(-1e-12, 1e-12 * inputs.M_E / inputs.Q_E, x, u, tri)
    w = inputs.Workload("large", m, [sp], 0.02 / nx / inputs.C_LIGHT, b0=0.01)
    out = []
    for whole in (False, True):
        s = fetdpic.Simulation(w, precision=precision, fuse_field_update=whole).load()
        s.step(5, "boris").sync()
        f, p = s.read_fields(), s.read_species(0)
        out.append([f["e"], f["b"], f["j"], p["x"], p["u"], p["cell"]])
        s.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out)) and np.abs(out[0][0]).max() > 0
