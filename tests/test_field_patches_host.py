"""Patch tables of the field update: checked on the host against the mesh, and allocation failures in
their threads reported instead of ending the process."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_patch_tables(tmp_path):
    from paper_1707_04333_gb300 import build_lib
    exe = str(tmp_path / "field_patches_host")
    cuda = os.path.join(build_lib._cuda_home(build_lib._nvcc()), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-ffp-contract=off", "-I", build_lib.INCLUDE, "-I", build_lib.SRC,
                    "-I", cuda, os.path.join(ROOT, "tests", "field_patches_host.cpp"),
                    os.path.join(build_lib.SRC, "field_patches.cpp"), os.path.join(build_lib.SRC, "mesh_setup.cpp"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, (out.returncode, out.stdout, out.stderr)
