"""Triangles are stored along a space-filling curve whatever the ratio of the mesh's scales."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_consecutive_triangles_are_neighbours(tmp_path):
    from paper_1707_04333_gb300 import build_lib
    exe = str(tmp_path / "triangle_order_host")
    cuda = os.path.join(build_lib._cuda_home(build_lib._nvcc()), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", build_lib.INCLUDE, "-I", build_lib.SRC, "-I", cuda,
                    os.path.join(ROOT, "tests", "triangle_order_host.cpp"), os.path.join(build_lib.SRC, "mesh_setup.cpp"),
                    "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
