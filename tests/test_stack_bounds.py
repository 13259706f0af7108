"""Host-side bounds and addressing of the window kernel on stacked images, without a GPU: tests/stack_bounds.cpp is
compiled with the host C++ compiler, linked against the built library (which exports the planner)
and run."""
import os
import shutil
import subprocess

import pytest

from paper_1908_11263_gb300 import build as qbuild

HERE = os.path.dirname(os.path.abspath(__file__))


def test_stacked_images(tmp_path):
    lib = qbuild.build()
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(qbuild.nvcc())))
    exe = str(tmp_path / "stack_bounds")
    subprocess.run([cxx, "-std=c++17", "-O1", f"-I{os.path.join(cuda, 'include')}",
                    os.path.join(HERE, "stack_bounds.cpp"), "-o", exe, lib, f"-Wl,-rpath,{os.path.dirname(lib)}",
                    f"-L{os.path.join(cuda, 'lib64')}", "-lcudart"], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.rstrip().endswith("fails=0"), out.stdout[-4000:]
