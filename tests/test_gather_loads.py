"""The gather kernel's loads, outputs and chunks, without a GPU: tests/gather_loads.cpp is compiled with the host C++
compiler, linked against the built library (which exports the planner) and run."""
import os
import shutil
import subprocess

import pytest

from paper_1908_11263_gb300 import build as qbuild

HERE = os.path.dirname(os.path.abspath(__file__))


def test_loads_outputs_and_chunks(tmp_path):
    lib = qbuild.build()
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(qbuild.nvcc())))
    exe = str(tmp_path / "gather_loads")
    subprocess.run([cxx, "-std=c++17", "-O1", f"-I{os.path.join(cuda, 'include')}",
                    os.path.join(HERE, "gather_loads.cpp"), "-o", exe, lib, f"-Wl,-rpath,{os.path.dirname(lib)}",
                    f"-L{os.path.join(cuda, 'lib64')}", "-lcudart"], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.rstrip().endswith("fails=0"), out.stdout[-4000:]
    # whole words, single bytes, chunks and more chunks than accumulators all occur
    assert "words 1 bytes 1 chunks 1 many 1" in out.stdout
    for word in ("flat", "im2col", "aligned", "bytes", "resident", "streamed"):
        assert f" {word} " in out.stdout or f" {word}\n" in out.stdout, word
