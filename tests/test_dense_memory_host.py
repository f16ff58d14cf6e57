"""Device memory of dense models, against a fake allocator on the host: the
build takes the factors alone, a sweep the intermediates of its precision
within their bound (also under a stream capture), and a refused allocation
drops the plan instead of the call."""
import importlib.util
import os
import subprocess

import pytest

from conftest import ROOT

PKG = os.path.join(ROOT, "paper_2103_00331_gb300")


def test_dense_memory(tmp_path):
    spec = importlib.util.spec_from_file_location("_cpmdp_build", os.path.join(PKG, "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "dense_memory")
    p = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-cudart", "none",
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"),
                        os.path.join(ROOT, "tests", "dense_memory_host.cu"),
                        os.path.join(ROOT, "tests", "fake_cudart.cpp"), "-o", exe], capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    p = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout + p.stderr
