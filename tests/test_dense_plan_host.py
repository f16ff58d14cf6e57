"""Dense models whose fused sweeps would be slower than one launch per mode
(modes of more than 1,024 states that few blocks walk through) get no plan;
the others keep theirs. Host check of the planner, no GPU."""
import importlib.util
import os
import subprocess

import pytest

from conftest import ROOT

PKG = os.path.join(ROOT, "paper_2103_00331_gb300")


def test_dense_plan(tmp_path):
    spec = importlib.util.spec_from_file_location("_cpmdp_build", os.path.join(PKG, "build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "dense_plan")
    p = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-cudart", "none",
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"),
                        os.path.join(ROOT, "tests", "dense_plan_host.cu"),
                        os.path.join(ROOT, "tests", "fake_cudart.cpp"), "-o", exe], capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    p = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, p.stdout + p.stderr
