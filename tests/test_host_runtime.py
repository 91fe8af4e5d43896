"""The host runtime on a fake CUDA runtime (no GPU): what it hands to the
kernels and what state it leaves after a failure; see host_runtime_check.cpp."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    out = str(tmp_path_factory.mktemp("host") / "host_runtime_check")
    subprocess.check_call([cxx, "-O1", "-std=c++17", "-pthread", "-ffp-contract=off", "-I", include,
                           "-I", os.path.join(ROOT, "paper_1902_08410_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "host_runtime_check.cpp"), "-o", out])
    return out


@pytest.mark.parametrize("check", ["phase", "failure", "large", "footprint", "tables", "pairs"])
def test_host_runtime(exe, check):
    r = subprocess.run([exe, check], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip() == "ok"
