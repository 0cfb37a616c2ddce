"""The per-cell device code, compiled for the host and run on the CPU.

tests/host/device_shim.h gives the CUDA intrinsics as host functions; a plain
C++ compiler then builds the device headers themselves, so these tests run the
library's own arithmetic, not a restatement of it.
"""
import ctypes as ct
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


def build(tmp_path_factory, name):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    lib = str(tmp_path_factory.mktemp("host") / f"{name}.so")
    cmd = ["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-fPIC", "-shared", "-I", CUDA_INC,
           "-I", os.path.join(ROOT, "include"),
           "-I", os.path.join(ROOT, "paper_1702_04910_gb300", "csrc"),
           os.path.join(ROOT, "tests", "host", f"{name}.cpp"), "-o", lib]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ct.CDLL(lib)


@pytest.fixture(scope="module")
def predicates(tmp_path_factory):
    return build(tmp_path_factory, "predicates")


@pytest.mark.parametrize("n", [32, 256, 768, 4096, 1 << 20, (1 << 24) + 2])
@pytest.mark.parametrize("D", [1.0, 8.0, 24.0, 24.37])
def test_filtered_predicates_decide_as_fp64(predicates, n, D):
    """Spheres across the periodic faces of short and long boxes: the FP32
    filter must leave every point that it cannot tell to the FP64 form, so no
    decision and no sample count differs."""
    out = (ct.c_longlong * 2)()
    predicates.filter_mismatches(n, ct.c_double(D), 100000 if n < 1000 else 40000, 7, out)
    assert list(out) == [0, 0]
