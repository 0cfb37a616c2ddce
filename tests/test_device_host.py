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


# ---- the fixed-point collision of FP64 populations against exact arithmetic -----------
@pytest.fixture(scope="module")
def collision(tmp_path_factory):
    lib = build(tmp_path_factory, "collision")
    lib.constant_product_error.restype = ct.c_double
    lib.variable_product_error.restype = ct.c_double
    return lib


def lambda_minus(tau, kind):
    return -1.0 / tau if kind == "BGK" else 1.0 / ((3.0 / 16.0) / (0.5 - tau) - 0.5)


@pytest.mark.parametrize("tau", [0.5001, 0.53, 0.6, 0.8, 1.0, 1.5, 2.0])
@pytest.mark.parametrize("kind", ["BGK", "TRT"])
def test_fixed_point_products(collision, tau, kind):
    """By a constant: half a unit of rounding and a low x low limb product below one
    unit, taken at its mean: one unit.  Of two variables: half a unit and signed low
    limbs, 2^62 / 2^64: three quarters."""
    lp, lm = -1.0 / tau, lambda_minus(tau, kind)
    for c in (-lp / 12, -lp / 36, -lp / 72, -lm / 6, -lm / 12):
        assert collision.constant_product_error(ct.c_double(c), 100000, 3) <= 1.0
    assert collision.variable_product_error(100000, 3) <= 0.75


@pytest.mark.parametrize("tau", [0.5001, 0.53, 0.8, 1.0, 2.0])
@pytest.mark.parametrize("kind", ["BGK", "TRT"])
def test_fixed_point_error_over_a_flow(collision, tau, kind):
    """Root mean square error over the cells of a flow: below the FP64 form's, and
    refused cells come back bit for bit."""
    out = (ct.c_double * 7)()
    for rho0, fext in ((1.0, (0.0, 0.0, 0.0)), (1.0, (3e-4, -1e-6, 2e-9)),
                       (1.37, (1e-5, 2e-5, -3e-5)), (0.75, (0.0, 0.0, 0.0))):
        for noise, drift in ((0.0, 0.1), (0.02, 0.05), (0.1, 0.1), (0.3, 0.1), (1e-4, 1e-3)):
            collision.collision_errors(ct.c_double(tau), ct.c_double(lambda_minus(tau, kind)),
                                       ct.c_double(rho0), (ct.c_double * 3)(*fext),
                                       ct.c_double(noise), ct.c_double(drift), 10000, 11, out)
            cells, fixed, fp64 = out[0], out[1], out[2]
            assert cells >= 100 and fixed < fp64, (rho0, fext, noise, drift, list(out))


def test_which_modes_collide_in_fixed_point(collision):
    from paper_1702_04910_gb300.binding import STORAGE
    for tau in (0.5001, 0.8, 2.0, 2.01, 100.0):
        t = ct.c_double(tau)
        assert collision.fixed_point_on(STORAGE["f64"], t) == (tau <= 2.0)
        assert collision.fixed_point_on(STORAGE["f64fx"], t) == 1
        assert collision.fixed_point_on(STORAGE["f64dp"], t) == 0
