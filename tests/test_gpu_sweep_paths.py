"""GPU: a sweep gives the same result however its cells are launched.

A profiled handle runs the near-particle sweep on a second stream beside the
bulk sweep, with an event between all kernels.  Without profiling the two are
one launch (small lattices) or share a stream and overlap.  The cells take the
same operations in both, and the force partials the same order: PDFs, forces and
particle states are equal.  Sizes: below a warp's 32 cells per row, odd, exactly
the largest one-launch lattice (2^18 cells) and above it; regions that overlap,
wrap around and touch a wall.
"""
import numpy as np
import pytest

from paper_1702_04910_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,bc_z,coupling,storage,n", [
    ((13, 14, 15), 0, "MEM_CLI", "f64", 1), ((17, 13, 19), 1, "PSM_M1B1", "f64", 1),
    ((31, 21, 33), 1, "MEM_MR", "f64", 3), ((30, 22, 25), 0, "PSM_M2B2", "f32", 3),
    ((64, 64, 64), 0, "MEM_BB", "f32", 2), ((64, 64, 65), 0, "MEM_CLI", "f64", 3),
    ((65, 64, 65), 1, "PSM_M2B2", "f32", 2), ((67, 63, 64), 2, "MEM_CLI", "f16s", 1),
    ((66, 64, 64), 0, "PSM_M1B1", "bf16s", 2), ((31, 17, 19), 1, "MEM_CLI", "f16s", 1)])
def test_same_result(lattice, shape, bc_z, coupling, storage, n):
    from paper_1702_04910_gb300.binding import Simulation, lbm_profile_enable
    _, w, _ = lattice
    case = {"shape": shape, "bc_z": bc_z, "coupling": coupling, "collision": "TRT", "tau": 0.8,
            "magic": 3.0 / 16.0, "fext": (1e-5, 0.0, -1e-5), "gravity": (0, 0, -1e-4), "rho0": 1.0,
            "subsample": 4, "subcycles": 2 if coupling.startswith("MEM") else 1,
            "wall_contact": int(bc_z == 1)}
    if bc_z == 2:
        case |= {"inflow": (0.0, 0.0, 0.02), "rho_out": 1.0}
    mid = [0.5 * s for s in shape]
    parts = [{"x": (mid[0] + 0.3, mid[1] - 0.2, mid[2] + 0.1), "u": (0.03, -0.02, 0.05),
              "omega": (0.0, 1e-3, 0.0), "diameter": 5.0, "density": 1.5, "fixed": 0},
             {"x": (mid[0] - 6.1, mid[1] - 0.4, mid[2]), "u": (0.0, 0.01, 0.0),
              "omega": (1e-3, 0.0, 0.0), "diameter": 4.0, "density": 2.0, "fixed": 0},
             {"x": (0.5, 0.2, 4.0), "u": (0.0, 0.0, 0.02), "omega": (0.0, 0.0, 1e-3),
              "diameter": 4.5, "density": 1.2, "fixed": 1}][:n]
    out = []
    for profiled in (False, True):
        s = Simulation(shape, storage=storage, **W.sim_kwargs(case))
        s.set_particles(parts)
        s.set_pdf_pre(W.perturbed_field(w, shape, 0.03, seed=5))
        if profiled:
            lbm_profile_enable(s.h, True)
        s.step(7)
        F, T = s.forces()
        P = s.get_particles()
        out.append([s.pdf_f64(), np.asarray(F), np.asarray(T)] +
                   [np.asarray([p[k] for p in P]) for k in ("x", "u", "omega")])
        s.close()
    tol = {"f64": 1.6e-13, "f32": 8.4e-5, "f16s": 14 * 2.0 ** -12, "bf16s": 14 * 2.0 ** -9}[storage]
    for k, (a, b) in enumerate(zip(*out)):
        assert np.all(np.isfinite(a))
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b)) * (100 if k else 1), k
