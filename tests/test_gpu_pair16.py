"""GPU: the 16-bit sweeps with two cells per thread against the FP64 oracle.

x-pairs at row lengths that take blocks of 32, 64 and 96 threads, whole and
partly filled; z-pairs for odd rows, an odd number of planes (the last plane
alone), walls and open boundaries, next to a sphere.  Bar: storage rounds the
shifted populations, |g| < 1.2e-2 here, by at most 2^-12 |g| (FP16) or 2^-9 |g|
(BF16) per sweep, 3e-6 or 2.4e-5; 8 sweeps of a collision that amplifies no
mode stay below 8 times that, relative to max f = 1/3: 7.2e-5 and 5.8e-4.
"""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_1702_04910_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,tol", [("f16s", 7.2e-5), ("bf16s", 5.8e-4)])
@pytest.mark.parametrize("shape,bc_z,coupling", [
    ((30, 14, 18), 0, "PSM_M2B2"), ((66, 14, 16), 1, "MEM_CLI"), ((130, 13, 15), 0, "NONE"),
    ((192, 14, 15), 1, "PSM_M1B1"), ((31, 17, 19), 0, "MEM_BB"), ((129, 14, 17), 1, "PSM_M2B2"),
    ((33, 15, 22), 2, "MEM_CLI"), ((34, 16, 21), 2, "PSM_M1B1")])
def test_two_cells_per_thread(lattice, shape, bc_z, coupling, storage, tol):
    from paper_1702_04910_gb300.binding import Simulation
    _, w, _ = lattice
    case = {"shape": shape, "bc_z": bc_z, "coupling": coupling, "collision": "TRT", "tau": 0.8,
            "magic": 3.0 / 16.0, "fext": (1e-5, 0.0, -1e-5), "gravity": (0, 0, 0), "rho0": 1.0,
            "subsample": 4, "subcycles": 1, "wall_contact": 0}
    if bc_z == 2:
        case |= {"inflow": (0.0, 0.0, 0.02), "rho_out": 1.0}
    kw = W.sim_kwargs(case)
    o = Oracle(shape, **kw)
    g = Simulation(shape, storage=storage, **kw)
    if coupling != "NONE":
        part = [{"x": tuple(0.5 * n + 0.3 for n in shape), "u": (0.01, -0.01, 0.01),
                 "omega": (0.0, 1e-3, 0.0), "diameter": 6.0, "density": 1.5, "fixed": 1}]
        o.set_particles(part)
        g.set_particles(part)
    f0 = W.perturbed_field(w, o.shape, 0.03, seed=3)
    o.set_pdf(f0)
    g.set_pdf_pre(f0)
    o.step(8)
    g.step(8)
    if coupling.startswith("MEM"):
        ref, mask = o.pdf("collide"), o.solid() == 0
    else:
        ref, mask = o.pdf("post"), np.ones(o.shape[::-1], dtype=bool)
    err = np.max(np.abs(g.pdf_f64()[:, mask] - ref[:, mask])) / np.max(np.abs(ref[:, mask]))
    assert err <= tol, err
