"""GPU: the fixed-point form of the FP64 fluid collision against the oracle.

Populations on both sides of the form's range (down to below 2^-6 and beyond
the upper ends, negative ones among them, in units of the power of two nearest
to rho0), so that neighbouring cells take the fixed-point and the FP64 form;
reference densities far from 1, with and without a body force.

Bar: the oracle's own rounding.  A collided value is a sum of fewer than 100
rounded FP64 operations on terms of at most 4 max|f|, so it lies within
100 * 4 * 2^-54 max|f| = 2.3e-14 max|f| of the exact one; the fixed point adds
about 2 units of 2^-58, far below.
"""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_1702_04910_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f64", "f64fx"])
@pytest.mark.parametrize("rho0,fext,collision", [
    (1.0, (0.0, 0.0, 0.0), "TRT"), (1.0, (3e-4, -1e-6, 2e-9), "BGK"),
    (1.37, (1e-5, 2e-5, -3e-5), "TRT"), (640.0, (0.0, 0.0, 0.0), "BGK"),
    (1.1 * 2.0 ** -9, (1e-9, 0.0, 4e-8), "TRT")])
def test_fixed_point_collision_against_the_oracle(lattice, rho0, fext, collision, storage):
    from paper_1702_04910_gb300.binding import Simulation
    _, w, _ = lattice
    case = {"shape": (45, 13, 9), "coupling": "NONE", "collision": collision, "tau": 0.57,
            "magic": 3.0 / 16.0, "fext": fext, "gravity": (0, 0, 0), "rho0": rho0, "bc_z": 1,
            "subsample": 4, "subcycles": 1, "wall_contact": 0}
    o = Oracle(case["shape"], **W.sim_kwargs(case))
    g = Simulation(case["shape"], storage=storage, **W.sim_kwargs(case))
    f0 = W.perturbed_field(w, o.shape, 0.6, seed=5) * rho0
    rng = np.random.default_rng(6)
    hit = rng.uniform(size=f0.shape)
    f0[hit < 0.004] *= 4.0          # beyond the upper ends
    f0[hit > 0.998] *= -0.2         # negative populations
    o.set_pdf(f0)
    g.set_pdf_pre(f0)
    for _ in range(2):  # a collision alone, then pull and collision
        o.step(1)
        g.step(1)
        ref, got = o.pdf("post"), g.pdf()
        assert np.max(np.abs(got - ref)) <= 2.3e-14 * np.max(np.abs(ref))

