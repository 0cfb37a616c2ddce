"""GPU: LBM_STORE_F64_DP collides every cell in FP64 arithmetic.

Where no cell is in the range of the fixed point (three times the rest density, so
every rest population lies above its upper end) LBM_STORE_F64 takes the same FP64
form in the same kernels: equal bits.  In the range the two differ by their
roundings, and both lie within the oracle's own (2.3e-14 of the largest
population, see test_gpu_fixed.py).
"""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_1702_04910_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def fluid(shape, collision, fext):
    return {"shape": shape, "coupling": "NONE", "collision": collision, "tau": 0.57,
            "magic": 3.0 / 16.0, "fext": fext, "gravity": (0, 0, 0), "rho0": 1.0, "bc_z": 1,
            "subsample": 4, "subcycles": 1, "wall_contact": 0}


@pytest.mark.parametrize("collision,fext", [("TRT", (0.0, 0.0, 0.0)), ("BGK", (3e-4, -1e-6, 2e-9))])
def test_against_f64_and_the_oracle(lattice, collision, fext):
    from paper_1702_04910_gb300.binding import Simulation
    _, w, _ = lattice
    case = fluid((45, 13, 9), collision, fext)
    for density in (3.0, 1.0):
        f0 = W.perturbed_field(w, case["shape"], 0.05, seed=5) * density
        o = Oracle(case["shape"], **W.sim_kwargs(case))
        o.set_pdf(f0)
        sims = {m: Simulation(case["shape"], storage=m, **W.sim_kwargs(case)) for m in ("f64", "f64dp")}
        for s in sims.values():
            s.set_pdf_pre(f0)
        for _ in range(2):
            o.step(1)
            for s in sims.values():
                s.step(1)
            ref, a, b = o.pdf("post"), sims["f64"].pdf(), sims["f64dp"].pdf()
            bar = 2.3e-14 * np.max(np.abs(ref))
            assert np.max(np.abs(b - ref)) <= bar and np.max(np.abs(a - ref)) <= bar
            assert np.array_equal(a, b) == (density == 3.0)


def test_every_entry_point():
    """Handle, batch and allocation-free sweep in FP64 arithmetic agree to FP64
    rounding over three sweeps with a moving sphere, and none of them takes the
    fixed point: LBM_STORE_F64 gives other last bits."""
    import torch

    from paper_1702_04910_gb300 import binding as B
    case = W.settling_sphere(D=8.0, shape=(24, 24, 40), ga=10.0, nu=0.03, drop_below_top=16.0,
                             coupling="MEM_CLI", seed=5)
    case["subcycles"] = 1
    case["particles"][0] |= {"fixed": 1, "u": (0.0, 0.0, -0.03)}
    kw = W.sim_kwargs(case)
    out = {}
    for mode in ("f64", "f64dp"):
        s = B.Simulation(case["shape"], storage=mode, **kw)
        s.set_particles(case["particles"])
        s.init_equilibrium()
        start = s.pdf()
        s.step(3)
        out["handle", mode] = s.pdf()
        fluid = s.flags() == 0
        s.close()

        b = B.Batch([case], storage=mode)
        b.step(3)
        b.synchronize()
        out["batch", mode] = b.pdf(0)
        b.close()

        buf = [torch.from_numpy(start).cuda(), torch.from_numpy(start).cuda()]
        ft = torch.zeros(6, dtype=torch.float64, device="cuda")
        cfg = B.make_config(case["shape"], storage=mode, **kw)
        for i in range(3):
            B.lbm_sweep_noalloc(cfg, buf[i % 2].data_ptr(), buf[1 - i % 2].data_ptr(),
                                case["particles"], ft.data_ptr())
        torch.cuda.synchronize()
        out["noalloc", mode] = buf[1].cpu().numpy()
    ref = out["handle", "f64dp"][:, fluid]
    for how in ("handle", "batch", "noalloc"):
        dp, fx = out[how, "f64dp"][:, fluid], out[how, "f64"][:, fluid]
        assert np.max(np.abs(dp - ref)) <= 1e-13 and np.max(np.abs(dp - fx)) <= 1e-13
        assert np.mean(dp != fx) > 0.01
