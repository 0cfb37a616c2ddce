"""GPU: launch forms that run the same kernels give the same bits.

An unprofiled handle overlaps or merges launches that a profiled one takes apart.
Where both run the same operations -- every 16-bit lattice, and FP64 and FP32 ones
above 2^18 cells (the smaller FP32 ones with the bulk sweep beside the near one on
one stream) -- nothing may differ but the order of execution, so with
prescribed motion PDFs and forces are equal.  The rigid-body update is one launch
with the force total in one form and alone in the other: its few FP64 operations
may be contracted differently, 1e-14 of the state after one step.

The allocation-free sweep has three forms: one launch (up to 2^18 cells), bulk
beside near, and bulk after near (above 2^22 cells).  It is called back to back on
two swapped buffers, where a block that read a stale cache line or ran ahead of
its input would show, and as a captured graph.
"""
import numpy as np
import pytest

from paper_1702_04910_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def scene(shape, bc_z, coupling, n, fixed, subcycles):
    case = {"shape": shape, "bc_z": bc_z, "coupling": coupling, "collision": "TRT", "tau": 0.8,
            "magic": 3.0 / 16.0, "fext": (1e-5, 0.0, -1e-5), "gravity": (0, 0, -1e-4), "rho0": 1.0,
            "subsample": 4, "subcycles": subcycles, "wall_contact": 0}
    if bc_z == 2:
        case |= {"inflow": (0.0, 0.0, 0.02), "rho_out": 1.0}
    mid = [0.5 * s for s in shape]
    case["particles"] = [
        {"x": (mid[0] + 0.3, mid[1] - 0.2, mid[2] + 0.1), "u": (0.03, -0.02, 0.05),
         "omega": (0.0, 1e-3, 0.0), "diameter": 9.0, "density": 1.5, "fixed": fixed},
        {"x": (mid[0] - 11.1, mid[1] - 0.4, mid[2]), "u": (0.0, 0.01, 0.0),
         "omega": (1e-3, 0.0, 0.0), "diameter": 7.0, "density": 2.0, "fixed": fixed},
        {"x": (0.5, 0.2, mid[2]), "u": (0.0, 0.0, 0.02), "omega": (0.0, 0.0, 1e-3),
         "diameter": 8.5, "density": 1.2, "fixed": fixed}][:n]
    return case


@pytest.mark.parametrize("shape,bc_z,coupling,storage,n", [
    ((67, 63, 64), 2, "MEM_CLI", "f16s", 1), ((66, 64, 64), 0, "PSM_M1B1", "bf16s", 2),
    ((31, 27, 29), 1, "MEM_MR", "f16s", 1), ((72, 64, 70), 0, "MEM_CLI", "f32", 3),
    ((71, 65, 70), 1, "PSM_M2B2", "f32", 2), ((72, 64, 70), 0, "MEM_BB", "f64", 3),
    ((73, 66, 70), 2, "PSM_M1B1", "f64fx", 1)])
def test_same_bits(lattice, shape, bc_z, coupling, storage, n):
    from paper_1702_04910_gb300.binding import Simulation, lbm_profile_enable
    _, w, _ = lattice
    for fixed, steps in ((1, 9), (0, 1)):
        case = scene(shape, bc_z, coupling, n, fixed, 2)
        out = []
        for profiled in (False, True):
            s = Simulation(shape, storage=storage, **W.sim_kwargs(case))
            s.set_particles(case["particles"])
            s.set_pdf_pre(W.perturbed_field(w, shape, 0.03, seed=5))
            if profiled:
                lbm_profile_enable(s.h, True)
            s.step(steps)
            F, T = s.forces()
            P = s.get_particles()
            out.append((s.pdf(), np.asarray(F), np.asarray(T),
                        np.asarray([p[k] for p in P for k in ("x", "u", "omega")])))
            s.close()
        (fa, Fa, Ta, Pa), (fb, Fb, Tb, Pb) = out
        assert np.all(np.isfinite(Fa)) and np.any(Fa != 0.0)
        assert np.array_equal(Fa, Fb) and np.array_equal(Ta, Tb)
        if fixed:
            assert np.array_equal(fa.view(np.uint8), fb.view(np.uint8))
        assert np.max(np.abs(Pa - Pb)) <= 1e-14 * np.max(np.abs(Pb))


@pytest.mark.parametrize("shape,n,coupling", [
    ((72, 70, 66), 3, "MEM_CLI"), ((72, 70, 66), 3, "PSM_M2B2"), ((71, 69, 67), 1, "MEM_MR"),
    ((168, 161, 160), 2, "MEM_BB"), ((168, 161, 160), 2, "PSM_M1B1")])
def test_noalloc_chain_matches_handle(lattice, shape, n, coupling):
    import torch

    from paper_1702_04910_gb300 import binding as B
    _, w, _ = lattice
    stream = torch.cuda.current_stream().cuda_stream
    case = scene(shape, 0, coupling, n, 1, 1)
    kw = W.sim_kwargs(case)
    sim = B.Simulation(shape, stream=stream, **kw)
    sim.set_particles(case["particles"])
    sim.set_pdf_pre(W.perturbed_field(w, shape, 0.02, seed=11))
    sim.step(1)
    state = sim.pdf()
    steps = 8
    sim.step(steps)
    ref, (F, T) = sim.pdf(), sim.forces()
    fluid = (sim.flags() == 0) if coupling.startswith("MEM") else np.ones(shape[::-1], bool)
    sim.close()

    cfg = B.make_config(shape, **kw)
    buf = [torch.from_numpy(state).cuda(), torch.from_numpy(state).cuda()]
    ft = torch.zeros((n, 6), dtype=torch.float64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def chain(st):
        for i in range(steps):
            B.lbm_sweep_noalloc(cfg, buf[i % 2].data_ptr(), buf[1 - i % 2].data_ptr(),
                                case["particles"], ft.data_ptr(), status_ptr=st,
                                stream=torch.cuda.current_stream().cuda_stream)

    def check():
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got = buf[0].cpu().numpy()  # an even number of sweeps
        assert np.max(np.abs(got[:, fluid] - ref[:, fluid])) <= 1e-12 * np.max(np.abs(ref))
        out = ft.cpu().numpy()
        for a, b in ((out[:, :3], F), (out[:, 3:], T)):
            scale = max(np.max(np.abs(b)), np.max(np.abs(F)))
            assert np.max(np.abs(a - b)) <= 1e-10 * scale

    chain(status.data_ptr())
    check()
    eager = buf[0].clone(), ft.clone()

    # captured: with the caller's status word, and with none (a memset leads the graph)
    for st in (status.data_ptr(), 0):
        start = torch.from_numpy(state).cuda()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain(st)
        for _ in range(3):
            buf[0].copy_(start)
            ft.zero_()
            graph.replay()
            check()
            assert torch.equal(buf[0][:, torch.from_numpy(fluid).cuda()],
                               eager[0][:, torch.from_numpy(fluid).cuda()])
            assert torch.equal(ft, eager[1])
        del graph


@pytest.mark.parametrize("coupling", ["MEM_CLI", "PSM_M1B1"])
def test_noalloc_one_launch_captured(lattice, coupling):
    test_noalloc_chain_matches_handle(lattice, (40, 38, 36), 1, coupling)
