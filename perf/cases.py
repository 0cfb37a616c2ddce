"""The work that users of this library have it do, as cases that can be timed and checked.

Five kinds of program, all through the public entry points of ``binding``:

* ``window``    one simulation handle advanced by some steps, with its forces read as the program
                reads them and the stored PDFs written to a device buffer at the end of the window:
                drag studies in a periodic box, settling spheres, the open benchmark frame;
* ``coarse``    a coarse sphere placed on a prescribed trajectory before every step, its force and
                its feature stencil read after it (data generation of the learned correction);
* ``ensemble``  a batch of uneven settling cases stepped together, every step's particle states and
                forces read;
* ``sweep``     the allocation-free sweep on buffers of the caller, several spheres;
* ``gradient``  loss and parameter gradient of the force-correction network on a training set.

Numbers read from a handle (forces, particle states) are given in the units rho0 u_ref^2 D^2, D
and u_ref and at the width of the PDFs that they come from.  ``exact`` restates the method in 64
bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_1702_04910_gb300.binding import (FIELD_PDF, MLP_IN, MLP_OUT, MLP_PARAMS, Batch, Mlp,
                                             Simulation, lbm_get_fields, lbm_set_fields,
                                             lbm_sweep_noalloc, make_config)

NQ = 19
C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
              (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])
WQ = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
OPP = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, NQ)]
TORCH = {"f64": torch.float64, "f64fx": torch.float64, "f32": torch.float32,
         "f16s": torch.float16, "bf16s": torch.bfloat16}
NUMPY = {"f64": np.float64, "f64fx": np.float64, "f32": np.float32, "f16s": np.float16,
         "bf16s": np.float16}
COUPLINGS = ("PSM_M1B1", "PSM_M2B2", "PSM_M3B2", "MEM_BB", "MEM_CLI", "MEM_MR")


def listed():
    return [
        # smallest calls: the parity and smoke size of a released sphere, momentum exchange with
        # re-mapping; a step is a chain of short kernels
        settle("settle-tiny", 24, 24, 40, 8.0, ga=10.0, nu=0.03, coupling="MEM_CLI", storage="f64",
               calls=20, per_call=1),
        # the drag study of the paper's Fig. 1: fixed sphere, body force, forces read per chunk
        box("drag-box", 32, 8.0, coupling="PSM_M1B1", storage="f64", calls=2, per_call=25),
        # the settling benchmark, FP64 parity run, two sweeps per step and re-mapping
        settle("settle-f64", 128, 128, 512, 24.0, coupling="MEM_MR", storage="f64", per_call=4),
        # the same sphere in single precision, with the re-mapping charge
        settle("settle-f32", 128, 128, 512, 24.0, coupling="MEM_CLI", storage="f32", per_call=8,
               charge=True),
        # the fast mode of long settling runs
        settle("settle-f16", 128, 128, 512, 24.0, coupling="PSM_M1B1", storage="f16s", per_call=20),
        # the large sphere (D = 36) in the other 16-bit format
        settle("settle-bf16-large", 192, 192, 768, 36.0, coupling="MEM_BB",
               storage="bf16s", per_call=6, charge=True),
        # calibration loop of the paper's benchmark frame (inflow and outflow): one step, read the
        # drag, next step
        frame("frame-f64fx", 18.0, coupling="MEM_CLI", storage="f64fx", calls=10),
        # the frame at an odd lattice width in 16 bits
        frame("frame-f16-odd", 19.0, coupling="MEM_CLI", storage="f16s", calls=10),
        # data generation of the learned correction at D = 12
        {"name": "coarse-features", "kind": "coarse", "coupling": "PSM_M2B2", "storage": "f32",
         "nx": 64, "ny": 64, "nz": 192, "d": 12.0, "ga": 140.0, "nu": 0.05 * 12.0 / 140.0,
         "steps": 10},
        # ensemble of uneven settling cases (D = 8..16), all couplings, FP64, with the charge
        {"name": "ensemble", "kind": "ensemble", "storage": "f64", "n": 12, "d_lo": 8, "d_hi": 16,
         "sizes": 0, "steps": 3},
        # one sweep on the caller's own buffers, four spheres
        {"name": "sweep-spheres", "kind": "sweep", "coupling": "MEM_BB", "nx": 96, "ny": 96,
         "nz": 96, "n": 4, "d": 16.0, "tau": 0.8},
        # full-batch gradient of the force-correction network on the five-number training set
        {"name": "mlp-gradient", "kind": "gradient", "n": 7200},
    ]


def settle(name, nx, ny, nz, d, coupling, storage, ga=144.0, nu=0.01, calls=1, per_call=1,
           charge=False):
    return {"name": name, "kind": "window", "flow": "settle", "coupling": coupling,
            "storage": storage, "nx": nx, "ny": ny, "nz": nz, "d": d, "ga": ga, "nu": nu,
            "calls": calls, "per_call": per_call, "charge": charge}


def box(name, n, d, coupling, storage, calls, per_call, tau=0.8):
    return {"name": name, "kind": "window", "flow": "box", "coupling": coupling,
            "storage": storage, "nx": n, "ny": n, "nz": n, "d": d, "tau": tau, "calls": calls,
            "per_call": per_call, "charge": False}


def frame(name, d, coupling, storage, calls):
    n = int(round(5.34 * d))
    return {"name": name, "kind": "window", "flow": "frame", "coupling": coupling,
            "storage": storage, "nx": n, "ny": n, "nz": int(round(16.0 * d)), "d": d,
            "calls": calls, "per_call": 1, "charge": False}


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(("settle", "settle", "settle", "box", "frame", "coarse", "ensemble", "sweep",
                       "gradient"))
    storage = rng.choice(("f64", "f64fx", "f32", "f16s", "bf16s"))
    if kind == "settle":
        # the settling box, 5.33 D x 5.33 D x 21.3 D in any whole numbers of cells
        d = round(log(8.0, 32.0), 1)
        nx, ny = (max(int(d) + 7, int(round(d * rng.uniform(4.0, 6.0)))) for _ in range(2))
        nz = int(round(d * rng.uniform(12.0, 22.0)))
        c = settle("", nx, ny, nz, d, rng.choice(("PSM_M1B1", "PSM_M2B2", "MEM_CLI", "MEM_MR")),
                   storage, ga=d * rng.uniform(3.0, 4.5), per_call=rng.randint(2, 5))
        c["charge"] = c["coupling"].startswith("MEM")
    elif kind == "box":
        n = int(round(log(24, 96)))
        c = box("", n, float(rng.randint(6, n // 2)), rng.choice(COUPLINGS), storage,
                rng.randint(1, 3), rng.randint(5, 25), tau=rng.choice((0.6, 0.8, 1.0, 1.5)))
        if c["coupling"] == "PSM_M3B2" and storage in ("f16s", "bf16s"):
            c["storage"] = "f32"
    elif kind == "frame":
        c = frame("", float(rng.randint(18, 23)), rng.choice(("PSM_M1B1", "PSM_M2B2", "MEM_BB",
                                                              "MEM_CLI", "MEM_MR")), storage,
                  rng.randint(3, 10))
    elif kind == "coarse":
        d = float(rng.randint(6, 16))
        c = {"name": "", "kind": "coarse", "coupling": rng.choice(("PSM_M2B2", "MEM_CLI")),
             "storage": rng.choice(("f64", "f32")), "nx": int(round(16.0 * d / 3.0)),
             "ny": int(round(16.0 * d / 3.0)), "nz": int(round(16.0 * d)), "d": d, "ga": 140.0,
             "nu": 0.05 * d / 140.0, "steps": rng.randint(3, 10)}
    elif kind == "ensemble":
        lo = rng.randint(6, 12)
        c = {"name": "", "kind": "ensemble", "storage": rng.choice(("f64", "f64fx")),
             "n": rng.randint(3, 12), "d_lo": lo, "d_hi": lo + rng.randint(1, 4),
             "sizes": rng.randint(1, 1000), "steps": rng.randint(2, 4)}
    elif kind == "sweep":
        n = rng.choice((1, 2, 4, 8))
        d = float(rng.randint(6, 16))
        side = [int(round(2.6 * d * (2 if n > k else 1) + rng.randint(0, 20))) for k in (1, 2, 4)]
        c = {"name": "", "kind": "sweep", "coupling": rng.choice(("PSM_M1B1", "PSM_M2B2", "MEM_BB",
                                                                  "MEM_CLI", "MEM_MR")),
             "nx": side[0], "ny": side[1], "nz": side[2], "n": n, "d": d,
             "tau": rng.choice((0.53, 0.6, 0.8))}
    else:
        c = {"name": "", "kind": "gradient", "n": int(round(log(100, 8000)))}
    del c["name"]
    return c


# ---- inputs -------------------------------------------------------------------------------------
def scene(case, seed):
    """Solver configuration and particles of a ``window`` or ``coarse`` case."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, d = case["nx"], case["ny"], case["nz"], case["d"]
    s = {"shape": (nx, ny, nz), "coupling": case["coupling"], "collision": "TRT", "magic": 3 / 16,
         "fext": (0.0, 0.0, 0.0), "gravity": (0.0, 0.0, 0.0), "rho0": 1.0, "bc_z": 0,
         "subsample": 4, "subcycles": 2 if case["coupling"].startswith("MEM") else 1,
         "wall_contact": 0, "inflow": (0.0, 0.0, 0.0), "rho_out": 1.0}
    off = rng.uniform(-0.25, 0.25, 3)
    p = {"x": tuple(np.array([nx / 2, ny / 2, nz / 2]) + off), "u": (0.0, 0.0, 0.0),
         "omega": (0.0, 0.0, 0.0), "diameter": d, "density": 1.5, "fixed": 1}
    if case.get("flow") == "box":
        s |= {"tau": case["tau"], "fext": (4.4e-6, 0.0, 0.0), "u_ref": 0.02, "mean": (0.01, 0, 0), "noise": 1.0}
        if case["coupling"] == "PSM_M3B2":
            s["subcycles"] = 2
    elif case.get("flow") == "frame":
        u_in = 1.285 * 144.0 * 0.01 / d
        s |= {"tau": 0.53, "bc_z": 2, "subcycles": 2, "inflow": (0.0, 0.0, u_in),
              "u_ref": u_in / 1.285, "mean": (0.0, 0.0, u_in), "noise": 0.1}
        if case["coupling"].startswith("PSM") and case["storage"].startswith("f64"):
            s["collision"] = "BGK"  # as printed; TRT keeps the reduced precisions stable
        p["x"] = (2.67 * d + off[0], 2.67 * d + off[1], 5.34 * d + off[2])
    else:  # settling: heavy sphere, closed bottom and top, already falling
        u_ref = case["ga"] * case["nu"] / d
        g = u_ref ** 2 / (0.5 * d)
        s |= {"tau": 3 * case["nu"] + 0.5, "bc_z": 1, "gravity": (0.0, 0.0, -g),
              "wall_contact": 1, "u_ref": u_ref, "mean": (0.0, 0.0, 0.0), "noise": 1.0}
        p |= {"x": (nx / 2 + off[0], ny / 2 + off[1], nz - 1.2 * d - 3 + off[2]),
              "u": (0.1 * u_ref * off[0], 0.1 * u_ref * off[1], -u_ref * rng.uniform(0.3, 0.6)),
              "omega": tuple(0.02 * u_ref * off), "fixed": 0}
    s["particles"] = [p]
    return s


def solver(s):
    return {k: v for k, v in s.items() if k not in ("shape", "particles", "u_ref", "mean", "noise")}


def waves(seed, n):
    """n smooth periodic fields' wave numbers, amplitudes and phases."""
    rng = np.random.default_rng([seed, 7])
    return [(rng.integers(0, 4, 3), rng.uniform(0.3, 1.0), rng.uniform(0, 2 * math.pi))
            for _ in range(n)]


def flow_pdf(s, storage, seed):
    """Stored PDFs of a smooth seeded flow about the mean velocity, in the storage's layout."""
    nx, ny, nz = s["shape"]
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) * (2 * math.pi / n)
          for n in (nx, ny, nz)]
    out = []
    for comp, wave in enumerate(zip(*[iter(waves(seed, 12))] * 3)):
        v = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.float64)
        for k, a, ph in wave:
            v += a * torch.sin(k[0] * ax[0][None, None, :] + k[1] * ax[1][None, :, None] +
                               k[2] * ax[2][:, None, None] + ph)
        out.append(v * ((0.1 * s["u_ref"] if comp else 0.001) * s["noise"]))
    rho, u = 1.0 + out[0], [out[1 + a] + s["mean"][a] for a in range(3)]
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    f = torch.empty((NQ, nz, ny, nx), device="cuda", dtype=TORCH[storage])
    for q in range(NQ):
        cu = sum(float(C[q][a]) * u[a] for a in range(3))
        e = WQ[q] * (rho + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
        f[q] = e - WQ[q] if storage in ("f16s", "bf16s") else e
    return f


def trajectory(case, s, k):
    """Prescribed state of a ``coarse`` case's sphere before step k: to and fro along z."""
    amp, om = 0.25 * s["shape"][2], 0.05 / (0.25 * s["shape"][2])
    p = dict(s["particles"][0])
    t = k * s["subcycles"]
    p["x"] = (p["x"][0], p["x"][1], 0.5 * s["shape"][2] + amp * math.cos(om * t))
    p["u"] = (0.002, -0.001, -amp * om * math.sin(om * t))
    p["omega"] = (0.0, 5e-4, 0.0)
    p["fixed"] = 1
    return p


def ensemble_scenes(case, seed):
    """Settling cases of uneven size (the sizes are the case's, the rest comes from the seed)."""
    sizes, rng = np.random.default_rng(case["sizes"]), np.random.default_rng(seed)
    out = []
    for c in range(case["n"]):
        d = float(sizes.integers(case["d_lo"], case["d_hi"] + 1))
        n_lat, n_z = int(round(5.3 * d)), int(round(16.0 * d))
        one = {"nx": n_lat, "ny": n_lat, "nz": n_z, "d": d, "ga": d * float(rng.uniform(3.0, 4.5)),
               "nu": 0.01,
               "coupling": ("PSM_M1B1", "PSM_M2B2", "MEM_BB", "MEM_CLI", "MEM_MR")[c % 5]}
        out.append(scene(one, int(rng.integers(1 << 30))))
    return out


def spheres(case, seed):
    """Configuration and moving spheres of a ``sweep`` case on a loose grid."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    cells = [2 if n > k else 1 for k in (1, 2, 4)]
    shape = (case["nx"], case["ny"], case["nz"])
    s = {"shape": shape, "coupling": case["coupling"], "collision": "TRT", "magic": 3 / 16,
         "fext": (1e-5, 0.0, 0.0), "gravity": (0.0, 0.0, 0.0), "rho0": 1.0, "bc_z": 0,
         "subsample": 4, "subcycles": 1, "wall_contact": 0, "inflow": (0.0, 0.0, 0.0),
         "rho_out": 1.0, "tau": case["tau"], "u_ref": 0.05, "mean": (0.0, 0.0, 0.0), "noise": 1.0}
    s["particles"] = []
    for i in range(n):
        at = (i % cells[0], i // cells[0] % cells[1], i // (cells[0] * cells[1]))
        x = [(at[a] + 0.5) * shape[a] / cells[a] + rng.uniform(-0.5, 0.5) for a in range(3)]
        s["particles"].append({"x": tuple(x), "u": tuple(rng.uniform(-0.03, 0.03, 3)),
                               "omega": tuple(rng.uniform(-1e-3, 1e-3, 3)),
                               "diameter": case["d"], "density": 1.5, "fixed": 0})
    return s


def network(n, seed):
    """Training set, parameters and normalisation as the training program has them."""
    rng = np.random.default_rng(seed)
    x = rng.normal(0.0, 1.0, (n, MLP_IN))
    x[:, :125] = rng.uniform(0.0, 1.0, (n, 125))  # solid indicators
    t = rng.normal(0.0, 1.0, (n, MLP_OUT)) * np.array([0.02, 0.02, 0.3, 0.01, 0.01, 0.01])
    p = []
    for a, b in ((MLP_IN, 64), (64, 64), (64, MLP_OUT)):
        r = math.sqrt(6.0 / (a + b))
        p += [rng.uniform(-r, r, a * b), rng.uniform(-0.01, 0.01, b)]
    p = np.concatenate(p).astype(np.float32)
    assert p.size == MLP_PARAMS
    x, t = x.astype(np.float32), t.astype(np.float32)
    sd = x.std(axis=0)
    norm = np.concatenate([x.mean(axis=0), 1.0 / sd, np.sqrt((t.astype(np.float64) ** 2).mean(axis=0))])
    return x, t, p, norm.astype(np.float32)


# ---- the measured program -----------------------------------------------------------------------
def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    kind = case["kind"]
    if kind in ("window", "coarse"):
        s = scene(case, seed)
        pdf = flow_pdf(s, case["storage"], seed)
        sim = Simulation(s["shape"], stream=stream, storage=case["storage"], **solver(s))
        sim.set_particles([trajectory(case, s, 0)] if kind == "coarse" else s["particles"])
        lbm_set_fields(sim.h, FIELD_PDF, pdf.data_ptr(), pdf.numel() * pdf.element_size(), True)
        if case.get("charge"):
            sim.set_remap_charge(True)
        if kind == "coarse":
            sim.set_force_model(None, s["u_ref"], mode=2)
        return {"case": case, "scene": s, "sim": sim, "pdf": pdf, "k": 0}
    if kind == "ensemble":
        batch = Batch(ensemble_scenes(case, seed), storage=case["storage"], stream=stream)
        batch.set_remap_charge(True)
        return {"case": case, "batch": batch}
    if kind == "sweep":
        s = spheres(case, seed)
        src = flow_pdf(s, "f64", seed)
        return {"case": case, "scene": s, "src": src, "dst": src.clone(), "stream": stream,
                "cfg": make_config(s["shape"], **solver(s)),
                "ft": torch.zeros((case["n"], 6), device="cuda", dtype=torch.float64),
                "status": torch.zeros(1, device="cuda", dtype=torch.int32)}
    x, t, p, norm = network(case["n"], seed)
    m = Mlp(stream)
    m.set_params(p)
    m.set_normalization(norm)
    return {"case": case, "mlp": m, "x": torch.from_numpy(x).cuda(), "t": torch.from_numpy(t).cuda()}


def units(s, storage, forces, torques, parts):
    """Read-outs in the units of the run, at the width of its PDFs."""
    u, d, ty = s["u_ref"], s["particles"][0]["diameter"], NUMPY[storage]
    return {"force": (np.asarray(forces) / (u * u * d * d)).astype(ty),
            "torque": (np.asarray(torques) / (u * u * d ** 3)).astype(ty),
            "x": np.asarray([p["x"] / d for p in parts]).astype(ty),
            "u": np.asarray([p["u"] / u for p in parts]).astype(ty),
            "omega": np.asarray([p["omega"] * (0.5 * d / u) for p in parts]).astype(ty)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "window":
        sim, pdf = state["sim"], state["pdf"]
        F, T = [], []
        for _ in range(case["calls"]):
            sim.step(case["per_call"])
            f, t = sim.forces()
            F.append(f)
            T.append(t)
        out = units(state["scene"], case["storage"], F, T, sim.get_particles())
        lbm_get_fields(sim.h, FIELD_PDF, pdf.data_ptr(), pdf.numel() * pdf.element_size(), True)
        out["pdf"] = pdf
        return out
    if kind == "coarse":
        sim, pdf, s = state["sim"], state["pdf"], state["scene"]
        F, T, feat = [], [], []
        for _ in range(case["steps"]):
            sim.set_particles([trajectory(case, s, state["k"])])
            sim.step(1)
            f, t = sim.forces()
            F.append(f)
            T.append(t)
            feat.append(sim.features())
            state["k"] += 1
        out = units(s, case["storage"], F, T, sim.get_particles())
        lbm_get_fields(sim.h, FIELD_PDF, pdf.data_ptr(), pdf.numel() * pdf.element_size(), True)
        out |= {"pdf": pdf, "features": np.asarray(feat)}
        return out
    if kind == "ensemble":
        b = state["batch"]
        rec = {"force": [], "torque": [], "x": [], "u": [], "omega": []}
        for _ in range(case["steps"]):
            b.step(1)
            F, T = b.forces()
            P = b.particles()
            rec["force"].append(F)
            rec["torque"].append(T)
            for k in ("x", "u", "omega"):
                rec[k].append([p[k] for p in P])
        return {k: np.asarray(v) for k, v in rec.items()}
    if kind == "sweep":
        s = state["scene"]
        lbm_sweep_noalloc(state["cfg"], state["src"].data_ptr(), state["dst"].data_ptr(),
                          s["particles"], state["ft"].data_ptr(), state["status"].data_ptr(),
                          state["stream"])
        return {"pdf": state["dst"], "force_torque": state["ft"], "status": state["status"]}
    g, loss = state["mlp"].gradient(state["x"].data_ptr(), state["t"].data_ptr(), case["n"])
    return {"gradient": g, "loss": loss}


def work(case):
    """Bytes and operations of one pass: per sweep every PDF read once and written once, the
    written-out PDFs read and written, the training set read; 250 operations per cell update."""
    kind = case["kind"]
    if kind == "gradient":
        layer = MLP_IN * 64 + 64 * 64 + 64 * MLP_OUT
        return {"bytes": 4.0 * (case["n"] * (MLP_IN + MLP_OUT) + 2 * MLP_PARAMS),
                "flops": case["n"] * 2.0 * (2 * layer + 64 * 64 + 64 * MLP_OUT)}
    if kind == "ensemble":
        cells = sum(int(np.prod(s["shape"])) * s["subcycles"] for s in ensemble_scenes(case, 0))
        return {"bytes": 304.0 * cells * case["steps"], "flops": 250.0 * cells * case["steps"]}
    cells = float(case["nx"]) * case["ny"] * case["nz"]
    if kind == "sweep":
        return {"bytes": 304.0 * cells, "flops": 250.0 * cells}
    steps = case["steps"] if kind == "coarse" else case["calls"] * case["per_call"]
    sweeps = steps * scene(case, 0)["subcycles"]
    size = 8 if case["storage"].startswith("f64") else 4 if case["storage"] == "f32" else 2
    return {"bytes": 38.0 * size * cells * (sweeps + 1), "flops": 250.0 * cells * sweeps}


# ---- the same results in 64 bits ----------------------------------------------------------------
class Exact:
    """The coupled step of one scene with plain torch in 64 bits.  ``f`` holds the post-collision
    PDFs of the last sweep, ``other`` the buffer the next sweep writes (the library leaves the
    cells inside MEM spheres as they are in the buffer)."""

    def __init__(self, s, pdf):
        self.s, self.shape = s, s["shape"]
        self.f = pdf
        self.dev = pdf.device
        self.parts = [{k: (np.array(v, dtype=np.float64) if k in ("x", "u", "omega") else v)
                       for k, v in p.items()} for p in s["particles"]]
        self.mem = s["coupling"].startswith("MEM")
        self.lp = -1.0 / s["tau"]
        self.lm = self.lp
        if s["collision"] == "TRT":
            self.lm = 1.0 / (s["magic"] / (0.5 - s["tau"]) - 0.5)
        w = torch.tensor(WQ, device=self.dev, dtype=torch.float64)
        self.other = (s["rho0"] * w)[:, None, None, None].expand_as(pdf).clone()
        self.c = torch.tensor(C, device=self.dev, dtype=torch.float64)
        self.charge = None
        self.owner = self.owners() if self.mem else None

    # geometry: minimum-image offsets from a particle, in the exact order of operations that the
    # solid tests are defined by (squares added x, y, z)
    def offset(self, x, a, p):
        d = x - p["x"][a]
        if a == 2 and self.s["bc_z"]:
            return d
        n = float(self.shape[a])
        return torch.where(d > 0.5 * n, d - n, torch.where(d < -0.5 * n, d + n, d))

    def axes(self, shift=0.5):
        return [torch.arange(n, device=self.dev, dtype=torch.float64) + shift for n in self.shape]

    def owners(self):
        ax = self.axes()
        own = torch.zeros(self.shape[::-1], device=self.dev, dtype=torch.int32)
        for k, p in reversed(list(enumerate(self.parts))):
            d = [self.offset(ax[a], a, p) ** 2 for a in range(3)]
            r2 = (d[0][None, None, :] + d[1][None, :, None]) + d[2][:, None, None]
            own[r2 <= (0.5 * p["diameter"]) ** 2] = k + 1
        return own

    def fractions(self):
        """Solid fraction of every particle in every cell from 4^3 samples."""
        out, n = [], 4
        for p in self.parts:
            r2, cnt = (0.5 * p["diameter"]) ** 2, 0
            d = [[self.offset(self.axes((i + 0.5) / n)[a], a, p) ** 2 for i in range(n)]
                 for a in range(3)]
            box = [torch.nonzero(torch.stack(d[a]).amin(0) <= r2 + 4 * p["diameter"] + 4).flatten()
                   for a in range(3)]
            for i in range(n):
                for j in range(n):
                    xy = d[0][i][box[0]][None, :] + d[1][j][box[1]][:, None]
                    for k in range(n):
                        cnt = cnt + (xy[None] + d[2][k][box[2]][:, None, None] <= r2).double()
            e = torch.zeros(self.shape[::-1], device=self.dev, dtype=torch.float64)
            e[box[2][:, None, None], box[1][None, :, None], box[0][None, None, :]] = cnt / n ** 3
            out.append(e)
        return out

    def arm(self, xyz, p):
        return torch.stack([self.offset(xyz[a], a, p) for a in range(3)])

    def body(self, xyz, p):
        r, w = self.arm(xyz, p), p["omega"]
        return torch.stack([p["u"][0] + (w[1] * r[2] - w[2] * r[1]),
                            p["u"][1] + (w[2] * r[0] - w[0] * r[2]),
                            p["u"][2] + (w[0] * r[1] - w[1] * r[0])])

    def wrap(self, i, a):
        return i if a == 2 and self.s["bc_z"] else i % self.shape[a]

    # fluid
    def equilibrium(self, q, rho, u, uu):
        cu = sum(float(C[q][a]) * u[a] for a in range(3) if C[q][a])
        return WQ[q] * (rho + self.s["rho0"] * (3 * cu + 4.5 * cu * cu - 1.5 * uu))

    def moments(self, f):
        rho = f.sum(0)
        j = [sum(float(C[q][a]) * f[q] for q in range(NQ) if C[q][a]) for a in range(3)]
        return rho, [v / self.s["rho0"] for v in j]

    def forcing(self, q, u):
        fe = self.s["fext"]
        cu = sum(float(C[q][a]) * u[a] for a in range(3))
        return WQ[q] * sum((3 * (float(C[q][a]) - u[a]) + 9 * cu * float(C[q][a])) * fe[a]
                           for a in range(3))

    def collide(self, f):
        """Post-collision values of f, [19, ...]."""
        rho, u = self.moments(f)
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        force = any(self.s["fext"])
        out = torch.empty_like(f)
        for q in range(NQ):
            b = OPP[q]
            eq, eb = self.equilibrium(q, rho, u, uu), self.equilibrium(b, rho, u, uu)
            out[q] = f[q] + self.lp * 0.5 * (f[q] + f[b] - eq - eb) + \
                self.lm * 0.5 * (f[q] - f[b] - eq + eb)
            if force:
                out[q] += self.forcing(q, u)
        return out

    def pull(self):
        s, f = self.s, self.f
        g = torch.empty_like(f)
        for q in range(NQ):
            g[q] = torch.roll(f[q], tuple(int(v) for v in C[q][::-1]), (0, 1, 2))
        if s["bc_z"]:
            for q in range(NQ):
                if C[q][2] > 0:
                    g[q, 0] = f[OPP[q], 0]
                    if s["bc_z"] == 2:
                        g[q, 0] += 6 * WQ[q] * s["rho0"] * float(C[q] @ np.array(s["inflow"]))
                elif C[q][2] < 0:
                    g[q, -1] = f[OPP[q], -1]
            if s["bc_z"] == 2:
                j = [sum(float(C[q][a]) * f[q, -1] for q in range(NQ)) for a in range(3)]
                u = [j[a] / s["rho0"] - s["fext"][a] / (2 * s["rho0"]) for a in range(3)]
                uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
                for q in range(NQ):
                    if C[q][2] < 0:
                        cu = sum(float(C[q][a]) * u[a] for a in range(3))
                        g[q, -1] = 2 * WQ[q] * (s["rho_out"] + s["rho0"] *
                                                (4.5 * cu * cu - 1.5 * uu)) - g[q, -1]
        return g

    # momentum exchange: every link between a fluid cell and a solid one
    def links(self, g, ft):
        s, f, own = self.s, self.f, self.owner
        variant = s["coupling"][4:]
        lam = -1.0 / self.lm - 0.5
        new = []
        for q in range(1, NQ):
            b = OPP[q]  # from the fluid cell to the solid one
            up = torch.roll(own, tuple(int(v) for v in C[q][::-1]), (0, 1, 2))
            if s["bc_z"] and C[q][2]:
                up[0 if C[q][2] > 0 else -1] = 0
            at = torch.nonzero((up > 0) & (own == 0))
            if not len(at):
                continue
            z, y, x = at.T
            i = (x, y, z)
            who = up[z, y, x]

            def node(k, i=i, q=q):
                """Cell k steps along c_q: indexes and whether it is a fluid cell."""
                j = [i[a] + k * int(C[q][a]) for a in range(3)]
                ok = torch.ones_like(x, dtype=torch.bool)
                if s["bc_z"]:
                    ok = (j[2] >= 0) & (j[2] < self.shape[2])
                    j[2] = j[2].clamp(0, self.shape[2] - 1)
                j = [self.wrap(j[a], a) for a in range(3)][::-1]
                return tuple(j), ok & (own[tuple(j)] == 0)

            xc = torch.stack([v.double() + 0.5 for v in i])
            cb = [float(v) for v in C[b]]
            delta = torch.full_like(xc[0], 0.5)
            vel, centre = torch.zeros_like(xc), []
            for k, p in enumerate(self.parts):
                mine = who == k + 1
                if variant != "BB":
                    r = self.arm(xc, p)
                    a2 = float((C[b] ** 2).sum())
                    bb = sum(cb[a] * r[a] for a in range(3))
                    cc = (r[0] ** 2 + r[1] ** 2 + r[2] ** 2) - (0.5 * p["diameter"]) ** 2
                    t = (-bb - (bb * bb - a2 * cc).clamp(min=0).sqrt()) / a2
                    delta = torch.where(mine, t.clamp(0, 1), delta)
            xb = torch.stack([xc[a] + delta * cb[a] for a in range(3)])
            for k, p in enumerate(self.parts):
                vel = torch.where(who == k + 1, self.body(xb, p), vel)
                centre.append(self.arm(xb, p))
            vc = sum(vel[a] * cb[a] for a in range(3))
            here = f[b][z, y, x]
            wall = 3 * WQ[q] * s["rho0"] * vc
            val = here - 2 * wall
            if variant != "BB":
                n2, ok2 = node(1)
                k0 = (1 - 2 * delta) / (1 + 2 * delta)
                cli = here + k0 * f[b][n2] - k0 * f[q][z, y, x] - 4 / (1 + 2 * delta) * wall
                val = torch.where(ok2, cli, val)
            if variant == "MR":
                n3, ok3 = node(2)
                cell = f[:, z, y, x]
                j = self.c.T @ cell
                d1 = (1 + delta) ** 2
                odd = 0.5 * (here - f[q][z, y, x]) - 3 * WQ[q] * sum(cb[a] * j[a] for a in range(3))
                mr = here + (1 - 2 * delta - 2 * delta ** 2) / d1 * (f[b][n2] - f[q][z, y, x]) + \
                    delta ** 2 / d1 * (f[b][n3] - f[q][n2]) - 4 / d1 * wall - \
                    4 * lam / (lam - 0.5) / d1 * odd
                val = torch.where(ok2 & ok3, mr, val)
            new.append((q, z, y, x, val))
            F = torch.stack([(cb[a] - vel[a]) * here - (-cb[a] - vel[a]) * val for a in range(3)])
            for k in range(len(self.parts)):
                mine = (who == k + 1).double()
                ft[k, :3] += (F * mine).sum(1)
                ft[k, 3:] += (torch.linalg.cross(centre[k], F, dim=0) * mine).sum(1)
        for q, z, y, x, val in new:
            g[q, z, y, x] = val

    # partially saturated cells
    def saturated(self, g, out, ft):
        s = self.s
        eps = self.fractions()
        at = torch.nonzero(sum(eps) > 0)
        z, y, x = at.T
        f = g[:, z, y, x]
        xc = torch.stack([v.double() + 0.5 for v in (x, y, z)])
        rho, u = self.moments(f)
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        fluid = self.collide(f) - f
        B, solid = 0.0, torch.zeros_like(f)
        feq = torch.stack([self.equilibrium(q, rho, u, uu) for q in range(NQ)])
        for k, p in enumerate(self.parts):
            e = eps[k][z, y, x]
            h = s["tau"] - 0.5
            Bs = e if s["coupling"] == "PSM_M1B1" else e * h / ((1 - e) + h)
            B = B + Bs
            v = self.body(xc, p)
            vv = v[0] ** 2 + v[1] ** 2 + v[2] ** 2
            fev = torch.stack([self.equilibrium(q, rho, v, vv) for q in range(NQ)])
            if s["coupling"] == "PSM_M1B1":
                cs = (f - feq)[OPP] - (f - fev)
            elif s["coupling"] == "PSM_M2B2":
                cs = (fev - f) + (1 - 1 / s["tau"]) * (f - feq)
            else:
                cs = (f - fev)[OPP] - (f - fev)
            solid += Bs * cs
            F = Bs * (self.c[OPP].T @ cs)
            ft[k, :3] += F.sum(1)
            ft[k, 3:] += torch.linalg.cross(self.arm(xc, p), F, dim=0).sum(1)
        out[:, z, y, x] = f + (1 - B) * fluid + solid

    def sweep(self):
        ft = torch.zeros((len(self.parts), 6), device=self.dev, dtype=torch.float64)
        g = self.pull()
        if self.mem:
            self.links(g, ft)
            out = torch.where(self.owner[None] > 0, self.other, self.collide(g))
        else:
            out = self.collide(g)
            self.saturated(g, out, ft)
        self.f, self.other, self.pre = out, self.f, g
        return ft

    def step(self):
        n = self.s["subcycles"]
        ft = sum(self.sweep() for _ in range(n)) / n
        if self.charge is not None:
            ft = ft - torch.tensor(self.charge, device=self.dev) / n
        self.ft = ft.cpu().numpy()
        for k, p in enumerate(self.parts):
            self.move(p, self.ft[k], float(n))
        if self.mem:
            self.remap(True)

    def move(self, p, ft, dt):
        if p["fixed"]:
            return
        d, s = p["diameter"], self.s
        vol = math.pi * d ** 3 / 6
        m = p["density"] * vol
        total = ft[:3] + (p["density"] - s["rho0"]) * vol * np.array(s["gravity"])
        p["x"] = p["x"] + dt * p["u"]
        p["u"] = p["u"] + dt * total / m
        p["omega"] = p["omega"] + dt * ft[3:] / (m * d * d / 10)
        for a in range(3):
            if not (a == 2 and s["bc_z"]):
                p["x"][a] %= self.shape[a]
        if s["wall_contact"]:
            r, top = 0.5 * d, self.shape[2] - 1.0
            if p["x"][2] - r < 1:
                p["x"][2], p["u"][2] = r + 1, max(p["u"][2], 0.0)
            if p["x"][2] + r > top:
                p["x"][2], p["u"][2] = top - r, min(p["u"][2], 0.0)

    def place(self, parts):
        """Particles replaced by the program between steps."""
        for p, new in zip(self.parts, parts):
            for k in ("x", "u", "omega"):
                p[k] = np.array(new[k], dtype=np.float64)
        if self.mem:
            self.remap(False)

    def remap(self, extrapolate):
        """Rebuilds the cells that the spheres have left (extrapolated along the normal, with the
        body's momentum; equilibrium after a replacement) and counts the exchanged momentum."""
        old, new, s = self.owner, self.owners(), self.s
        self.owner = new
        keep = [np.zeros(6) for _ in self.parts]
        count = extrapolate and self.charge is not None
        if count:
            at = torch.nonzero((old == 0) & (new > 0)).cpu().numpy()
            for z, y, x in at:
                k = int(new[z, y, x]) - 1
                self.account(keep[k], k, x, y, z, self.pre[:, z, y, x].cpu().numpy(), -1.0)
        at = torch.nonzero((old > 0) & (new == 0)).cpu().numpy()
        for z, y, x in at:
            k = int(old[z, y, x]) - 1
            p = self.parts[k]
            xc = torch.tensor([x + 0.5, y + 0.5, z + 0.5], dtype=torch.float64)
            v = self.body(xc[:, None], p)[:, 0].numpy()
            nrm = self.arm(xc[:, None], p)[:, 0].numpy()
            nodes = []
            if extrapolate:
                qn = 1 + int(np.argmax(C[1:] @ (nrm / max(np.linalg.norm(nrm), 1e-300))))
                for i in (1, 2, 3):
                    j = self.usable(old, new, x, y, z, i * C[qn])
                    if j is None:
                        break
                    nodes.append(self.pre[(slice(None),) + j].cpu().numpy())
            if nodes:
                wt = {1: (1,), 2: (2, -1), 3: (3, -3, 1)}[len(nodes)]
                f = sum(a * b for a, b in zip(wt, nodes))
                f = f + C @ (s["rho0"] * v - C.T @ f) / 10
            else:
                rho = s["rho0"]
                if extrapolate:
                    near = [self.usable(old, new, x, y, z, C[q]) for q in range(1, NQ)]
                    near = [float(self.pre[(slice(None),) + j].sum()) for j in near if j]
                    rho = sum(near) / len(near) if near else rho
                f = np.array([self.equilibrium(q, rho, v, v @ v) for q in range(NQ)])
            if count:
                self.account(keep[k], k, x, y, z, f, 1.0)
            t = torch.tensor(f, device=self.dev)[:, None]
            self.f[:, z, y, x] = self.collide(t)[:, 0]
        if count:
            self.charge = np.array(keep)
        elif self.charge is not None:
            self.charge = np.zeros((len(self.parts), 6))

    def usable(self, old, new, x, y, z, step):
        i = [int(x + step[0]) % self.shape[0], int(y + step[1]) % self.shape[1], int(z + step[2])]
        if not s_in(i[2], self.shape[2], self.s["bc_z"]):
            return None
        i[2] %= self.shape[2]
        j = (i[2], i[1], i[0])
        return None if int(old[j]) or int(new[j]) else j

    def account(self, keep, k, x, y, z, f, sign):
        xc = torch.tensor([x + 0.5, y + 0.5, z + 0.5], dtype=torch.float64)
        r = self.arm(xc[:, None], self.parts[k])[:, 0].numpy()
        j = C.T @ f
        keep[:3] += sign * j
        keep[3:] += sign * np.cross(r, j)

    def features(self, u_ref):
        """The 5 x 5 x 5 stencil of solid indicator and relative velocity, and the body's state."""
        p, s = self.parts[0], self.s
        h = 0.5 * (0.5 * p["diameter"] + 2.0)
        grid = (np.arange(5) - 2) * h
        pos = np.stack(np.meshgrid(grid, grid, grid, indexing="ij"), -1)
        pos = pos.transpose(2, 1, 0, 3).reshape(-1, 3) + p["x"] - 0.5
        base = np.floor(pos)
        fr = pos - base
        eps, vel = np.zeros(125), np.zeros((125, 3))
        solid = None if self.mem else sum(self.fractions()).clamp(max=1.0)
        for corner in range(8):
            d = np.array([corner & 1, corner >> 1 & 1, corner >> 2 & 1])
            w = np.prod(np.where(d, fr, 1 - fr), axis=1)
            i = (base + d).astype(np.int64)
            inside = np.array([s_in(int(k), self.shape[2], s["bc_z"]) for k in i[:, 2]])
            i = np.stack([i[:, a] % self.shape[a] for a in range(3)], 1)
            x, y, z = (torch.tensor(i[:, a], device=self.dev) for a in range(3))
            u = (self.c.T @ self.f[:, z, y, x]).T / s["rho0"]
            if self.mem:
                own = self.owner_used[z, y, x] > 0
                xc = torch.stack([v.double() + 0.5 for v in (x, y, z)])
                u = torch.where(own[:, None], self.body(xc, p).T, u)
                e = own.double()
            else:
                e = solid[z, y, x]
            w = w * inside
            eps += w * e.cpu().numpy()
            vel += w[:, None] * u.cpu().numpy()
        d = p["diameter"]
        fs = s["rho0"] * u_ref ** 2 * d ** 2
        return np.concatenate([eps, ((vel - p["u"]) / u_ref).T.reshape(-1), p["u"] / u_ref,
                               p["omega"] * (0.5 * d) / u_ref, self.ft[0, :3] / fs,
                               self.ft[0, 3:] / (fs * d)])


def s_in(z, n, closed):
    return not closed or 0 <= z < n


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        return exact_gradient(*network(case["n"], seed))
    if kind == "ensemble":
        rec = {"force": [], "torque": [], "x": [], "u": [], "omega": []}
        for s in ensemble_scenes(case, seed):
            nx, ny, nz = s["shape"]
            w = torch.tensor(WQ, device="cuda", dtype=torch.float64)
            e = Exact(s, (s["rho0"] * w)[:, None, None, None].expand(NQ, nz, ny, nx).clone())
            e.charge = np.zeros((1, 6))
            one = {k: [] for k in rec}
            for _ in range(case["steps"]):
                e.step()
                one["force"].append(e.ft[0, :3])
                one["torque"].append(e.ft[0, 3:])
                for k in ("x", "u", "omega"):
                    one[k].append(e.parts[0][k].copy())
            for k in rec:
                rec[k].append(one[k])
        return {k: np.asarray(v).transpose(1, 0, 2) for k, v in rec.items()}
    if kind == "sweep":
        s = spheres(case, seed)
        src = flow_pdf(s, "f64", seed)
        e = Exact(s, src)
        e.other = src.clone()
        ft = e.sweep()
        return {"pdf": e.f, "force_torque": ft, "status": None}
    s = scene(case, seed)
    if kind == "coarse":
        s["particles"] = [trajectory(case, s, 0)]
    shift = case["storage"] in ("f16s", "bf16s")
    w = torch.tensor(WQ, device="cuda", dtype=torch.float64)[:, None, None, None]
    pdf = flow_pdf(s, case["storage"], seed).double()
    e = Exact(s, pdf + w if shift else pdf)
    if case.get("charge"):
        e.charge = np.zeros((len(e.parts), 6))
    F, T, feat = [], [], []
    if kind == "coarse":
        for k in range(case["steps"]):
            e.place([trajectory(case, s, k)])
            e.owner_used = e.owner
            e.step()
            F.append(e.ft[:, :3])
            T.append(e.ft[:, 3:])
            feat.append([e.features(s["u_ref"])])
    else:
        for _ in range(case["calls"]):
            for _ in range(case["per_call"]):
                e.step()
            F.append(e.ft[:, :3])
            T.append(e.ft[:, 3:])
    u, d = s["u_ref"], s["particles"][0]["diameter"]
    out = {"force": np.asarray(F) / (u * u * d * d), "torque": np.asarray(T) / (u * u * d ** 3),
           "x": np.asarray([p["x"] / d for p in e.parts]),
           "u": np.asarray([p["u"] / u for p in e.parts]),
           "omega": np.asarray([p["omega"] * (0.5 * d / u) for p in e.parts]),
           "pdf": e.f - w if shift else e.f}
    if feat:
        out["features"] = np.asarray(feat)[:, 0]
    return out


def exact_gradient(x, t, p, norm):
    x, t, p, norm = (torch.from_numpy(a).cuda().double() for a in (x, t, p, norm))
    shapes, parts, at = ((MLP_IN, 64), (64,), (64, 64), (64,), (64, MLP_OUT), (MLP_OUT,)), [], 0
    for sh in shapes:
        k = int(np.prod(sh))
        parts.append(p[at:at + k].reshape(sh).clone().requires_grad_())
        at += k
    w1, b1, w2, b2, w3, b3 = parts
    scale = norm[2 * MLP_IN:]
    h = torch.tanh(torch.tanh((x - norm[:MLP_IN]) * norm[MLP_IN:2 * MLP_IN] @ w1 + b1) @ w2 + b2)
    e = h @ w3 + b3 - t / scale
    loss = 0.5 / x.shape[0] * ((scale / scale.max()) ** 2 * e * e).sum()
    g = torch.autograd.grad(loss, parts)
    return {"gradient": torch.cat([v.reshape(-1) for v in g]), "loss": float(loss)}
