"""The work that users of the library have it do, as cases to be timed.

Every case goes through the public binding (`paper_1410_3219_gb300.rich`).
A simulation's pass is what a program's main loop does: advance it by a few
steps and read the result; the simulation goes on from pass to pass.  The
Courant time step over a caller's device arrays has cases of its own, since
it is the one entry point that works on device data.

Whole time steps have no closed form: a 64-bit reference would be a second
implementation of the tessellation and the scheme, so `exact` covers the
Courant time step only.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1410_3219_gb300 import rich
from paper_1410_3219_gb300 import workloads as W

# a step reads and writes each cell's points and conserved state and reads
# its connectivity (124 bytes), in about 1,100 floating-point operations
STEP_BYTES, STEP_FLOPS = 124, 1100
# the six fields (points and conserved state, or points and primitives) read
# back in FP64
READ_BYTES = 48

_DOUBLES = ctypes.POINTER(ctypes.c_double)


def listed():
    return [
        # The smallest call: the time step of a small simulation held in
        # device arrays, where launches and latency count.
        {"name": "dt_4097", "kind": "dt", "n": 4097, "moving": True},
        # The same over a mesh that fills the entry point's range (2^24
        # cells), an odd size, static mesh.
        {"name": "dt_12000007_static", "kind": "dt", "n": 12000007, "moving": False},
        # A small shock tube between walls, one step a pass: an interactive
        # run, bound by latency.
        {"name": "sod_4096", "kind": "step", "problem": "sod", "n": 4096, "steps": 1, "precision": "fp64",
         "scheme": "extrapolated", "motion": "moving"},
        # A periodic vortex of an odd size, ten steps a call: a test-sized
        # production run that reads its result now and then.
        {"name": "gresho_10201_x10", "kind": "step", "problem": "gresho", "n": 10201, "steps": 10,
         "precision": "fp64", "scheme": "extrapolated", "motion": "moving"},
        # Irregular points between walls, an odd count.
        {"name": "scattered_50625", "kind": "step", "problem": "scattered", "n": 50625, "steps": 2, "precision": "fp64",
         "scheme": "extrapolated", "motion": "moving"},
        # The paper's own time-centred scheme: two sweeps and two meshes per step.
        {"name": "sod_16384_time_centred", "kind": "step", "problem": "sod", "n": 16384, "steps": 2,
         "precision": "fp64", "scheme": "time_centred", "motion": "moving"},
        # A static (Eulerian) mesh.
        {"name": "wave_90000_static", "kind": "step", "problem": "wave", "n": 90000, "steps": 2,
         "precision": "fp64", "scheme": "extrapolated", "motion": "static"},
        # Split precision at an ordinary size; its primitives are FP32.
        {"name": "kh_262144_split", "kind": "step", "problem": "kh", "n": 262144, "steps": 1, "precision": "split",
         "scheme": "extrapolated", "motion": "moving"},
        # The benchmark's size, FP64.
        {"name": "kh_1048576", "kind": "step", "problem": "kh", "n": 1048576, "steps": 2, "precision": "fp64",
         "scheme": "extrapolated", "motion": "moving"},
        # Many small simulations of different sizes and problems stepped together.
        {"name": "batch_48", "kind": "batch", "sims": 48, "n_min": 1000, "n_max": 16000, "precision": "fp64"},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dt", "step", "step", "step", "step", "batch"])
    if kind == "dt":
        return {"kind": "dt", "n": _log_uniform(rng, 1000, 12000000) | 1, "moving": rng.random() < 0.7}
    if kind == "batch":
        lo = _log_uniform(rng, 300, 3000)
        return {"kind": "batch", "sims": rng.randint(8, 64), "n_min": lo, "n_max": lo * rng.randint(4, 12),
                "precision": "fp64"}
    problem = rng.choice(["sod", "gresho", "scattered", "kh", "wave"])
    scheme = "time_centred" if rng.random() < 0.25 else "extrapolated"
    n = _log_uniform(rng, 1000, 250000 if scheme == "time_centred" else 800000)
    side = max(32, int(round(math.sqrt(n))))
    return {"kind": "step", "problem": problem, "n": side * side,
            "steps": rng.randint(1, 4) if n < 200000 else rng.randint(1, 2), "precision": rng.choice(["fp64", "fp64", "split"]),
            "scheme": scheme, "motion": "static" if rng.random() < 0.15 else "moving"}


def _workload(problem, n, seed, precision, scheme="extrapolated", motion="moving"):
    mesh = W.MESH_EULERIAN if motion == "static" else W.MESH_LAGRANGIAN
    side = int(round(math.sqrt(n)))
    if problem == "sod":
        wl = W.sod(n_side=side, seed=seed, motion=mesh)
    elif problem == "gresho":
        wl = W.gresho(n_side=side, seed=seed, motion=mesh)
    elif problem == "kh":
        wl = W.kelvin_helmholtz(n_side=side, seed=seed, motion=mesh)
    elif problem == "wave":
        wl = W.sound_wave(n_side=side, seed=seed, motion=mesh)
    else:
        # (independent random points hold pairs so close that the scheme, which
        # has no floor, can stop with an emptied cell in its first steps)
        wl = W.sod(n_side=side, seed=seed, jitter=0.4, motion=mesh)
    wl["cfg"]["precision"] = W.FP32_SPLIT if precision == "split" else W.FP64
    wl["cfg"]["scheme"] = W.SCHEME_TIME_CENTRED if scheme == "time_centred" else W.SCHEME_EXTRAPOLATED
    return wl


def _dt_inputs(case, seed):
    """Device arrays of a smooth flow with noise on a mesh of n cells."""
    n = case["n"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def u(lo, hi):
        return torch.empty(n, dtype=torch.float64, device="cuda").uniform_(lo, hi, generator=g)

    a = {"area": u(0.6, 1.4) / n, "rho": u(0.5, 2.0), "vx": u(-1.0, 1.0), "vy": u(-1.0, 1.0), "p": u(0.5, 3.0)}
    if case["moving"]:
        # the mesh moves with the flow but for the rounding velocity
        a["wx"] = a["vx"] + u(-0.1, 0.1)
        a["wy"] = a["vy"] + u(-0.1, 0.1)
    return a


def _dt_cfg(case):
    return W.default_cfg(motion=W.MESH_LAGRANGIAN if case["moving"] else W.MESH_EULERIAN)


def _batch_members(case, seed):
    # sizes spread over the range, the same for every seed
    sizes = np.exp(np.linspace(math.log(case["n_min"]), math.log(case["n_max"]), case["sims"]))
    problems = ["sod", "gresho", "scattered"]
    return [_workload(problems[k % 3], max(200, int(round(nk))), seed * 64 + k, case["precision"])
            for k, nk in enumerate(sizes)]


def prepare(case, seed):
    if case["kind"] == "dt":
        a = _dt_inputs(case, seed)
        return {"case": case, "cfg": rich.rich_config.from_dict(_dt_cfg(case)), "arrays": a,
                "dt": torch.zeros(1, dtype=torch.float64, device="cuda")}
    if case["kind"] == "batch":
        members = _batch_members(case, seed)
        b = rich.Batch(precision=members[0]["cfg"]["precision"], max_cells=sum(len(m["x"]) for m in members))
        return {"case": case, "batch": b, "ids": [b.add(m) for m in members]}
    wl = _workload(case["problem"], case["n"], seed, case["precision"], case["scheme"], case["motion"])
    # a program's main loop keeps the arrays that it reads the state into
    names = ("x", "y", "rho", "vx", "vy", "p") if case["precision"] == "split" else ("x", "y", "m", "px", "py", "E")
    return {"case": case, "sim": rich.Sim(wl), "out": {k: np.zeros(case["n"]) for k in names}}


def run(state):
    case = state["case"]
    if case["kind"] == "dt":
        a = state["arrays"]
        ptr = [a[k].data_ptr() if k in a else 0 for k in ("area", "rho", "vx", "vy", "p", "wx", "wy")]
        rich.rich_courant_dt_noalloc(state["cfg"], case["n"], *ptr, state["dt"].data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
        return state["dt"]
    if case["kind"] == "batch":
        state["batch"].step()
        parts = [state["batch"].conserved(k) for k in state["ids"]]
        return {f: np.concatenate([q[f] for q in parts]) for f in parts[0]}
    sim, arrays = state["sim"], state["out"]
    info = sim.step(case["steps"])
    ptr = [a.ctypes.data_as(_DOUBLES) for a in arrays.values()]
    if case["precision"] == "split":
        _check(rich.lib().rich_get_state(sim.h, sim.n, *ptr, None))
        # the primitives of a split simulation are FP32 numbers
        out = {k: a if k in ("x", "y") else a.astype(np.float32) for k, a in arrays.items()}
    else:
        _check(rich.lib().rich_get_conserved(sim.h, sim.n, *ptr))
        out = dict(arrays)
    out["t"] = info["t"]
    return out


def _check(rc):
    if rc:
        raise RuntimeError(rich.lib().rich_last_error().decode())


def work(case):
    n = case["n"] if case["kind"] != "batch" else None
    if case["kind"] == "dt":
        # five to seven arrays read, about 14 operations a cell
        return {"bytes": 8 * n * (7 if case["moving"] else 5) + 8, "flops": 14 * n}
    if case["kind"] == "batch":
        lo, hi = case["n_min"], case["n_max"]
        n = case["sims"] * (hi - lo) / math.log(hi / lo)  # the mean of the log-uniform sizes
        return {"bytes": (STEP_BYTES + READ_BYTES) * n, "flops": STEP_FLOPS * n}
    sweeps = case["steps"] * (2 if case["scheme"] == "time_centred" else 1)
    return {"bytes": (STEP_BYTES * sweeps + READ_BYTES) * n, "flops": STEP_FLOPS * sweeps * n}


def exact(case, seed):
    if case["kind"] != "dt":
        return None
    a = _dt_inputs(case, seed)
    cfg = _dt_cfg(case)
    cs = torch.sqrt(cfg["gamma"] * a["p"] / a["rho"])
    ux, uy = (a["vx"] - a["wx"], a["vy"] - a["wy"]) if case["moving"] else (a["vx"], a["vy"])
    dt = torch.sqrt(a["area"] / math.pi) / (cs + torch.sqrt(ux * ux + uy * uy))
    return (cfg["cfl"] * dt.min()).reshape(1)
