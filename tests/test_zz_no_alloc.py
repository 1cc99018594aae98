"""The allocation-free time-step entry point (rich_courant_dt_noalloc).

It exists for callers that cannot allocate GPU memory where they need a time
step: code inside a device memory pool or arena that owns the GPU, and code
where the implicit device synchronisation of an allocation or free is not
allowed.  These tests check, through the C ABI, that two calls in a row
return the same time step as the regular step entry point (rich_step)
computed from the same cell values, within the tolerance of the other parity
tests, for a moving and a static mesh (where the mesh velocity may be NULL);
that it rejects what the other entry points reject; and that a bad cell
shows in the result instead of being skipped.  It lives in a file of its own
that pytest collects last."""
import math

import numpy as np
import pytest

from paper_1410_3219_gb300 import workloads as W
from tests.gpu_common import TOL

pytestmark = pytest.mark.gpu

FIELDS = ("area", "rho", "vx", "vy", "p", "wx", "wy")


def _lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_3219_gb300 import rich
    return rich


@pytest.mark.parametrize("motion", [W.MESH_LAGRANGIAN, W.MESH_EULERIAN])
def test_noalloc_time_step_matches_step_entry_point(motion):
    import torch
    rich = _lib()

    wl = W.sedov(n=20000, seed=12, motion=motion)
    sim = rich.Sim(wl)
    n = sim.n
    stream = torch.cuda.current_stream()
    out = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    for call in range(2):
        info = sim.step(1)  # regular entry point: its dt comes from the sweep's own reduction
        fields = {k: torch.tensor(sim.field(k), dtype=torch.float64, device="cuda") for k in FIELDS}
        ptrs = [fields[k].data_ptr() for k in FIELDS]
        if motion == W.MESH_EULERIAN:
            ptrs[5] = ptrs[6] = 0  # a static mesh needs no mesh velocity
        rich.rich_courant_dt_noalloc(wl["cfg"], n, *ptrs, out.data_ptr(), stream.cuda_stream)
        torch.cuda.synchronize()
        dt = float(out.item())
        assert abs(dt - info["dt_last"]) <= TOL * info["dt_last"], (call, dt, info["dt_last"])
        out.fill_(-1.0)
    sim.close()


def test_noalloc_rejects_bad_sizes_and_configs():
    import torch
    rich = _lib()

    x = torch.ones(4, dtype=torch.float64, device="cuda")
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    cfg = W.default_cfg()
    ptrs = [x.data_ptr()] * 7
    for bad_n in (0, (1 << 24) + 1):
        with pytest.raises(rich.RichError) as e:
            rich.rich_courant_dt_noalloc(cfg, bad_n, *ptrs, out.data_ptr())
        assert e.value.code == -1
    for bad in (dict(gamma=1.0), dict(cfl=0.0), dict(motion=7)):
        with pytest.raises(rich.RichError) as e:
            rich.rich_courant_dt_noalloc(dict(cfg, **bad), 4, *ptrs, out.data_ptr())
        assert e.value.code == -1
    with pytest.raises(rich.RichError):  # a moving mesh needs wx, wy
        rich.rich_courant_dt_noalloc(cfg, 4, *ptrs[:5], 0, 0, out.data_ptr())


def test_noalloc_bad_cell_gives_nan():
    import torch
    rich = _lib()

    n = 3000
    h = 1.0 / 64
    gamma = 1.4
    area = np.full(n, h * h)
    rho = np.full(n, 1.0)
    p = np.full(n, 1.0)
    v = np.zeros(n)
    cfg = W.default_cfg(gamma=gamma, motion=W.MESH_EULERIAN)
    dev = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    good = [dev(a) for a in (area, rho, v, v, p)]
    rich.rich_courant_dt_noalloc(cfg, n, *[t.data_ptr() for t in good], 0, 0, out.data_ptr())
    torch.cuda.synchronize()
    expect = cfg["cfl"] * math.sqrt(h * h / math.pi) / math.sqrt(gamma)
    assert abs(float(out.item()) - expect) <= TOL * expect
    p_bad = p.copy()
    p_bad[1234] = -1.0  # negative pressure: NaN sound speed
    bad = [dev(a) for a in (area, rho, v, v, p_bad)]
    rich.rich_courant_dt_noalloc(cfg, n, *[t.data_ptr() for t in bad], 0, 0, out.data_ptr())
    torch.cuda.synchronize()
    assert math.isnan(float(out.item()))


@pytest.mark.parametrize("n", [1, 31, 255, 1023, 1024, 1025, 1216 * 1024 + 1, 3000001])
@pytest.mark.parametrize("case", ["smooth", "equal", "wide", "huge_gamma", "still"])
def test_noalloc_minimum_over_all_cells(n, case):
    """The FP32 estimate that picks the cells to evaluate never loses the
    smallest time step: sizes around a thread's, block's and grid's share;
    cells all but equal; values far beyond the estimate's range; a fluid at
    rest.  Against the same formula over every cell in FP64: a square root
    or division is rounded once on both sides, and the sums under the second
    root differ by a fused multiply-add, so 4 ulps cover the quotient."""
    import torch
    rich = _lib()
    g = torch.Generator(device="cuda").manual_seed(n + len(case))

    def u(lo, hi):
        return torch.empty(n, dtype=torch.float64, device="cuda").uniform_(lo, hi, generator=g)

    a = {"area": u(0.5, 1.5) / n, "rho": u(0.5, 2.0), "vx": u(-1, 1), "vy": u(-1, 1), "p": u(0.5, 2.0),
         "wx": u(-1, 1), "wy": u(-1, 1)}
    gamma = 5.0 / 3.0
    if case == "equal":
        # time steps within 1e-9 of each other
        for k in FIELDS:
            a[k] = torch.ones_like(a[k]) * (1.0 + 0.1 * len(k))
        a["area"] = a["area"] * (1.0 + 1e-9 * u(0, 1))
    elif case == "wide":
        for k in ("area", "rho", "p"):
            a[k] = torch.exp2(u(-300, 300))
        a["vx"] = a["vx"] * torch.exp2(u(-200, 200))
    elif case == "huge_gamma":
        gamma = 1e30
    elif case == "still":
        a["wx"], a["wy"] = a["vx"].clone(), a["vy"].clone()
        a["wx"][: n // 2] += 1e-300
    out = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    cfg = W.default_cfg(gamma=gamma)
    for _ in range(2):
        rich.rich_courant_dt_noalloc(cfg, n, *[a[k].data_ptr() for k in FIELDS], out.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    ux, uy = a["vx"] - a["wx"], a["vy"] - a["wy"]
    dt = torch.sqrt(a["area"] * (1.0 / math.pi)) / (torch.sqrt(gamma * a["p"] / a["rho"]) + torch.sqrt(ux * ux + uy * uy))
    dt = dt[torch.isfinite(dt)]
    want = cfg["cfl"] * float(dt.min())
    assert abs(float(out.item()) - want) <= 4 * 2.0 ** -52 * want


def test_noalloc_calls_after_overlapping_ones():
    """Calls that overlap on the GPU race for the shared scratch (their own
    results are not looked at), but must not spoil the calls after them; and
    captured calls of different sizes, replayed, count their own blocks."""
    import torch
    rich = _lib()
    g = torch.Generator(device="cuda").manual_seed(3)
    n_max = 2000001
    a = {k: torch.empty(n_max, dtype=torch.float64, device="cuda").uniform_(0.5, 2.0, generator=g) for k in FIELDS}
    cfg = W.default_cfg()

    def call(n, out, stream):
        rich.rich_courant_dt_noalloc(cfg, n, *[a[k].data_ptr() for k in FIELDS], out.data_ptr(), stream.cuda_stream)

    def want(n):
        q = {k: a[k][:n] for k in FIELDS}
        ux, uy = q["vx"] - q["wx"], q["vy"] - q["wy"]
        dt = torch.sqrt(q["area"] * (1.0 / math.pi)) / (torch.sqrt(cfg["gamma"] * q["p"] / q["rho"]) +
                                                        torch.sqrt(ux * ux + uy * uy))
        return cfg["cfl"] * float(dt.min())

    sizes = [1, 700, 4097, 60001, 467000, n_max]
    wants = [want(n) for n in sizes]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    o1, o2 = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    call(1, o1, s1)
    torch.cuda.synchronize()
    graphs, outs = [], []
    for n in sizes:
        outs.append(torch.zeros(1, dtype=torch.float64, device="cuda"))
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            call(n, outs[-1], torch.cuda.current_stream())
    for rep in range(3):
        for k in range(40):
            call(sizes[(k + rep) % 6], o1, s1)
            call(sizes[(3 * k + 1) % 6], o2, s2)
        torch.cuda.synchronize()
        for n, w in zip(sizes, wants):
            call(n, o1, s1)
            s1.synchronize()
            assert abs(float(o1.item()) - w) <= 4 * 2.0 ** -52 * w, n
        for graph, out, w in zip(graphs, outs, wants):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert abs(float(out.item()) - w) <= 4 * 2.0 ** -52 * w
