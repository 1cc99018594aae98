"""GPU edge cases through the C ABI, against the oracle where a step is
defined: the fewest points a box takes, collinear generating points (the
mirror images make the set two-dimensional), coincident points (rejected),
and a step that must land exactly on t_end."""
import numpy as np
import pytest

from paper_1410_3219_gb300 import workloads as W
from tests.gpu_common import TOL, compare_conserved

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_3219_gb300 import rich
    return rich


def _wl(x, y, boundary, seed=0):
    rng = np.random.default_rng(seed)
    n = len(x)
    cfg = W.default_cfg(boundary=boundary, gamma=1.4)
    return dict(name="edge", seed=seed, cfg=cfg, x=np.asarray(x, np.float64), y=np.asarray(y, np.float64),
                rho=1.0 + 0.2 * rng.random(n), vx=0.1 * rng.standard_normal(n), vy=0.1 * rng.standard_normal(n),
                p=1.0 + 0.2 * rng.random(n))


@pytest.mark.parametrize("boundary", [W.BC_PERIODIC, W.BC_REFLECTIVE])
@pytest.mark.parametrize("n", [3, 4, 7])
def test_fewest_points_match_oracle(R, oracle, n, boundary):
    rng = np.random.default_rng(100 + n)
    wl = _wl(0.1 + 0.8 * rng.random(n), 0.1 + 0.8 * rng.random(n), boundary, seed=n)
    gpu, ref = R.Sim(wl), oracle.Sim(wl)
    for _ in range(3):
        info = gpu.step(1)
        dt = ref.step()
        assert abs(info["dt_last"] - dt) <= 10 * TOL * dt
    compare_conserved(gpu, ref, wl["cfg"], tol=1e-11)
    gpu.close()


def test_collinear_points_match_oracle(R, oracle):
    """Generating points on one line: the Voronoi cells are strips between
    the walls, and every quadruple of two neighbours and their mirror images
    is co-circular.  One step is compared: the line is not a stable state of
    the scheme (in the oracle too, a point's distance from the line grows by
    ~10^4 per step from round-off, and with random velocities a strip
    empties in the second step), so later steps amplify each side's own
    round-off.  The tolerance is 1e-10: a strip of width w between walls a
    distance 1 apart gets its area from cross products of vectors ~1/(2 w)
    times longer than the strip is wide, so its geometry carries that much
    more round-off than a round cell's."""
    rng = np.random.default_rng(7)
    x = np.sort(rng.uniform(0.05, 0.95, 40))
    wl = _wl(x, np.full(40, 0.5), W.BC_REFLECTIVE, seed=7)
    wl["vx"] = np.zeros(40)
    wl["vy"] = np.zeros(40)
    wl["p"] = np.ones(40)
    gpu, ref = R.Sim(wl), oracle.Sim(wl)
    info = gpu.step(1)
    dt = ref.step()
    assert abs(info["dt_last"] - dt) <= 1e-10 * dt
    compare_conserved(gpu, ref, wl["cfg"], tol=1e-10)
    gpu.close()


def test_coincident_points_are_rejected(R):
    wl = W.sod(n_side=8)
    wl["x"], wl["y"] = wl["x"].copy(), wl["y"].copy()
    wl["x"][5], wl["y"][5] = wl["x"][9], wl["y"][9]
    with pytest.raises(R.RichError) as e:
        R.Sim(wl)
    assert e.value.code == R.RICH_EDUPLICATE


def test_last_step_lands_on_t_end(R, oracle):
    wl = W.sod(n_side=16)
    gpu, ref = R.Sim(wl), oracle.Sim(wl)
    dt0 = ref.step()  # one full step, then aim a little past it
    t_end = 1.5 * dt0
    ref.step(t_end)
    info = gpu.step(10, t_end)
    assert info["steps_done"] == 2
    assert info["t"] == t_end and R.rich_time(gpu.h) == t_end
    compare_conserved(gpu, ref, wl["cfg"])
    gpu.close()


@pytest.mark.parametrize("name", ["sod_reflective", "kh_periodic", "random_reflective", "tiny_periodic",
                                  "lattice_periodic"])
def test_device_edge_list_equals_host_list(R, name):
    """The edge list the sweep uses is built on the device from the rings;
    it must equal, entry by entry, the list the host builder makes for the
    same mesh: a reflective box, a periodic box, random points, a periodic
    box so small that cells neighbour their own images, and a co-circular
    lattice."""
    if name == "sod_reflective":
        wl = W.sod(n_side=40, seed=31)
    elif name == "kh_periodic":
        wl = W.kelvin_helmholtz(n_side=48, seed=32)
    elif name == "random_reflective":
        wl = W.random_mixed(n=3000, seed=33)
    elif name == "tiny_periodic":
        wl = W.uniform(n_side=2, jitter=0.2, seed=34)
    else:
        wl = W.uniform(n_side=12, jitter=0.0, seed=35)
    edges, bad = R.rich_edge_list_check(wl["cfg"], wl["x"], wl["y"])
    assert edges > 0 and bad == 0, (name, edges, bad)


@pytest.mark.parametrize("limiter", [W.LIM_SWITCHED, W.LIM_AREPO, W.LIM_TESS])
@pytest.mark.parametrize("power", [-300, -130, 120, 127, 128, 140, 200, 300])
def test_units_of_mass_scale_out(R, power, limiter):
    """Density and pressure times a power of two: every FP64 operation of a
    step scales exactly, so the points and velocities stay the same bits and
    the conserved state is the unscaled one times that power.  The FP32
    estimates behind the limiter's decisions do not scale (they end at 2^128),
    and must leave such values to FP64."""
    wl = W.random_mixed(n=400, seed=8)
    wl["cfg"]["limiter"] = limiter
    big = dict(wl, rho=np.ldexp(wl["rho"], power), p=np.ldexp(wl["p"], power))
    a, b = R.Sim(wl), R.Sim(big)
    for _ in range(3):
        ia, ib = a.step(1), b.step(1)
        assert ia["dt_last"] == ib["dt_last"]
    ca, cb = a.conserved(), b.conserved()
    for k in ("x", "y"):
        assert np.array_equal(ca[k], cb[k]), k
    for k in ("m", "px", "py", "E"):
        assert np.array_equal(np.ldexp(ca[k], power), cb[k]), k
    a.close()
    b.close()


@pytest.mark.parametrize("delta_p,drop,fires", [(1e-50, 1e-53, True), (1e-50, 1e-47, False), (1e-43, 1e-45, True),
                                                 (1e-37, 1e-39, True), (0.0, 1e-53, False), (0.7, 0.5, True),
                                                 (0.7, 0.9, False)])
def test_pressure_switch_at_any_threshold(R, delta_p, drop, fires):
    """min(p_i, p_j) < delta_p max(p_i, p_j) over the edges of a disc of low
    pressure in a gas at rest: the switch fires in the cells beside its rim or
    nowhere, for thresholds that FP32 cannot hold too."""
    wl = W.uniform(n_side=20, vx=0.0, vy=0.0)
    wl["cfg"]["delta_p"], wl["cfg"]["delta_v"] = delta_p, 1e300
    inside = np.hypot(wl["x"] - 0.5, wl["y"] - 0.5) < 0.25
    wl["p"] = np.where(inside, 1e25 * drop, 1e25)
    sim = R.Sim(wl)
    try:
        sim.step(1)
    except R.RichError:
        pass  # (cells of such a jump may empty; the switch describes the attempt)
    tess = sim.field("tess")
    assert (tess.sum() > 20) == fires and (fires or tess.sum() == 0)
    sim.close()


@pytest.mark.parametrize("bulk", [16.0, 128.0, 1024.0, -1024.0])
def test_mass_fluxes_do_not_depend_on_the_frame(R, bulk):
    """A step in a frame that moves through the box at up to 1,000 sound
    speeds.  On a lattice of 2^-5 spacings with densities of 1 and 2, a
    gamma of 2 and pressures of 12 bits the primitives, the gradients and the
    velocities relative to the moving edges are exact in both frames, so the
    predicted states and the mass fluxes must have the same bits: nothing on
    the way to them may be rounded at the speed of the frame."""
    wl = W.advection(n_side=32)
    rng = np.random.default_rng(7)
    wl["cfg"].update(gamma=2.0, chi=0.0)
    n = wl["x"].size
    wl["rho"] = np.where(rng.random(n) < 0.5, 1.0, 2.0)
    wl["p"] = rng.integers(3000, 5000, n) / 4096.0
    out = []
    for v in (0.0, bulk):
        sim = R.Sim(dict(wl, vx=np.full(n, v), vy=np.full(n, -0.5 * v)))
        dt = sim.step(1)["dt_last"]
        out.append((dt, sim.conserved()["m"]))
        sim.close()
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
    assert np.abs(out[0][1] / 2.0 ** -10 - wl["rho"]).max() > 1e-3


@pytest.mark.parametrize("n_side", [127, 128, 129, 138, 139])
def test_reads_on_both_sides_of_the_page_locked_size(R, n_side):
    """Reads through page-locked memory (up to 7/8 MB: 19,114 cells of six
    fields, 16,384 of seven) and through the device's memory give the caller's
    cells in the caller's order, null outputs left out."""
    wl = W.kelvin_helmholtz(n_side=n_side, seed=n_side)
    sim = R.Sim(wl)
    c, s = sim.conserved(), sim.state()
    for k in ("x", "y"):
        assert np.array_equal(c[k], wl[k]) and np.array_equal(s[k], wl[k])
    assert np.array_equal(np.rint(s["rho"]), np.rint(wl["rho"]))
    assert np.allclose(c["m"], s["rho"] * s["area"], rtol=1e-12)
    import ctypes as C
    m = np.zeros(sim.n)
    assert R.lib().rich_get_conserved(sim.h, sim.n, None, None, m.ctypes.data_as(C.POINTER(C.c_double)), None, None,
                                      None) == 0
    assert np.array_equal(m, c["m"])
    sim.close()
