"""The device's mesh update (star splaying over the cells whose neighbours
changed) run serially on the host: its meshes equal fresh host builds entry
by entry (rings, offsets, processing order, ghosts), over periodic and walled
boxes, co-circular lattices (every edge decided by the exact predicates and
the tie-break), points crossing walls and periodic boundaries, sheared rows
(large reconnections), drifts of several cells a step, elongated and offset
boxes, and the smallest sizes."""
import numpy as np
import pytest

from paper_1410_3219_gb300 import rich as R
from paper_1410_3219_gb300 import workloads as W


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build_library()


def _walk(box, boundary, nx, ny, jitter, step, steps, drift=0.0, rows=0.0, seed=0):
    """Successive point sets: a jittered lattice whose points move by up to
    `step` spacings at random, drift together, and slide in alternate bands."""
    x0, x1, y0, y1 = box
    rng = np.random.default_rng(seed)
    hx, hy = (x1 - x0) / nx, (y1 - y0) / ny
    x, y = W.jittered_lattice(nx, ny, x0, x1, y0, y1, jitter, rng)
    xs, ys = [x], [y]
    for _ in range(steps - 1):
        x = x + rng.uniform(-step, step, x.size) * hx + drift * hx * rng.uniform(-1, 1)
        y = y + rng.uniform(-step, step, y.size) * hy + drift * hy * rng.uniform(-1, 1)
        if rows:
            u = (x - x0) / (x1 - x0)
            x = x + np.where(np.floor((y - y0) / (y1 - y0) * 8) % 2 == 0, rows, -rows) * hx * (
                1.0 if boundary else 4.0 * u * (1.0 - u))
        if boundary == W.BC_PERIODIC:
            x, y = x0 + np.mod(x - x0, x1 - x0), y0 + np.mod(y - y0, y1 - y0)
            x, y = np.where(x >= x1, x0, x), np.where(y >= y1, y0, y)
        else:
            x = np.where(x <= x0, 2 * x0 - x, np.where(x >= x1, 2 * x1 - x, x))
            y = np.where(y <= y0, 2 * y0 - y, np.where(y >= y1, 2 * y1 - y, y))
        xs.append(x)
        ys.append(y)
    return np.array(xs), np.array(ys)


UNIT = (0.0, 1.0, 0.0, 1.0)


@pytest.mark.parametrize("boundary", [W.BC_PERIODIC, W.BC_REFLECTIVE])
@pytest.mark.parametrize("name,kw,least", [
    ("jittered", dict(box=UNIT, nx=40, ny=40, jitter=0.1, step=0.02, steps=12), 11),
    ("rough", dict(box=UNIT, nx=33, ny=37, jitter=0.45, step=0.1, steps=12), 11),
    ("lattice_at_rest", dict(box=UNIT, nx=32, ny=32, jitter=0.0, step=0.0, steps=3), 2),
    ("lattice_inexact", dict(box=(-0.3, 0.7, 0.1, 1.1), nx=29, ny=29, jitter=0.0, step=0.0, steps=3), 2),
    ("lattice_sheared", dict(box=UNIT, nx=32, ny=32, jitter=0.0, step=0.0, rows=0.25, steps=9), 8),
    ("large_moves", dict(box=UNIT, nx=32, ny=32, jitter=0.1, step=0.25, steps=10), 9),
    ("sliding_rows", dict(box=UNIT, nx=48, ny=48, jitter=0.1, step=0.02, rows=0.4, steps=12), 11),
    ("elongated_box", dict(box=(-4.0, 12.0, 3.0, 5.0), nx=96, ny=12, jitter=0.2, step=0.05, steps=10), 9),
    ("tiny_box_far_away", dict(box=(7.0, 7.0 + 1e-6, -3.0, -3.0 + 1e-6), nx=24, ny=24, jitter=0.2, step=0.05, steps=6),
     5),
    ("eight_by_eight", dict(box=UNIT, nx=8, ny=8, jitter=0.1, step=0.03, steps=12), 6),
])
def test_update_equals_fresh_build(name, kw, least, boundary):
    xs, ys = _walk(boundary=boundary, **kw)
    box = kw["box"]
    cfg = W.default_cfg(boundary=boundary, x0=box[0], x1=box[1], y0=box[2], y1=box[3])
    mismatched, updated, _ = R.rich_device_update_check(cfg, xs, ys)
    assert mismatched == 0
    assert updated >= least


def test_update_follows_a_drift_through_the_periodic_boundary():
    xs, ys = _walk(UNIT, W.BC_PERIODIC, 32, 32, 0.1, 0.02, 20, drift=3.0)
    mismatched, updated, _ = R.rich_device_update_check(W.default_cfg(), xs, ys)
    assert (mismatched, updated) == (0, 19)


@pytest.mark.parametrize("n", [3, 5, 16, 64, 257, 1023, 1025])
@pytest.mark.parametrize("boundary", [W.BC_PERIODIC, W.BC_REFLECTIVE])
def test_random_points_of_ragged_sizes(n, boundary):
    """What the update cannot make (small boxes) it leaves to the host; what
    it makes equals the fresh build."""
    rng = np.random.default_rng(n)
    x, y = rng.uniform(0.02, 0.98, n), rng.uniform(0.02, 0.98, n)
    d = 0.05 / np.sqrt(n)
    sets = []
    for _ in range(6):
        sets.append((x, y))
        x = np.clip(x + rng.uniform(-d, d, n), 0.001, 0.999)
        y = np.clip(y + rng.uniform(-d, d, n), 0.001, 0.999)
    cfg = W.default_cfg(boundary=boundary)
    mismatched, updated, _ = R.rich_device_update_check(cfg, np.array([s[0] for s in sets]),
                                                        np.array([s[1] for s in sets]))
    assert mismatched == 0
    if n >= 257:
        assert updated == 5


def test_coincident_points_are_left_to_the_host_builder():
    rng = np.random.default_rng(3)
    x, y = W.jittered_lattice(16, 16, 0.0, 1.0, 0.0, 1.0, 0.1, rng)
    x2, y2 = x.copy(), y.copy()
    x2[17], y2[17] = x[18], y[18]
    with pytest.raises(R.RichError, match="EDUPLICATE"):
        R.rich_device_update_check(W.default_cfg(), np.array([x, x2]), np.array([y, y2]))


@pytest.mark.parametrize("boundary", [W.BC_PERIODIC, W.BC_REFLECTIVE])
@pytest.mark.parametrize("points,radius,noise,seed", [(4, 4e-12, 1e-5, 76), (5, 2e-12, 1e-5, 110), (8, 2e-12, 1e-5, 71),
                                                       (25, 7e-12, 1e-4, 3), (6, 1e-10, 1e-5, 5), (6, 1e-8, 1e-6, 6)])
def test_clusters_far_below_the_spacing(points, radius, noise, seed, boundary):
    """Points on a circle of 1e-11 to 1e-7 mean spacings among 200 others: the
    products of FP32 in-circle sums fall below its normal range, and their
    signs must not be taken."""
    rng = np.random.default_rng(seed)
    x, y = W.jittered_lattice(15, 15, 0.0, 1.0, 0.0, 1.0, 0.3, rng)
    c = rng.uniform(0.3, 0.7, 2)
    far = np.hypot(x - c[0], y - c[1]) > 0.03
    x, y = x[far], y[far]
    angle = 2 * np.pi * (np.arange(points) + rng.uniform(-0.3, 0.3, points)) / points
    sets = []
    for _ in range(2):
        r = radius * (1 + rng.uniform(-noise, noise, points))
        sets.append((np.concatenate([x, c[0] + r * np.cos(angle)]), np.concatenate([y, c[1] + r * np.sin(angle)])))
    mismatched, updated, _ = R.rich_device_update_check(W.default_cfg(boundary=boundary),
                                                        np.array([s[0] for s in sets]), np.array([s[1] for s in sets]))
    assert (mismatched, updated) == (0, 1)


@pytest.mark.parametrize("boundary", [W.BC_PERIODIC, W.BC_REFLECTIVE])
@pytest.mark.parametrize("side", [1e-60, 1e-38, 1e-35, 1e-34, 1e-30, 1e38, 1e60])
def test_boxes_of_any_unit(side, boundary):
    """Offsets are scaled by the point spacing before FP32 holds them, so a
    box's unit does not cut them to zero or infinity."""
    for seed in range(4):
        xs, ys = _walk((0.0, side, 0.0, side), boundary, 20, 20, 0.05 * (1 + seed), 0.02, 6, seed=seed)
        cfg = W.default_cfg(boundary=boundary, x0=0.0, x1=side, y0=0.0, y1=side)
        mismatched, updated, _ = R.rich_device_update_check(cfg, xs, ys)
        assert (mismatched, updated) == (0, 5)


def _drifting(n_side, noise, steps, holes, seed=0):
    """A square lattice (with holes of 2 x 2 points: eight co-circular points
    around each) that drifts through a periodic box, its positions off the
    lattice by their rounding and by `noise`."""
    wl = W.advection(n_side=n_side)
    x, y = wl["x"], wl["y"]
    if holes:
        i, j = np.arange(n_side * n_side) % n_side, np.arange(n_side * n_side) // n_side
        keep = ~(((i % 8) // 2 == 0) & ((j % 8) // 2 == 0))
        x, y = x[keep], y[keep]
    rng = np.random.default_rng(seed)
    xs, ys = [], []
    for _ in range(steps):
        x, y = -0.5 + np.mod(x + 0.5, 1.0), -0.5 + np.mod(y + 0.5, 1.0)
        x, y = np.where(x >= 0.5, -0.5, x), np.where(y >= 0.5, -0.5, y)
        xs.append(x)
        ys.append(y)
        x = x + 0.231 / n_side + rng.uniform(-noise, noise, x.size)
        y = y + 0.231 / n_side + rng.uniform(-noise, noise, y.size)
    return np.array(xs), np.array(ys), wl["cfg"]


@pytest.mark.parametrize("holes", [False, True])
@pytest.mark.parametrize("n_side", [24, 33])
@pytest.mark.parametrize("noise", [0.0, 1e-16, 1e-15, 1e-14])
def test_near_ties_across_the_periodic_boundary(n_side, noise, holes):
    """In-circle tests that the rounding of periodic images decides: every copy
    of the four points must come to the same answer, in the update and in the
    host builder (fresh and in place, whose lists must close)."""
    xs, ys, cfg = _drifting(n_side, noise, 40, holes)
    mismatched, updated, _ = R.rich_device_update_check(cfg, xs, ys)
    assert (mismatched, updated) == (0, 39)
    assert R.rich_mesh_update_check(cfg, xs, ys)[0] == 0
