"""The mesh a simulation holds on the device after steps, updated there from
step to step, equals a fresh host build of its points entry by entry, and the
steps are made by the update and not by the host builder."""
import numpy as np
import pytest

from paper_1410_3219_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_3219_gb300 import rich
    return rich


def _drift():
    wl = W.kelvin_helmholtz(n_side=64)
    wl["vx"] = wl["vx"] + 40.0  # several cells a step through the boundary
    return wl


@pytest.mark.parametrize("name,make,steps,share", [
    ("sod_64", lambda: W.sod(n_side=64), 60, 1.0),
    ("sod_rough_53", lambda: W.sod(n_side=53, jitter=0.45), 40, 1.0),
    ("kh_128", lambda: W.kelvin_helmholtz(n_side=128, amp=0.1), 40, 1.0),
    ("kh_drift", _drift, 40, 1.0),
    ("advection", lambda: W.advection(n_side=32, jitter=0.1), 20, 1.0),
    ("static", lambda: W.uniform(n_side=40, motion=W.MESH_EULERIAN), 8, None),
    ("sedov_20000", lambda: W.sedov(n=20000, seed=2), 12, 0.5),
    ("random_257", lambda: W.random_smooth(n=257), 20, 0.5),
    ("small_8", lambda: W.gresho(n_side=8), 20, 0.5),
    ("below_the_update", lambda: W.gresho(n_side=7), 4, 0.0),
])
@pytest.mark.parametrize("scheme", [W.SCHEME_EXTRAPOLATED, W.SCHEME_TIME_CENTRED])
def test_device_mesh_equals_fresh_build(R, name, make, steps, share, scheme):
    wl = make()
    wl["cfg"]["scheme"] = scheme
    sim = R.Sim(wl)
    meshes = steps * (2 if scheme == W.SCHEME_TIME_CENTRED else 1)
    for k in range(4):
        sim.step(steps // 4)
        if share is not None and share < 1.0:
            sim.tessellate()  # (a mesh left to the host is built by the next use)
        mismatched, updates = R.rich_mesh_check(sim.h)
        assert mismatched == 0, (k, updates)
    if not share:
        assert updates == 0  # a static mesh stays; a tiny one is left to the host
    else:
        assert updates >= share * meshes - 1, (updates, meshes)
    sim.close()


@pytest.mark.parametrize("n_side", [32, 33])
def test_drifting_lattice_stays_closed(R, n_side):
    """Every quadrilateral of a lattice that drifts through a periodic
    boundary is co-circular but for the rounding of its positions, which
    differs from cell to cell's own frame: the stars on the two sides of the
    boundary must still agree, every step."""
    sim = R.Sim(W.advection(n_side=n_side))
    try:
        sim.step(1)
    except R.RichError:
        pytest.skip("the host builder's own first mesh does not close")
    sim.step(150)
    _, updates = R.rich_mesh_check(sim.h)
    assert updates == 151
    sim.close()


def test_failed_and_repeated_steps_keep_the_mesh(R):
    """A failed step leaves the mesh of the points it started from; the
    pieces API updates the same mesh again."""
    wl = W.random_mixed(n=400, seed=8)
    wl["p"] = np.where(np.arange(400) == 7, 1e12, wl["p"])
    sim = R.Sim(wl)
    failed = False
    for _ in range(30):
        try:
            sim.step(1)
        except R.RichError:
            failed = True
            break
    sim.tessellate()
    assert R.rich_mesh_check(sim.h)[0] == 0
    sim.tessellate()
    assert R.rich_mesh_check(sim.h)[0] == 0
    assert failed or sim.conserved()["m"].min() > 0
    sim.close()


def test_batch_membership_changes_repack_updated_meshes(R):
    """Simulations that leave and join between steps: the others' meshes come
    from the device, and every result equals its solo run bit for bit."""
    wls = [W.sod(n_side=24, seed=1), W.gresho(n_side=30, seed=2), W.kelvin_helmholtz(n_side=20, seed=3),
           W.sod(n_side=31, seed=4), W.gresho(n_side=6, seed=5)]
    budget = [9, 4, 14, 6, 5]
    b = R.Batch(max_cells=1 << 20)
    ids = [b.add(w, max_steps=k) for w, k in zip(wls[:3], budget[:3])]
    for k in range(14):
        if k == 2:
            ids.append(b.add(wls[3], max_steps=budget[3]))
        if k == 7:
            ids.append(b.add(wls[4], max_steps=budget[4]))
        b.step()
    for w, sid, k in zip(wls, ids, budget):
        q = b.query(sid)
        assert q["state"] == "done" and q["steps"] == k
        solo = R.Sim(w)
        solo.step(k)
        got, want = b.conserved(sid), solo.conserved()
        for f in want:
            assert np.array_equal(got[f], want[f]), (sid, f)
        solo.close()
    b.close()


def test_a_second_round_after_quiet_updates(R):
    """After a run of updates that one round settled only one is launched at
    first; a rough mesh that joins then needs a second, and every result
    equals its solo run (whose first updates launch two) bit for bit."""
    quiet, rough = W.gresho(n_side=24, seed=2), W.sod(n_side=225, seed=3, jitter=0.4)
    b = R.Batch(max_cells=1 << 20)
    ids = [b.add(quiet, max_steps=14)]
    for k in range(14):
        if k == 11:
            ids.append(b.add(rough, max_steps=3))
        b.step()
    for w, sid, k in ((quiet, ids[0], 14), (rough, ids[1], 3)):
        assert b.query(sid)["state"] == "done"
        solo = R.Sim(w)
        solo.step(k)
        got, want = b.conserved(sid), solo.conserved()
        for f in want:
            assert np.array_equal(got[f], want[f]), (sid, f)
        solo.close()
    b.close()


@pytest.mark.parametrize("boundary", [W.BC_PERIODIC, W.BC_REFLECTIVE])
@pytest.mark.parametrize("points,radius", [(4, 4e-12), (5, 2e-12), (25, 7e-12), (8, 1e-9)])
def test_clusters_far_below_the_spacing(R, points, radius, boundary):
    """A few points on a circle of 1e-11 to 1e-8 mean spacings, moving apart at
    random: the kernels' FP32 in-circle sums are subnormal there, and the
    update must leave them to FP64 (the mesh equals a fresh host build)."""
    rng = np.random.default_rng(points)
    x, y = W.jittered_lattice(15, 15, 0.0, 1.0, 0.0, 1.0, 0.3, rng)
    c = np.array([0.431, 0.562])
    far = np.hypot(x - c[0], y - c[1]) > 0.03
    angle = 2 * np.pi * (np.arange(points) + rng.uniform(-0.3, 0.3, points)) / points
    x = np.concatenate([x[far], c[0] + radius * np.cos(angle)])
    y = np.concatenate([y[far], c[1] + radius * np.sin(angle)])
    wl = dict(name="cluster", seed=points, cfg=W.default_cfg(boundary=boundary, gamma=1.4), x=x, y=y,
              rho=np.ones(x.size), vx=rng.uniform(-1, 1, x.size), vy=rng.uniform(-1, 1, x.size), p=np.ones(x.size))
    sim = R.Sim(wl)
    for k in range(3):
        try:
            sim.step(1)
        except R.RichError:
            # (cells this unequal may empty: the mesh is then that of the last good step)
            sim.tessellate()
        mismatched, updates = R.rich_mesh_check(sim.h)
        assert mismatched == 0
        assert updates >= 1
    sim.close()


@pytest.mark.parametrize("seed", [3, 4, 5])
def test_refill_after_members_ended_together(R, seed):
    """Every member of a batch ends in a step whose mesh update needed another
    round than the one launched (after quiet updates, a rough mesh's first
    step): what that update had told cells of others must not reach the
    smaller simulations that fill the batch next, whose results equal their
    solo runs bit for bit."""
    b = R.Batch(max_cells=1 << 20)
    b.add(W.gresho(n_side=24, seed=2), max_steps=12)
    for k in range(12):
        if k == 11:
            b.add(W.sod(n_side=225, seed=seed, jitter=0.4), max_steps=1)
        b.step()
    wls = [W.sod(n_side=40, seed=seed, jitter=0.4), W.kelvin_helmholtz(n_side=50, seed=seed, amp=0.2),
           W.sod(n_side=33, seed=seed + 10, jitter=0.3)]
    ids = [b.add(w, max_steps=6) for w in wls]
    for _ in range(6):
        b.step()
    for w, sid in zip(wls, ids):
        assert b.query(sid)["state"] == "done"
        solo = R.Sim(w)
        solo.step(6)
        got, want = b.conserved(sid), solo.conserved()
        for f in want:
            assert np.array_equal(got[f], want[f]), (sid, f)
        solo.close()
    b.close()


def test_flags_of_a_larger_packing_are_cleared(R):
    """A batch of three, two and three simulations: the first packing's third
    one (a box too small for the update) leaves its flag in one of the two
    counter buffers, which the second packing's update does not reach; the
    third packing's third simulation must be updated on the device."""
    b = R.Batch(max_cells=1 << 20)
    for k, steps in ((24, 8), (28, 8)):
        b.add(W.gresho(n_side=k, seed=k), max_steps=steps)
    b.add(W.uniform(n_side=2, jitter=0.2, seed=34), max_steps=1)
    b.step()
    b.step()
    late = b.add(W.gresho(n_side=32, seed=6), max_steps=4)
    for _ in range(4):
        b.step()
    assert b.query(late)["state"] == "done"
    # the four first meshes only; two members' updates after each of six
    # steps, and the late one's after its first three
    assert b.mesh_counts() == (2 * 6 + 3, 4)
    b.close()


def _hub(spokes=40, n_side=20):
    """A gas at rest with one cell of `spokes` neighbours."""
    wl = W.uniform(n_side=n_side, vx=0.0, vy=0.0, jitter=0.2)
    far = np.hypot(wl["x"] - 0.5, wl["y"] - 0.5) > 0.2
    angle = 2 * np.pi * (np.arange(spokes) + 0.5) / spokes
    wl["x"] = np.concatenate([[0.5], wl["x"][far], 0.5 + 0.16 * np.cos(angle)])
    wl["y"] = np.concatenate([[0.5], wl["y"][far], 0.5 + 0.16 * np.sin(angle)])
    for k, v in (("rho", 1.0), ("vx", 0.0), ("vy", 0.0), ("p", 1.0)):
        wl[k] = np.full(wl["x"].size, v)
    wl["cfg"]["chi"] = 0.0  # (no rounding: the ring stays)
    return wl


@pytest.mark.parametrize("place", [0, 1, 2])
def test_a_member_left_to_the_host_leaves_the_others_on_the_device(R, place):
    """A cell of more than 32 neighbours beside small ones is more than the
    update's lists take: that simulation's meshes are built on the host, and
    only its."""
    wls = [W.gresho(n_side=24, seed=2), W.sod(n_side=30, seed=3)]
    wls.insert(place, _hub())
    b = R.Batch(max_cells=1 << 20)
    ids = [b.add(w, max_steps=6) for w in wls]
    for _ in range(6):
        b.step()
    updated, built = b.mesh_counts()
    assert (updated, built) == (2 * 5, 3 + 5)
    for w, sid in zip(wls, ids):
        assert b.query(sid)["state"] == "done"
        solo = R.Sim(w)
        solo.step(6)
        got, want = b.conserved(sid), solo.conserved()
        for f in want:
            assert np.array_equal(got[f], want[f]), (sid, f)
        solo.close()
    b.close()


@pytest.mark.parametrize("n_side", [32, 33])
def test_drifting_lattice_equals_fresh_builds_and_restarts(R, n_side):
    """Near-ties across the periodic boundary: the device's mesh is the host's
    entry by entry at every step, and a restart from a checkpoint, whose
    first mesh is the host's, continues bit for bit."""
    sim = R.Sim(W.advection(n_side=n_side))
    for k in range(40):
        sim.step(3)
        assert R.rich_mesh_check(sim.h) == (0, 3 * (k + 1))
        if k == 20:
            other = R.Sim.restart(W.advection(n_side=n_side)["cfg"], sim.checkpoint())
    other.step(3 * 19)
    got, want = other.conserved(), sim.conserved()
    for f in want:
        assert np.array_equal(got[f], want[f]), f
    sim.close()
    other.close()


def _mesh_is_current(R, sim):
    try:
        assert R.rich_mesh_check(sim.h)[0] == 0
        return True
    except R.RichError as e:
        assert e.code == R.RICH_ESTATE
        return False


@pytest.mark.parametrize("scheme", [W.SCHEME_EXTRAPOLATED, W.SCHEME_TIME_CENTRED])
@pytest.mark.parametrize("name", ["hub", "small"])
def test_meshes_left_to_the_host_are_built_beside_the_sweep(R, name, scheme):
    """Where the update keeps failing (a cell of 40 neighbours) or is not tried
    (49 cells), the host builds the next mesh while the sweep ends, so a step
    leaves the mesh of its points; now and then the update is tried again.
    Results equal those of the pieces API, which builds every mesh anew."""
    wl = _hub() if name == "hub" else W.gresho(n_side=7)
    wl["cfg"]["scheme"] = scheme
    sim = R.Sim(wl)
    current = 0
    for _ in range(20):
        sim.step(1)
        current += _mesh_is_current(R, sim)
    assert current >= (20 if name == "small" else 12)
    if name == "small":
        sim.step(1, R.rich_time(sim.h) + 1e-9)  # lands on t_end: no mesh is built
        assert not _mesh_is_current(R, sim)
    pieces = R.Sim(wl)
    for _ in range(20 * (2 if scheme == W.SCHEME_TIME_CENTRED else 1)):
        pieces.tessellate()
        pieces.sweep()
        pieces.sync()
    if name == "small":
        pieces.tessellate()
        pieces.sweep(R.rich_time(pieces.h) + 1e-9)
        pieces.sync()
        if scheme == W.SCHEME_TIME_CENTRED:
            pieces.tessellate()
            pieces.sweep(R.rich_time(pieces.h) + 1e-9)
            pieces.sync()
    got, want = sim.conserved(), pieces.conserved()
    for f in want:
        assert np.array_equal(got[f], want[f]), f
    sim.close()
    pieces.close()


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("others", [False, True])
def test_members_that_keep_failing_are_built_beside_the_sweep(R, mode, others):
    """Simulations whose every update fails, alone and beside others: their
    meshes come from the host (in a staged sweep while it ends), each once, and
    results equal the solo runs bit for bit, also when members end or fail."""
    wls = [_hub(), _hub(36, 24), _hub(50, 30)]
    budget = [20, 13, 17]
    if others:
        wls += [W.gresho(n_side=24, seed=2), W.sod(n_side=30, seed=3)]
        budget += [20, 9]
    bad = W.random_mixed(n=400, seed=8)
    bad["p"] = np.where(np.arange(400) == 7, 1e12, bad["p"])
    b = R.Batch(max_cells=1 << 20)
    b.set_launch(mode, 256)
    ids = [b.add(w, max_steps=k) for w, k in zip(wls, budget)]
    if others:
        b.add(bad, max_steps=20)
    for _ in range(20):
        b.step()
    updated, built = b.mesh_counts()
    if not others:
        assert (updated, built) == (0, sum(budget))
    for w, sid, k in zip(wls, ids, budget):
        q = b.query(sid)
        assert q["state"] == "done" and q["steps"] == k
        solo = R.Sim(w)
        solo.step(k)
        got, want = b.conserved(sid), solo.conserved()
        for f in want:
            assert np.array_equal(got[f], want[f]), (sid, f)
        solo.close()
    b.close()
