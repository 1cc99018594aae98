"""Device memory that runs out: what a simulation or a batch can do without is
given up, and the results stay those of a run with room."""
import contextlib

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


@contextlib.contextmanager
def _filled(keep):
    """All but about `keep` bytes of device memory taken."""
    import torch
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = [torch.empty(max(0, free - keep), dtype=torch.uint8, device="cuda")]
    try:
        yield
    finally:
        held.clear()
        torch.cuda.empty_cache()


def _same(got, want):
    for f in want:
        assert np.array_equal(got[f], want[f]), f


def test_creation_after_one_that_found_no_memory(R):
    """A failed allocation fails its own call only."""
    wl = W.kelvin_helmholtz(n_side=512)
    with _filled(64 << 20):
        with pytest.raises(R.RichError) as e:
            R.Sim(wl)
        assert e.value.code == R.RICH_ENOMEM
    sim = R.Sim(wl)
    sim.step(1)
    sim.close()


def test_a_step_without_room_for_the_update(R):
    """The first step's update finds no memory: the host builds the meshes, and
    once there is room the update takes over again."""
    wl = W.kelvin_helmholtz(n_side=512)
    ref, sim = R.Sim(wl), R.Sim(wl)
    ref.step(3)
    with _filled(24 << 20):
        sim.step(3)
        sim.tessellate()
        assert R.rich_mesh_check(sim.h) == (0, 0)
    _same(sim.conserved(), ref.conserved())
    ref.step(20)
    sim.step(20)
    mismatched, updates = R.rich_mesh_check(sim.h)
    assert mismatched == 0 and updates >= 8
    _same(sim.conserved(), ref.conserved())
    ref.close()
    sim.close()


def test_where_a_simulation_fits_its_steps_do(R):
    """With the least memory that a simulation can be created in (to 8 MiB) it
    steps as well, whatever of the update's room did not fit."""
    wl = W.kelvin_helmholtz(n_side=400)
    ref = R.Sim(wl)
    ref.step(3)
    sim = None
    for keep in range(64, 1024, 8):
        with _filled(keep << 20):
            try:
                sim = R.Sim(wl)
            except R.RichError as e:
                assert e.code == R.RICH_ENOMEM
                continue
            sim.step(3)
        break
    _same(sim.conserved(), ref.conserved())
    ref.close()
    sim.close()


@pytest.mark.parametrize("mode", [1, 2])
def test_a_batch_without_room_for_the_update(R, mode):
    import torch
    wls = [W.kelvin_helmholtz(n_side=300, seed=k) for k in range(3)]
    solo = []
    for w in wls:
        s = R.Sim(w)
        s.step(12)
        solo.append(s.conserved())
        s.close()
    b = R.Batch(max_cells=1 << 20)
    b.set_launch(mode, 256)
    ids = [b.add(w, max_steps=12) for w in wls]
    # the packed arrays of a first step, with a few MiB beside them for the
    # update, which needs some 70
    probe = R.Batch(max_cells=1 << 20)
    probe.set_launch(mode, 256)
    for w in wls:
        probe.add(dict(w, cfg=dict(w["cfg"], motion=W.MESH_EULERIAN)))
    before = torch.cuda.mem_get_info()[0]
    probe.step()
    packed = before - torch.cuda.mem_get_info()[0]
    probe.close()
    with _filled(packed + (24 << 20)):
        for _ in range(4):
            b.step()
        updated, built = b.mesh_counts()
        assert updated == 0 and built >= 12
    for _ in range(8):
        b.step()
    assert b.mesh_counts()[0] > 0
    for sid, want in zip(ids, solo):
        _same(b.conserved(sid), want)
    b.close()


@pytest.mark.parametrize("precision", [W.FP64, W.FP32_SPLIT])
def test_reads_without_room_on_the_device(R, precision):
    """A read that finds no device memory to reorder in is reordered by the host."""
    wl = W.kelvin_helmholtz(n_side=512)
    wl["cfg"]["precision"] = precision
    ref, sim = R.Sim(wl), R.Sim(wl)
    b = R.Batch(precision=precision, max_cells=1 << 20)
    sid = b.add(wl)
    b.step()
    ref.step(1)
    sim.step(1)
    want = ref.conserved(), ref.state()
    sim.tessellate()
    with _filled(4 << 20):
        got, state, member = sim.conserved(), sim.state(), b.conserved(sid)
    _same(got, want[0])
    _same(state, want[1])
    _same(member, want[0])
    for h in (ref, sim, b):
        h.close()
