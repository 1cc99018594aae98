"""Device memory that runs out."""
import contextlib

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
