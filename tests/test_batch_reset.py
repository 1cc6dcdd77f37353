"""The reset of a batch: as fast as its members' resets alone where they are
large (the same bytes are cleared)."""
import time

import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    L.lib.debug_fail_alloc(-1)


def _fastest(reset):
    best = 1e9
    for _ in range(10):
        t0 = time.perf_counter()
        reset()  # returns with the device idle
        best = min(best, time.perf_counter() - t0)
    return best


def test_large_members_reset_at_the_rate_of_their_handles():
    cells = I.channel(8192, 4094)
    one = L.Lattice(cells, 0.8, 0.02, residual_every=0)
    alone = _fastest(one.reset)
    one.close()
    two = L.Batch([dict(cells=cells, tau=0.8, u_max=0.02)] * 2, residual_every=0)
    together = _fastest(two.reset)
    two.close()
    assert together < 1.4 * 2 * alone, (together, alone)


def test_reset_succeeds_without_memory_for_its_list():
    members = [dict(cells=I.channel(64 + 8 * i, 14), tau=0.8, u_max=0.02) for i in range(3)]
    b = L.Batch(members, residual_every=0)
    first = [r["dp"] for r in b.solve(40)]
    L.lib.debug_fail_alloc(0)  # the next device allocation fails
    b.reset()
    L.lib.debug_fail_alloc(-1)
    assert [r["dp"] for r in b.solve(40)] == first
    b.close()
