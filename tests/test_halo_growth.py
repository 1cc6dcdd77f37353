"""The halo buffer of the on-chip resident steps when it cannot grow: the
solve steps per phase, nothing of the freed buffer is used afterwards (a
shorter list solves again on the chip with a buffer of its own), and every
result equals that of the one-launch-per-phase kernel bit for bit."""
import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FIELDS = (L.FIELD_MASK, L.FIELD_DRHO, L.FIELD_UX, L.FIELD_UY, L.FIELD_POPS)


@pytest.fixture(autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield
    L.lib.debug_fail_alloc(-1)


def test_a_shorter_list_after_a_failed_growth():
    # 640 segments of 12,736 words: room for 1,824 at first, an exchange of 1,300 cells may need 1,940
    cells = np.ones((400, 1024), np.uint8)
    cells[150:170] = 0
    a, b = (L.Lattice(cells, 0.8, 0.01, residual_every=0) for _ in range(2))
    b.set_step_config(8, persistent=False)

    def both(step, on_chip):
        n0 = L.kernel_launches()
        ra = step(a)
        n1 = L.kernel_launches()
        L.lib.debug_fail_alloc(-1)
        rb = step(b)
        assert (n1 - n0 < L.kernel_launches() - n1) == on_chip
        assert ra["dp"] == rb["dp"]
        for f in FIELDS:
            assert np.array_equal(a.read(f), b.read(f)), f

    both(lambda h: h.solve(40), True)
    both(lambda h: h.optimize_step(3, 40), True)  # the exchange's scratch exists from here on
    L.lib.debug_fail_alloc(0)
    both(lambda h: h.optimize_step(1300, 40), False)
    a.reset()
    b.reset()
    both(lambda h: h.solve(40), True)
    both(lambda h: h.optimize_step(1300, 40), True)
    a.close()
    b.close()


def _two_groups():
    """Channels of 10,016, 8,992 and 8,000 segments: one in the first group, two in the second, whose halo is larger."""
    return [dict(cells=I.channel(1000, h), tau=0.7, u_max=0.02) for h in (313, 281, 250)]


def test_groups_when_any_allocation_of_theirs_fails():
    members = _two_groups()
    ref = L.Batch(members, residual_every=0)
    ref.set_step_config(8, persistent=False)
    want = [r["dp"] for r in ref.solve(256)]
    pops = [ref.read(i, L.FIELD_POPS) for i in range(3)]
    ref.close()
    groups = 0
    for after in range(36):
        b = L.Batch(members, residual_every=0)
        L.lib.debug_fail_alloc(after)
        try:
            got = [r["dp"] for r in b.solve(256)]
        except L.LbmError as e:
            assert e.status == 3  # LBM_ERR_OOM
            got = None
        L.lib.debug_fail_alloc(-1)
        groups = max(groups, b.step_groups())
        if got is None:
            b.reset()
            got = [r["dp"] for r in b.solve(256)]
        assert got == want, after
        for i in range(3):
            assert np.array_equal(b.read(i, L.FIELD_POPS), pops[i]), (after, i)
        b.close()
    assert groups == 2


def test_a_batch_without_room_for_its_groups_steps_as_one_set():
    members = _two_groups()
    ref = L.Batch(members, residual_every=0)
    want = [r["dp"] for r in ref.solve(256)]
    ref.close()
    for after in (0, 5, 12):  # in the first group's buffers and in the second's
        b = L.Batch(members, residual_every=0)
        L.lib.debug_fail_alloc(after)
        assert [r["dp"] for r in b.solve(256)] == want
        L.lib.debug_fail_alloc(-1)
        assert b.step_groups() == 1
        b.close()
