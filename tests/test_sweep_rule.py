"""The rule that sends a lattice to sweeps, unforced: where it says no, a solve
launches what it would without sweeps, also after an exchange and a reset."""
import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _pillars(nx, ny):
    """A channel with a solid cell at every second place both ways: a wall in every tile row."""
    cells = I.channel(nx, ny - 2)
    cells[2:-2:2, 4:-4:2] = 1
    return cells


def _launches(lat, step):
    n0 = L.kernel_launches()
    step(lat)
    return L.kernel_launches() - n0


def test_no_row_list_where_the_answer_stays_no(monkeypatch):
    cells = _pillars(2600, 2600)  # 182 MB of fluid populations, walls everywhere: asked once, then no
    steps = (lambda h: h.solve(16), lambda h: h.optimize_step(5, 16), lambda h: h.reset(), lambda h: h.solve(16),
             lambda h: h.optimize_step(5, 16))
    a = L.Lattice(cells, 0.8, 0.01, residual_every=0)
    got = [_launches(a, s) for s in steps]
    a.close()
    monkeypatch.setenv("LBM_SWEEP", "0")
    b = L.Lattice(cells, 0.8, 0.01, residual_every=0)
    want = [_launches(b, s) for s in steps]
    b.close()
    assert got[0] > want[0]  # the first question is asked
    assert got[1:] == want[1:]


FIELDS = (L.FIELD_MASK, L.FIELD_DRHO, L.FIELD_UX, L.FIELD_UY, L.FIELD_POPS)


@pytest.mark.parametrize("fails", [-1, 0, 1])  # no allocation; the row list's; the second buffer's
def test_the_rule_takes_sweeps_beyond_the_cache(fails):
    cells = I.channel_array(4000, 2000, 4)  # 144 MB of fluid populations in open rows
    a, b = (L.Lattice(cells, 0.6, 0.05, residual_every=20) for _ in range(2))
    b.set_step_config(8, persistent=False)
    for i, step in enumerate((lambda h: h.solve(8), lambda h: h.solve(100), lambda h: h.optimize_step(200, 40),
                              lambda h: h.solve(8), lambda h: h.solve(50))):
        if i == 1:
            L.lib.debug_fail_alloc(fails)
        n0 = L.kernel_launches()
        ra = step(a)
        n1 = L.kernel_launches()
        L.lib.debug_fail_alloc(-1)
        rb = step(b)
        per_phase = L.kernel_launches() - n1
        if i in (0, 3) or (i == 1 and fails >= 0):  # short, or no memory: one launch per phase
            assert n1 - n0 >= per_phase, i
        else:
            assert n1 - n0 < per_phase, i
        assert ra["dp"] == rb["dp"] and ra["m_in"] == rb["m_in"] and ra["residual"] == rb["residual"], i
        assert list(ra["m_out"]) == list(rb["m_out"])
        for f in FIELDS:
            assert np.array_equal(a.read(f), b.read(f)), (i, f)
    a.close()
    b.close()
