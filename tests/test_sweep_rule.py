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
