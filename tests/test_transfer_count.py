"""lbm_transfer_bytes counts the copies of a reset: of every member its fluid
count (8 bytes) and of the set its list's length (4), back to the host; of a
batch the list of what is cleared (three entries of two pointers and a size a
member) to the device."""
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3])
def test_reset(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cells = I.channel(64, 14)
    h = L.Lattice(cells, 0.8, 0.02) if n == 1 else L.Batch([dict(cells=cells, tau=0.8, u_max=0.02)] * n)
    h.solve(20)
    h2d, d2h = L.transfer_bytes()
    h.reset()
    after = L.transfer_bytes()
    assert after[1] - d2h == 8 * n + 4
    assert after[0] - h2d == (0 if n == 1 else n * 3 * 24)
    h.close()
