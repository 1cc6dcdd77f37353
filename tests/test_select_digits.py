"""The selection where its digit search ends early, late or in the index
digits, with more candidates than a block takes at once, against the oracle,
exactly: all scores equal, two or a few values, scores that differ in their
last bits, spread over the whole exponent range."""
import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FIELDS = {
    "zero": lambda r, s: np.zeros(s),
    "two values": lambda r, s: r.choice([0.01, 0.02], s),
    "few values": lambda r, s: np.round(0.05 * r.standard_normal(s) * 40) / 40,
    "last bits": lambda r, s: 0.03 * (1 + r.integers(0, 5, s) * 2.0 ** -23),
    "spread": lambda r, s: 10.0 ** r.uniform(-18, 2, s),
}


@pytest.mark.parametrize("name", FIELDS)
def test_selection_equals_oracle(ora, name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny = 421, 213
    cells = I.random_blobs(nx, ny, 4, density=0.35)
    rng = np.random.default_rng(8)
    ux, uy = (FIELDS[name](rng, (ny, nx)).astype(np.float32) for _ in range(2))
    drho = np.zeros((ny, nx), np.float32)
    lat = L.Lattice(cells, 0.7, 0.02)
    p = ora.make_params(nx, ny, 0.7, 1.0, 0.02)
    cand, score = ora.scores(p, cells, 1.0 + drho.astype(np.float64), ux.astype(np.float64), uy.astype(np.float64))
    most = len(lat.select_swaps(drho, ux, uy, 10 ** 6)[0])
    for n in (1, 2, 33, most // 2, most - 1, most):
        fi, si = lat.select_swaps(drho, ux, uy, n)
        fo, so = ora.select(p, cand, score, n)
        assert np.array_equal(fi, fo) and np.array_equal(si, so), n
    lat.close()
