"""A reported launch shape can be set: what lbm_step_config says of a solve is
accepted by lbm_set_step_config on the same lattice, on the chip with one, two
and several segments a warp, and gives the same bits."""
import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,channels", [(300, 100, 2), (800, 300, 4), (1000, 500, 4), (1400, 700, 2), (2500, 1200, 4)])
def test_reported_shape_is_accepted(nx, ny, channels):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cells = I.channel_array(nx, ny, channels)
    a, b = (L.Lattice(cells, 0.6, 0.05, residual_every=0) for _ in range(2))
    dp = a.solve(300)["dp"]
    wpb, _, persistent, cpt, stages = a.step_config()
    b.set_step_config(wpb, persistent=persistent, cells_per_thread=cpt, stages=stages)
    assert b.step_config()[2] == persistent
    assert b.solve(300)["dp"] == dp
    assert np.array_equal(a.read(L.FIELD_POPS), b.read(L.FIELD_POPS))
    a.close()
    b.close()
