"""Bounded device waits that give up, forced by the test hook (no device
fault: a tag or a row that is taken as late): the solve reports
LBM_ERR_TIMEOUT, and after a reset the same handle gives its reference
result again."""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_a_list_of_several_pairs_per_warp():
    lat = L.Lattice(I.channel_array(1000, 500, 4), 0.6, 0.05, residual_every=0)
    assert lat.task_counts()[0] > 48 * 146
    dp = lat.solve(100)["dp"]
    pops = lat.read(L.FIELD_POPS)
    lat.reset()
    L.lib.debug_barrier_timeout(True)
    try:
        with pytest.raises(L.LbmError) as e:
            lat.solve(100)
        assert e.value.status == 6  # LBM_ERR_TIMEOUT
    finally:
        L.lib.debug_barrier_timeout(False)
    lat.reset()
    assert lat.solve(100)["dp"] == dp
    assert np.array_equal(lat.read(L.FIELD_POPS), pops)
    lat.close()


SWEEP = """
import sys
sys.path.insert(0, {root!r})
import numpy as np
import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I
for cells in (I.channel(20, 9), I.channel(1000, 300), I.random_blobs(1501, 751, 3, density=0.05)):
    lat = L.Lattice(cells, 0.7, 0.03, residual_every=0)
    dp = lat.solve(50)["dp"]
    pops = lat.read(L.FIELD_POPS)
    for _ in range(2):
        lat.reset()
        L.lib.debug_barrier_timeout(True)
        try:
            lat.solve(50)
            print("NO TIMEOUT", cells.shape)
        except L.LbmError as e:
            assert e.status == 6, e
        L.lib.debug_barrier_timeout(False)
        lat.reset()
        assert lat.solve(50)["dp"] == dp and np.array_equal(lat.read(L.FIELD_POPS), pops)
    lat.close()
print("DONE")
"""


def test_sweeps():
    env = dict(os.environ, LBM_SWEEP="1", LBM_RESIDENT="0")
    r = subprocess.run([sys.executable, "-c", SWEEP.format(root=ROOT)], env=env, capture_output=True, text=True,
                       timeout=200)
    assert r.returncode == 0 and "DONE" in r.stdout and "NO TIMEOUT" not in r.stdout, r.stdout + r.stderr[-2000:]
