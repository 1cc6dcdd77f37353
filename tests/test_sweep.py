"""Sweeps (four time steps in one pass over memory) against the
one-launch-per-phase kernel, bit for bit: tiles at both ends of a row, sizes
around the tile's width, walls inside and at the edges of windows, runs cut
by walls and by the blocks' shares, ports of both schemes, through an
exchange.  LBM_SWEEP=1 takes sweeps wherever they can run (lattices that fit the chip step there first, so LBM_RESIDENT=0 too):
both are read by the library in the process, so the cases run in a child."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
sys.path.insert(0, {root!r})
import numpy as np
import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I
cases = {{
    "narrow": (I.channel(20, 9), 0.8, 0.04, {{}}),
    "one tile": (I.random_blobs(240, 37, 3, density=0.1), 0.7, 0.03, {{}}),
    "tile and one": (I.random_blobs(249, 40, 4, density=0.2), 0.7, 0.03, dict(ports=L.PORTS_ZOU_HE)),
    "two tiles": (I.random_blobs(481, 70, 5, density=0.05), 0.7, 0.03, {{}}),
    "open": (I.channel(1000, 300), 0.6, 0.05, {{}}),
    "channels": (I.channel_array(1501, 403, 7), 0.6, 0.05, {{}}),
    "tree": (I.tree(1501, 751, 4, 46, seed=3), 0.53, 0.0163, {{}}),
    "thin": (I.channel(3000, 2), 0.8, 0.04, {{}}),
}}
for name, (cells, tau, u, kw) in cases.items():
    a = L.Lattice(cells, tau, u, residual_every=20, **kw)
    b = L.Lattice(cells, tau, u, residual_every=20, **kw)
    b.set_step_config(8, persistent=False)
    for i, step in enumerate((lambda h: h.solve(16), lambda h: h.solve(62), lambda h: h.optimize_step(7, 40))):
        n0 = L.kernel_launches()
        ra = step(a)
        n1 = L.kernel_launches()
        rb = step(b)
        assert i != 1 or n1 - n0 < (L.kernel_launches() - n1) // 2, name  # not one launch per phase
        for k in ("dp", "m_in", "residual"):
            assert ra[k] == rb[k], (name, k, ra[k], rb[k])
        assert list(ra["m_out"]) == list(rb["m_out"]), name
        for f in (L.FIELD_MASK, L.FIELD_DRHO, L.FIELD_UX, L.FIELD_UY, L.FIELD_POPS):
            assert np.array_equal(a.read(f), b.read(f)), (name, f)
    a.close()
    b.close()
print("EQUAL")
"""


def test_sweeps_equal_per_phase_kernel():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    env = dict(os.environ, LBM_SWEEP="1", LBM_RESIDENT="0")
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "EQUAL" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]
