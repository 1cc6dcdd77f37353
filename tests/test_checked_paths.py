"""The bounds-checked build on the paths that solves take by rule: on the chip
with one, two and several segments a warp, with a symmetry plane and another
collision model, in sweeps, through exchanges -- no violation, and for the BGK
cases the bits of the normal build (the other models leave the compiler free to
contract; another build may do it elsewhere)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import hashlib, sys
sys.path.insert(0, {root!r})
import numpy as np
import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I
half = I.random_blobs(300, 200, 7, density=0.1)[100:]
cases = [
    (I.random_blobs(256, 130, 11, density=0.2), "f32", {{}}),
    (I.channel(450, 440), "f16", {{}}),
    (I.random_blobs(995, 561, 12, density=0.15), "bf16", dict(outlet=1)),
    (np.ascontiguousarray(half), "f32", dict(mirror=True, collision=L.COLLIDE_SMAGORINSKY, c_smag=0.1)),
]
for cells, precision, kw in cases:
    lat = L.Lattice(cells, 0.7, 0.02, precision=precision, residual_every=20, **kw)
    lat.solve(50)
    lat.optimize_step(5, 30)
    for f in (L.FIELD_MASK, L.FIELD_DRHO, L.FIELD_UX, L.FIELD_UY, L.FIELD_POPS):
        print("bits", hashlib.sha256(np.ascontiguousarray(lat.read(f)).tobytes()).hexdigest())
    lat.close()
print("DONE", flush=True)
"""


def _run(**env):
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], env=dict(os.environ, **env),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "DONE" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
    assert "lbm bounds" not in r.stdout, r.stdout[:2000]
    return [line for line in r.stdout.splitlines() if line.startswith("bits")]


def test_no_access_outside():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1303_0107_gb300 import build
    build.build(checked=True)
    want = _run()
    assert len(want) == 20
    assert _run(LBM_CHECKED="1")[:15] == want[:15]
    assert _run(LBM_CHECKED="1", LBM_RESIDENT="0", LBM_SWEEP="1")[:15] == want[:15]  # sweeps, and per phase
