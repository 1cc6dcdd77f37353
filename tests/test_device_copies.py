"""States and fields through device buffers against the same through host
buffers, byte for byte: row lengths and buffer addresses of every alignment,
single rows of a warp's piece and several, every storage type, two and three
dimensions; and the reset of a batch against fresh handles."""
import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _on_device(torch, nbytes, shift):
    return torch.full((nbytes + 64,), 0xA5, dtype=torch.uint8, device="cuda")[shift:shift + nbytes]


def _check(torch, lat, fields, pops, shift):
    for f in fields:
        host = np.ascontiguousarray(lat.read(f))
        buf = _on_device(torch, host.nbytes, shift)
        lat.read(f, out=buf)
        assert np.array_equal(buf.cpu().numpy(), host.view(np.uint8).reshape(-1)), f
        base = buf.storage_offset()
        around = torch.as_strided(buf, (host.nbytes + 64,), (1,), 0).cpu().numpy()
        assert (around[:base] == 0xA5).all() and (around[base + host.nbytes:] == 0xA5).all()  # nothing beside it
    host = np.ascontiguousarray(lat.read(pops))
    rng = np.random.default_rng(3)
    state = rng.integers(0, 255, host.nbytes, dtype=np.uint8)
    buf = _on_device(torch, host.nbytes, shift)
    buf.copy_(torch.from_numpy(state))
    lat.load_state(buf)
    assert np.array_equal(np.ascontiguousarray(lat.read(pops)).view(np.uint8).reshape(-1), state)


@pytest.mark.parametrize("precision", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny,shift", [(20, 9, 0), (33, 12, 4), (513, 40, 2), (1027, 30, 8), (640, 64, 16)])
def test_planes_2d(nx, ny, shift, precision):
    torch = _torch()
    if precision == "f32" and shift % 4:
        shift = 4
    lat = L.Lattice(I.channel(nx, ny), 0.8, 0.04, precision=precision, residual_every=0)
    lat.solve(10)
    _check(torch, lat, (L.FIELD_MASK, L.FIELD_RHO, L.FIELD_DRHO, L.FIELD_UX, L.FIELD_UY, L.FIELD_POPS), L.FIELD_POPS,
           shift)
    lat.close()


@pytest.mark.parametrize("precision", ["f32", "bf16"])
@pytest.mark.parametrize("n,shift", [(12, 0), (13, 4), (37, 8)])
def test_planes_3d(n, shift, precision):
    torch = _torch()
    cells = I.duct3d(2 * n + 1, n + 1, n)
    lat = L.Lattice3(cells, 0.8, 0.02, precision=precision)
    lat.solve(4)
    _check(torch, lat, (L.FIELD3_MASK, L.FIELD3_UX, L.FIELD3_POPS), L.FIELD3_POPS, shift)
    lat.close()


def test_batch_reset_equals_fresh_handles():
    _torch()
    cands = I.config_candidates(6, base_seed=9)
    members = [dict(cells=c["cells"], tau=c["tau"], u_max=c["u_max"]) for c in cands] + [
        dict(cells=I.channel(21, 9), tau=0.8, u_max=0.02)]
    a, b = L.Batch(members, residual_every=0), L.Batch(members, residual_every=0)
    a.solve(60)
    a.optimize_step([5] * len(members), 20)
    a.reset()
    fields = (L.FIELD_MASK, L.FIELD_POPS, L.FIELD_DRHO, L.FIELD_UX, L.FIELD_UY)
    for run in (lambda x: None, lambda x: x.solve(20)):
        ra, rb = run(a), run(b)
        assert ra is None or [r["dp"] for r in ra] == [r["dp"] for r in rb]
        for i in range(len(members)):
            for f in fields:
                assert np.array_equal(a.read(i, f), b.read(i, f)), (i, f)
    a.close()
    b.close()
