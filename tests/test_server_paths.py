"""The request loop's two forms of a tick -- on the chip where the set fits,
cell tasks per phase where it does not -- and what decides between them: the
results are those of each request alone, bit for bit."""
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


def _serve(reqs, precision="f32", **cfg):
    """reqs: (cells, tau, u_max, steps, iterations, swapped) -> results by number, statistics."""
    srv = L.Server(precision=precision, **cfg)
    for k, (cells, tau, u, steps, n_iter, n_swap) in enumerate(reqs):
        srv.submit(k, cells, tau, u, steps, n_iter=n_iter, n_swap=n_swap, keep_fields=True)
    srv.wait_idle(300)
    done = {}
    while len(done) < len(reqs):
        for d in srv.poll(64):
            done[d["tag"]] = d
    stats = srv.stats()
    srv.close()
    return done, stats


def _check_alone(reqs, done, precision="f32"):
    for k, (cells, tau, u, steps, n_iter, n_swap) in enumerate(reqs):
        h = L.Lattice(cells, tau, u, precision=precision, residual_every=0)
        h.set_step_config(8, persistent=False)
        first = last = h.solve(steps)
        for _ in range(n_iter):
            last = h.optimize_step(n_swap, steps)
        assert done[k]["status"] == 0
        assert done[k]["dp_first"] == first["dp"] and done[k]["last"]["dp"] == last["dp"], k
        for name, f in (("mask", L.FIELD_MASK), ("drho", L.FIELD_DRHO), ("ux", L.FIELD_UX), ("uy", L.FIELD_UY)):
            assert np.array_equal(done[k]["fields"][name], h.read(f)), (k, name)
        h.close()


def test_device_memory_stays_within_the_budget():
    """Small lattices: their halo words would take more than all they are charged."""
    t = I.config_t_junction()
    reqs = [(t["cells"], t["tau"], t["u_max"], 6000 + 200 * k, 0, 0) for k in range(6)]
    budget = 6 * L.Server.footprint(128, 64, 0)
    done, stats = _serve(reqs, hbm_budget_bytes=budget, max_tick_steps=100)
    assert stats["peak_active"] >= 2
    assert 0 < stats["peak_device_bytes"] <= budget
    _check_alone(reqs, done)


@pytest.mark.parametrize("precision", ["f32", "bf16"])
def test_a_set_beyond_the_chip_and_back(precision):
    """Requests of 20,160, 10,080 and 5,040 segments: alone or two small ones
    fit the chip (18,240), the three together and the largest do not, so ticks
    change between the two forms within one run, exchanges in both."""
    reqs = [(I.channel(1000, 630), 0.7, 0.02, 6000, 0, 0),
            (I.channel(1000, 315), 0.8, 0.02, 8000, 2, 40),
            (np.ascontiguousarray(I.random_blobs(500, 317, 5, density=0.1)), 0.75, 0.02, 9000, 1, 30)]
    srv_calls = L.kernel_launches()
    done, stats = _serve(reqs, precision=precision, max_tick_steps=400)
    steps = sum(s * (1 + n) for _, _, _, s, n, _ in reqs)
    assert stats["peak_active"] == 3
    # between one launch a step (all per phase) and one a tick (all on the chip)
    launches = L.kernel_launches() - srv_calls
    assert 6000 <= launches < steps
    _check_alone(reqs, done, precision)
