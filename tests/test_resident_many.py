"""Lists beyond two segments per warp on the chip (one copy of the
populations, several pairs of segments per warp) against the
one-launch-per-phase kernel, bit for bit, through exchanges: just above the
smaller kernel's limit, near this one's own, port schemes and outlets, the
symmetry plane, the other collision models, every storage type; and a batch
cut into groups that fit the chip against the same batch as one set."""
import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BLOBS = I.random_blobs(995, 561, 12, density=0.15)  # 17,900 segments
CASES = {
    "channels": dict(cells=I.channel_array(1000, 500, 4), tau=0.6, u_max=0.05),
    "zou_he": dict(cells=I.channel_array(1200, 601, 5), tau=0.6, u_max=0.05, ports=L.PORTS_ZOU_HE),
    "wide": dict(cells=I.channel_array(1411, 700, 2), tau=0.6, u_max=0.05),
    "neumann": dict(cells=BLOBS, tau=0.7, u_max=0.03, outlet=1),
    "smagorinsky": dict(cells=BLOBS, tau=0.7, u_max=0.03, collision=L.COLLIDE_SMAGORINSKY, c_smag=0.1),
    "regularized": dict(cells=BLOBS, tau=0.7, u_max=0.03, collision=L.COLLIDE_REGULARIZED),
    "plane": dict(cells=np.ascontiguousarray(I.channel(900, 1000)[500:]), tau=0.7, u_max=0.03, mirror=True),
    "plane_smagorinsky": dict(cells=np.ascontiguousarray(I.random_blobs(900, 900, 7, density=0.1)[450:]), tau=0.7,
                              u_max=0.02, mirror=True, collision=L.COLLIDE_SMAGORINSKY, c_smag=0.12),
    "narrow": dict(cells=I.channel(40, 7001), tau=0.8, u_max=0.04),
}


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("precision", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("name", CASES)
def test_many_segments_per_block_equal_per_phase_kernel(name, precision):
    _gpu()
    case = CASES[name]
    a, b = (L.Lattice(case["cells"], case["tau"], case["u_max"], precision=precision, residual_every=20,
                      **{k: v for k, v in case.items() if k not in ("cells", "tau", "u_max")}) for _ in range(2))
    b.set_step_config(8, persistent=False)
    assert b.task_counts()[0] > 48 * 146
    for step in (lambda h: h.solve(8), lambda h: h.solve(50), lambda h: h.optimize_step(50, 30)):
        n0 = L.kernel_launches()
        ra = step(a)
        n1 = L.kernel_launches()
        rb = step(b)
        assert n1 - n0 < L.kernel_launches() - n1  # one launch for the steps, not one per phase
        assert ra["dp"] == rb["dp"] and ra["m_in"] == rb["m_in"] and ra["residual"] == rb["residual"]
        assert list(ra["m_out"]) == list(rb["m_out"])
        for f in (L.FIELD_MASK, L.FIELD_DRHO, L.FIELD_UX, L.FIELD_UY, L.FIELD_POPS):
            assert np.array_equal(a.read(f), b.read(f)), f
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["f32", "bf16"])
def test_groups_that_fit_the_chip_equal_the_batch_as_one_set(precision):
    _gpu()
    cands = I.config_candidates(48, base_seed=3)
    members = [dict(cells=c["cells"], tau=c["tau"], u_max=c["u_max"] * (0.9 + 0.004 * i)) for i, c in enumerate(cands)]
    a, b = (L.Batch(members, precision=precision, residual_every=20) for _ in range(2))
    b.set_step_config(8, persistent=False)
    n = [max(1, int((c["cells"] == 0).sum()) // 300) for c in cands]
    # the groups are built at 256 steps; 8 steps run as one set again, 40 in groups
    for step in (lambda h: h.solve(300), lambda h: h.optimize_step(n, 40), lambda h: h.solve(8),
                 lambda h: h.optimize_step(n, 8), lambda h: h.solve(40)):
        ra, rb = step(a), step(b)
        assert [x["dp"] for x in ra] == [x["dp"] for x in rb]
        assert [x["residual"] for x in ra] == [x["residual"] for x in rb]
    assert a.step_groups() > 1 and b.step_groups() == 1
    for i in range(len(members)):
        for f in (L.FIELD_MASK, L.FIELD_POPS, L.FIELD_UX, L.FIELD_DRHO):
            assert np.array_equal(a.read(i, f), b.read(i, f)), (i, f)
    a.close()
    b.close()
