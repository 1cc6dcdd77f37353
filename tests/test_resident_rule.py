"""Lattices that fit the chip step there by rule (no explicit request): plain,
with the symmetry plane and with the other collision models, one and two
segments per warp, port cells in every segment, both ports in one segment --
against the same lattice on the one-launch-per-phase kernel, bit for bit,
through an exchange."""
import numpy as np
import pytest

import paper_1303_0107_gb300 as L
from paper_1303_0107_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _half(cells):
    """The rows above the middle of a channel: the plane lies below row 0."""
    return np.ascontiguousarray(cells[cells.shape[0] // 2:])


CASES = {
    "one_word": dict(cells=I.channel(20, 9), tau=0.8, u_max=0.04),
    "one_block": dict(cells=I.channel(64, 14), tau=0.9, u_max=0.04, ports=L.PORTS_ZOU_HE),
    "ragged_smagorinsky": dict(cells=I.random_blobs(95, 61, 12, density=0.15), tau=0.7, u_max=0.03,
                               collision=L.COLLIDE_SMAGORINSKY, c_smag=0.1),
    "neumann_regularized": dict(cells=I.random_blobs(130, 70, 5, density=0.1), tau=0.75, u_max=0.03, outlet=1,
                                collision=L.COLLIDE_REGULARIZED),
    "plane": dict(cells=I.config_collector()["cells"], tau=0.53, u_max=0.03, mirror=True),
    "plane_smagorinsky": dict(cells=_half(I.random_blobs(70, 60, 7, density=0.1)), tau=0.7, u_max=0.02, mirror=True,
                              collision=L.COLLIDE_SMAGORINSKY, c_smag=0.12),
    "two_per_warp": dict(cells=I.channel(450, 440), tau=0.6, u_max=0.05),
    "two_per_warp_smagorinsky": dict(cells=I.channel(450, 440), tau=0.6, u_max=0.05,
                                     collision=L.COLLIDE_SMAGORINSKY, c_smag=0.1),
}


def _handle(case, precision):
    return L.Lattice(case["cells"], case["tau"], case["u_max"], precision=precision, residual_every=20,
                     **{k: v for k, v in case.items() if k not in ("cells", "tau", "u_max")})


@pytest.mark.parametrize("precision", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("name", CASES)
def test_rule_equals_per_phase_kernel(name, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    case = CASES[name]
    a, b = _handle(case, precision), _handle(case, precision)
    b.set_step_config(8, persistent=False)
    for step in (lambda h: h.solve(8), lambda h: h.solve(50), lambda h: h.optimize_step(5, 30)):
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
