"""Which buffers the copy kernels take: memory of the device that one
allocation holds from the first byte to the last.  Anything else goes to the
runtime's copies, which check it themselves (nothing is accessed here)."""
import ctypes

import numpy as np
import pytest

import paper_1303_0107_gb300 as L

pytestmark = pytest.mark.gpu


def test_only_whole_buffers_of_one_allocation():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    inside = L.load_library().lbm_debug_on_device
    n = 64 << 20  # beyond what the caching allocator splits
    buf = torch.zeros(n, dtype=torch.uint8, device="cuda")
    p = buf.data_ptr()
    assert inside(p, n) == 1 and inside(p, 1) == 1 and inside(p + 3, n - 3) == 1 and inside(p + n - 1, 1) == 1
    assert inside(p, 1 << 40) == 0 and inside(p + n - 1, 1 << 40) == 0 and inside(p, (1 << 64) - 1) == 0
    host = np.zeros(64, np.uint8)
    assert inside(host.ctypes.data, 64) == 0
    pinned = torch.zeros(64, dtype=torch.uint8).pin_memory()
    assert inside(pinned.data_ptr(), 64) == 0
    assert inside(ctypes.c_void_p(None), 1) == 0
