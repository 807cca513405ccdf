"""The first call on a context does not depend on what its device memory held
before: a time step taken from small allocations that were filled and freed."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402


def _dirty(word):
    """Fill small device allocations with a 64-bit word and free all but a few,
    which keep the memory from going back to the system."""
    cu = ctypes.CDLL("libcuda.so.1")
    blocks = []
    for k in range(256):
        p = ctypes.c_uint64()
        n = 64 << (k % 4)
        assert cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(n)) == 0
        host = np.full(n // 8, word, dtype=np.uint64)
        assert cu.cuMemcpyHtoD_v2(p, ctypes.c_void_p(host.ctypes.data), ctypes.c_size_t(n)) == 0
        blocks.append(p)
    for k, p in enumerate(blocks):
        if k % 16:
            assert cu.cuMemFree_v2(p) == 0
    return [blocks[k] for k in range(0, len(blocks), 16)], cu


@pytest.mark.parametrize("first", ["cfl_dt", "step"])
def test_first_call_on_dirty_memory(first):
    """FP64 against the oracle, bit for bit.  The word is the address of a buffer
    of the test, so that a pointer read from dirty memory leads there: its values
    stay as they were."""
    own = torch.full((4096,), -1.0, dtype=torch.float64, device="cuda")
    cfg = I.sod_config()
    o = oracle.Oracle(cfg)
    prim = I.ic_sod(cfg, o.geometry())
    o.set_state(o.keys(), prim)
    dt = o.cfl_dt()
    o.step(2)
    kept, cu = _dirty(own.data_ptr())
    g = mrb.Context(cfg, 16)
    g.set_state(o.keys(), prim)
    if first == "cfl_dt":
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        g.cfl_dt(out)
        assert np.array_equal(out.cpu().numpy(), dt)
    g.step(2)
    assert np.array_equal(g.get_state(o.keys()).cpu().numpy(), o.get_state())
    assert g.status() == mrb.MRB_OK
    assert bool((own == -1.0).all())
    g.close()
    for p in kept:
        assert cu.cuMemFree_v2(p) == 0
