"""Totals over blocks at the sizes where the reduction changes shape: fewer blocks
than a warp has lanes, one lane more than the rest, and around the four blocks a
lane takes at once."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402


@pytest.mark.parametrize("n", [1, 31, 32, 33, 96, 97, 127, 128, 129, 300])
def test_block_totals_against_exact_sums(n):
    """A cell passes 16 additions in its thread, 5 + 8 in its block, the scaling by
    dx^3 (2 roundings), n / 32 in its lane and 5 across lanes: that many half-ulps
    of the sum of magnitudes bound the error."""
    rng = np.random.default_rng(n)
    blocks = rng.normal(size=(n, 5, 16, 16, 16))
    lv = rng.integers(0, 4, n).astype(np.int32)
    out = torch.empty(5, dtype=torch.float64, device="cuda")
    dev, levels = torch.from_numpy(blocks).cuda(), torch.from_numpy(lv).cuda()
    assert mrb.lib().mrb_block_sums_noalloc(dev.data_ptr(), n, levels.data_ptr(), 1.0 / 32, torch.cuda.current_stream().cuda_stream,
                                            out.data_ptr()) == mrb.MRB_OK
    got = out.cpu().numpy()
    w = np.ldexp(1.0, -3 * (lv + 5))
    for v in range(5):
        x = (blocks[:, v].reshape(n, -1) * w[:, None]).ravel()        # (powers of two: exact)
        assert abs(got[v] - math.fsum(x)) <= (16 + 13 + 2 + n // 32 + 1 + 5) * 2.0 ** -53 * np.abs(x).sum()
