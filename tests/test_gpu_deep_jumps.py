"""Resolution jumps of several levels: a corner refined step by step beside leaves
of level 0 and 1 (walls between, and periodic sides that bring it beside its own
siblings), and a whole side three levels finer."""
import dataclasses

import numpy as np
import pytest

from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402

from test_gpu_parity import make_pair, wrap  # noqa: E402

P, S = I.BC_PERIODIC, I.BC_SYMMETRY


def _plans(shape, levels):
    def corner(l):
        return lambda g: (g[:, 0] == l) & (g[:, 1] == 1 << l) & (g[:, 2] == 0) & (g[:, 3] == 0)

    def side(l):
        return lambda g: (g[:, 0] == l) & (g[:, 1] == 1 << l)

    return [(corner if shape == "corner" else side)(l) for l in range(levels)]


# FP64 in the oracle's operation order: bit for bit.
@pytest.mark.parametrize("bc", [(P,) * 6, (S,) * 6], ids=["periodic", "walls"])
@pytest.mark.parametrize("shape,levels,lts", [("corner", 2, 0), ("corner", 5, 0), ("side", 3, 0), ("corner", 4, 1)])
def test_deep_jumps_against_oracle(shape, levels, lts, bc):
    cfg = dataclasses.replace(I.explosion_config(lmax=levels, base_blocks=(2, 1, 1), bc=bc, eps=1e9), lts=lts)
    o, g = make_pair(cfg, wrap(I.ic_random_smooth), _plans(shape, levels), n_slots=400)
    assert {0, 1, levels} <= set(o.geometry()[:, 0])
    if not lts:
        o.fill_halos()
        g.fill_halos()
        assert np.array_equal(g.compute_rhs().cpu().numpy(), o.compute_rhs())
    o.step(1)
    g.step(1)
    assert g.status() == mrb.MRB_OK and np.array_equal(g.keys(), o.keys())
    assert np.array_equal(g.get_state().cpu().numpy(), o.get_state())
