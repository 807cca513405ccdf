"""Local time stepping where the coarse levels are blended in time as the
predictions read them: parent boxes that reach over walls of each condition, over
periodic sides, and over stored halos of the parent (jumps two levels deep)."""
import dataclasses

import numpy as np
import pytest

from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402

from test_gpu_parity import close, make_pair, wrap  # noqa: E402

Z, P, S = I.BC_ZERO_GRADIENT, I.BC_PERIODIC, I.BC_SYMMETRY


# FP64 in the oracle's operation order: 1e-11 per cell, the bound of the other
# macro-step comparisons.
@pytest.mark.parametrize("rk", [2, 3])
@pytest.mark.parametrize("bc", [(Z, Z, S, S, P, P), (S, Z, Z, S, S, S)])
def test_lts_macro_step_at_boundaries(bc, rk):
    cfg = dataclasses.replace(I.explosion_config(lmax=3, bc=bc, base_blocks=(2, 1, 1)), lts=1, rk_stages=rk)
    plans = [lambda g: np.ones(len(g), bool), lambda g: g[:, 1] + g[:, 2] <= 1,
             lambda g: (g[:, 0] == 2) & (g[:, 1] == 0) & (g[:, 3] <= 1)]
    o, g = make_pair(cfg, wrap(I.ic_random_smooth), plans, n_slots=2000)
    assert len(set(o.geometry()[:, 0])) >= 2
    o.step(1)
    g.step(1)
    assert g.status() == mrb.MRB_OK
    keys = g.keys()
    assert np.array_equal(keys, o.keys())
    print("values not bit-identical:", close(g.get_state(keys).cpu().numpy(), o.get_state(keys), what="macro step"))
