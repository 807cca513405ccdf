"""Ghost cells of the stage kernels, which map boundary cells themselves: every
pair of conditions, blocks that touch both sides of an axis, and jumps at a wall."""
import numpy as np
import pytest

import oracle
from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402

Z, P, S = I.BC_ZERO_GRADIENT, I.BC_PERIODIC, I.BC_SYMMETRY


# FP64: bit for bit.  Mixed precision: 2e-5 of each variable's largest |L|, the
# bound of its parity tests on the same random states.
@pytest.mark.parametrize("bc", [(Z, Z, S, S, P, P), (S, Z, P, P, Z, S), (P, P, Z, S, S, S)])
@pytest.mark.parametrize("base,refine", [((1, 2, 1), False), ((2, 1, 2), True)])
def test_rhs_at_boundaries(bc, base, refine):
    for precision in (I.FP64, I.FP32_ACC64):
        cfg = I.explosion_config(lmax=2, bc=bc, base_blocks=base, precision=precision)
        o, g = oracle.Oracle(I.explosion_config(lmax=2, bc=bc, base_blocks=base)), mrb.Context(cfg, 300)
        for plan in (None, lambda geo: np.ones(len(geo), bool), lambda geo: geo[:, 1] % 2 == 0)[: 3 if refine else 1]:
            if plan is not None:
                mask = plan(o.geometry()).astype(np.int8)
                for q in (o, g):
                    q.fill_halos()
                    q.remesh(mask)
            keys, geo = o.keys(), o.geometry()
            prim = I.random_states(len(keys), seed=5, rho=(1.0, 1.5), p=(1.0, 1.5), vmax=0.3)
            o.set_state(keys, prim)
            g.set_state(keys, prim)
        o.project()
        g.mr_project()
        o.fill_halos()
        g.fill_halos()
        ref, got = o.compute_rhs(), g.compute_rhs().cpu().numpy()
        if precision == I.FP64:
            assert np.array_equal(got, ref)
            o.step(2)
            g.step(2)
            assert np.array_equal(o.keys(), g.keys())
            assert np.array_equal(o.get_state(), g.get_state().cpu().numpy())
        else:
            scale = np.abs(ref).max(axis=(0, 2, 3, 4), keepdims=True)
            assert (np.abs(got - ref) < 2e-5 * scale).all()
