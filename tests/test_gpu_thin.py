"""Slabs of two planes (few leaves) against slabs of four, bit for bit: the same
blocks in a run of one instance and in one of eight, which has too many leaves
for thin slabs."""
import dataclasses

import numpy as np
import pytest

from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402

Z, P, S = I.BC_ZERO_GRADIENT, I.BC_PERIODIC, I.BC_SYMMETRY
VARIANTS = [dict(recon=r, flux=f) for r in (I.RECON_WENO, I.RECON_LINEAR, I.RECON_TENO, I.RECON_WENOAO)
            for f in (I.FLUX_ROE, I.FLUX_LLF, I.FLUX_HLLC)] + [dict(mu=1e-3), dict(gravity=(0.1, -0.2, 0.3)), dict(rk_stages=2)]


def _run(cfg, prim, n):
    g = mrb.Context(dataclasses.replace(cfg, n_instances=n, lmax=(0,) * n), 8 * n)
    keys, _ = g.list_blocks()
    assert len(keys) == 8 * n
    g.set_state(keys, np.concatenate([prim] * n))
    g.fill_halos()
    out = [g.compute_rhs().cpu().numpy()[:8]]
    dt = torch.full((n,), 1e-3, dtype=torch.float64, device="cuda")
    for stage in range(cfg.rk_stages):
        g.fill_halos()
        g.rk_stage(stage, dt)
        out.append(g.get_state(keys).cpu().numpy()[:8])
    assert g.status() == mrb.MRB_OK
    return out


@pytest.mark.parametrize("data", ["rough", "flat in z", "flat in x and z", "flat but one plane"])
@pytest.mark.parametrize("kw", VARIANTS, ids=lambda kw: "-".join(f"{k}{v}" for k, v in kw.items()))
def test_thin_slabs_equal_slabs_of_four(kw, data):
    cfg = I.explosion_config(lmax=0, bc=(Z, S, P, P, S, Z), precision=I.FP32_ACC64, **kw)
    prim = I.random_states(8, seed=11, rho=(1.0, 1.5), p=(1.0, 1.5), vmax=0.3)
    if data != "rough":
        prim[:] = prim[:1, :, 5:6]
    if data == "flat in x and z":
        prim[:] = prim[..., 7:8]
    if data == "flat but one plane":
        prim[3, 0, 9] *= 1.01
    for a, b in zip(_run(cfg, prim, 1), _run(cfg, prim, 8)):
        assert np.array_equal(a.view(np.uint64), b.view(np.uint64))


def test_replayed_steps_of_a_tree_that_grew():
    """Graphs captured on 8 leaves, then a tree of hundreds: the same states as
    with graphs captured on that tree."""
    cfg = I.explosion_config(lmax=2, precision=I.FP32_ACC64, recon=I.RECON_WENO)
    states = []
    for recapture in (False, True):
        g = mrb.Context(cfg, 700)
        keys, geo = g.list_blocks()
        g.set_state(keys, I.ic_explosion(cfg, geo))
        g.step(1)
        g.set_state(g.keys(), I.ic_explosion(cfg, g.list_blocks()[1]))
        mrb.init_tree(g, I.ic_explosion)
        if recapture:
            g.set_tune(g.get_tune())
        g.step(2)
        assert g.status() == mrb.MRB_OK
        states.append((g.keys(), g.get_state(g.keys()).cpu().numpy()))
    assert len(states[0][0]) > 64 and np.array_equal(states[0][0], states[1][0])
    assert np.array_equal(states[0][1].view(np.uint64), states[1][1].view(np.uint64))
