"""Refinement by the caller's own tags without a halo fill before it: the same
tree and states as with one, whatever moved the state or the tree on since the
halos were last stored."""

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


def _cfg(**kw):
    # (details stay below this eps: steps keep the tree, of levels 0 and 1)
    return I.explosion_config(lmax=2, base_blocks=(2, 1, 2), bc=(Z, S, P, P, S, Z), eps=1e9, **kw)


def _start(cfg):
    g = mrb.Context(cfg, 300)
    keys, geo = g.list_blocks()
    g.set_state(keys, I.ic_random_smooth(cfg, geo))
    g.fill_halos()
    g.remesh((geo[:, 1] == geo[:, 3]).astype(np.int8))
    keys, geo = g.list_blocks()
    g.set_state(keys, I.ic_random_smooth(cfg, geo))
    g.mr_project()
    g.fill_halos()
    return g


def _tags(geo):
    return ((geo[:, 0] == 1) & ((geo[:, 1] + geo[:, 2]) % 2 == 0) | (geo[:, 0] == 0) & (geo[:, 1] == 0)).astype(np.int8)


def _move(g, what):
    keys, geo = g.list_blocks()
    if what == "step":
        g.step(2)
    elif what == "stage":
        g.rk_stage(0, torch.full((1,), 1e-3, dtype=torch.float64, device="cuda"))
        g.mr_project()
    elif what == "state":
        prim = I.ic_random_smooth(g.cfg, geo)
        prim[:, 0] *= 1.25
        g.set_state(keys, prim)
        g.mr_project()
    else:
        g.remesh(((geo[:, 0] == 1) & (geo[:, 1] == 1)).astype(np.int8))


@pytest.mark.parametrize("what", ["step", "stage", "state", "tree"])
@pytest.mark.parametrize("kw", [dict(), dict(precision=I.FP32_ACC64), dict(lts=1), dict(precision=I.FP32_ACC64, mu=1e-3)],
                         ids=["fp64", "fp32", "lts", "viscous"])
def test_refinement_without_a_fill(kw, what):
    out = []
    for fill in (False, True):
        g = _start(_cfg(**kw))
        _move(g, what)
        if fill:
            g.fill_halos()
        g.remesh(_tags(g.geometry()))
        assert g.status() == mrb.MRB_OK
        nodes = g.keys(leaves_only=False)
        out.append((nodes, g.get_state(nodes).cpu().numpy()))
        g.close()
    assert out[0][0].size > 30 and np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1].view(np.uint64), out[1][1].view(np.uint64))


def test_refinement_after_steps_against_oracle():
    """FP64, bit for bit."""
    cfg = _cfg()
    g, o = _start(cfg), oracle.Oracle(cfg)
    o.set_state(o.keys(), I.ic_random_smooth(cfg, o.geometry()))
    o.fill_halos()
    geo = o.geometry()
    o.remesh((geo[:, 1] == geo[:, 3]).astype(np.int8))
    o.set_state(o.keys(), I.ic_random_smooth(cfg, o.geometry()))
    o.project()
    g.step(2)
    o.step(2)
    assert np.array_equal(g.keys(), o.keys())
    o.fill_halos()
    o.remesh(_tags(o.geometry()))
    g.remesh(_tags(g.geometry()))
    assert np.array_equal(g.keys(), o.keys())
    assert np.array_equal(g.get_state().cpu().numpy(), o.get_state())


READERS = {
    "state": lambda g: g.get_state(with_halo=True),
    "rhs": lambda g: g.compute_rhs(),
    "tags": lambda g: g.mr_predict_and_tag()[1],
    "census": lambda g: torch.from_numpy(g.flux_census().astype(np.int64)),
    "samples": lambda g: g.face_samples(stride=7)[0],
}


def _stage(g):
    g.rk_stage(0, torch.full((1,), 1e-3, dtype=torch.float64, device="cuda"))
    return g.get_state()


@pytest.mark.parametrize("what", ["step", "stage"])
@pytest.mark.parametrize("kw", [dict(), dict(precision=I.FP32_ACC64), dict(precision=I.FP32_ACC64, mu=1e-3)],
                         ids=["fp64", "fp32", "viscous"])
def test_calls_that_read_halos_after_a_stage_or_step(kw, what):
    """Their results do not depend on a halo fill before them (FP64 stages leave
    scratch in the stored halos)."""
    for name, read in list(READERS.items()) + [("next stage", _stage)]:
        if name == "samples" and "precision" not in kw:
            continue
        out = []
        for fill in (False, True):
            g = _start(_cfg(**kw))
            _move(g, what)
            if fill:
                g.fill_halos()
            out.append(read(g).cpu().numpy())
            assert g.status() == mrb.MRB_OK
            g.close()
        assert np.array_equal(out[0].view(np.uint8), out[1].view(np.uint8)), name


@pytest.mark.parametrize("precision", [I.FP64, I.FP32_ACC64])
def test_stored_halos_after_a_refinement_without_a_fill(precision):
    """Halos of one state throughout: those of a complete fill after the remesh."""
    out = []
    for fill in (False, True):
        g = _start(_cfg(precision=precision))
        _move(g, "state")
        g.remesh(_tags(g.geometry()))
        if fill:
            g.fill_halos()
        out.append(g.get_state(with_halo=True).cpu().numpy())
        g.close()
    assert np.array_equal(out[0].view(np.uint64), out[1].view(np.uint64))
