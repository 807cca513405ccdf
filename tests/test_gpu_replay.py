"""Steps replayed from graphs that were captured on another tree: the same states
as with graphs captured on the present one.  The trees differ by less than a
factor of two in every count, so that the graphs are kept, and lie on both sides
of the thin slabs' limit, so that a fresh capture would choose the other kernel."""
import numpy as np
import pytest

from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402


def _counts(g):
    return [g.n_blocks(level, leaves) for level in (-1, 0, 1, 2) for leaves in (False, True)]


def _run(cfg, grow, recapture):
    g = mrb.Context(cfg, 100)
    keys, geo = g.list_blocks()
    g.set_state(keys, I.ic_random_smooth(cfg, geo))
    g.refine_keys(keys[geo[:, 1] == 0])
    if not grow:                   # one level-1 block refined: the step coarsens it again
        g.refine_keys(g.keys(level=1)[5:6])
    keys, geo = g.list_blocks()
    g.set_state(keys, I.ic_random_smooth(cfg, geo))
    g.mr_project()
    leaves = [g.n_leaves()]
    before = _counts(g)
    g.step(1)                      # captured here
    if grow:
        g.refine_keys(g.keys(level=0)[:1])
    leaves.append(g.n_leaves())
    # (graphs are captured again when a count above 32 has doubled or halved)
    assert all(max(a, b) <= 32 or max(a, b) <= 2 * min(a, b) for a, b in zip(before, _counts(g)))
    if recapture:
        g.set_tune(g.get_tune())
    g.step(2)
    assert g.status() == mrb.MRB_OK and g.n_leaves() == leaves[1]
    out = g.get_state(g.keys(leaves_only=False)).cpu().numpy()
    g.close()
    return leaves, out


@pytest.mark.parametrize("grow", [True, False], ids=["grown", "shrunk"])
@pytest.mark.parametrize("precision", [I.FP64, I.FP32_ACC64])
def test_replayed_graphs_of_another_tree(precision, grow):
    cfg = I.explosion_config(lmax=2, precision=precision, eps=1e9)
    runs = [_run(cfg, grow, recapture) for recapture in (False, True)]
    few, many = sorted(runs[0][0])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert runs[0][0] == runs[1][0] and 8 * few <= 2 * sms < 8 * many
    assert np.array_equal(runs[0][1].view(np.uint64), runs[1][1].view(np.uint64))
