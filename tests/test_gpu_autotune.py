"""The autotuner times what its parameters shape: complete halo fills for the
copies (a single level, whose stages fill nothing, has no other)."""
import pytest

from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402


def test_copies_are_timed_on_complete_fills():
    """Counted in launches: one right-hand side is one stage launch here, the seven
    timed stage shapes and the time step before them are known, and what is left
    holds the default's and three shapes' fills."""
    cfg = I.explosion_config(lmax=0, precision=I.FP32_ACC64)
    g = mrb.Context(cfg, 8)
    keys, geo = g.list_blocks()
    g.set_state(keys, I.ic_explosion(cfg, geo))

    def launches(f):
        g.profile(True)
        f()
        n = g.profile_read()[2]
        g.profile(False)
        return n

    fill, reps = launches(g.fill_halos), 2
    assert fill > 0 and launches(g.compute_rhs) == 1
    n = launches(lambda: g.autotune(reps=reps))
    assert n - (1 + 7 * (reps + 1)) == 4 * (reps + 1) * fill
    g.close()
