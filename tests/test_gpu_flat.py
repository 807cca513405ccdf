"""Mixed-precision stage on data that do not vary along some directions: slabs
with constant pencils take one face per pencil (and uniform ones none), next to
slabs that take the general path."""
import dataclasses

import numpy as np
import pytest

from paper_2012_04385_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import learned, mrb  # noqa: E402


def layered(cfg, geo, axes, edge):
    """Two states meeting at a plane across each of `axes`, `edge` cells off the
    block boundary at 1/2 (0: on it, so that stencils cross it only through
    halos), with a moving background; constant along the other axes."""
    X = I.cell_centres(cfg, geo)[:3]
    h = 16 * cfg.dx0 + edge * cfg.dx0 * 0.5 ** cfg.lmax_of(0)
    s = np.zeros(X[0].shape, bool)
    for a in axes:
        s ^= X[a] > h
    out = np.zeros((len(geo), 5, 16, 16, 16))
    for v, (lo, hi) in enumerate([(1.0, 0.4), (0.3, -0.2), (0.1, 0.0), (0.0, 0.25), (1.0, 0.5)]):
        out[:, v] = np.where(s, hi, lo)
    return out


# One perturbed cell per slab sends every slab to the general path.  After n
# stages it has reached at most 3 n cells along x and along y (stencils are
# lines), so beyond those the two runs must agree bit for bit.
@pytest.mark.parametrize("axes", [(0,), (1,), (2,), (0, 2), ()])
@pytest.mark.parametrize("edge", [0, 3])
@pytest.mark.parametrize("recon,flux", [(0, 0), (1, 0), (2, 0), (3, 1), (4, 2), (0, 2)])
def test_constant_slabs_equal_the_general_path(axes, edge, recon, flux):
    cfg = dataclasses.replace(I.periodic_config(base=(2, 2, 2), lmax=0), precision=I.FP32_ACC64, recon=recon, flux=flux,
                              mlp_tau=0.02)
    params = torch.from_numpy(learned.init_params(0)).cuda() if recon == 1 else None
    dt = torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")
    runs = []
    for perturbed in (False, True):
        g = mrb.Context(cfg, 8, mlp_params=params)
        keys, geo = g.list_blocks()
        prim = layered(cfg, geo, axes, edge)
        if perturbed:
            prim[:, 0, 1::4, 8, 8] *= 1.01
        g.set_state(keys, prim)
        g.fill_halos()
        out = [g.compute_rhs().cpu().numpy()]
        for stage in range(2):
            g.fill_halos()
            g.rk_stage(stage, dt)
            out.append(g.get_state(keys).cpu().numpy())
        runs.append(out)
    far = np.maximum(np.abs(np.arange(16) - 8)[:, None], np.abs(np.arange(16) - 8)[None, :])     # [y][x]
    for n, a, b in zip((1, 1, 2), *runs):
        m = np.broadcast_to(far > 3 * n, a.shape)
        assert np.array_equal(a[m].view(np.uint64), b[m].view(np.uint64))
        assert not np.array_equal(a, b)
    if not axes:
        assert not runs[0][0].any()
