"""The selector's threshold on the device where its digit passes can go wrong:
keys that differ in one digit only (7, 7, 6, 6 and 6 bits from the top), ties
around the selected rank, infinities, one CTA and several.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2012_04385_gb300 import mrb  # noqa: E402


def _logits(kind, n, rng):
    if kind == "ties":
        return rng.choice(np.float32([-2.5, -0.0, 1.0, 1.5]), n).astype(np.float32)
    if kind == "extremes":
        v = np.float32([-np.inf, -3.4e38, -1e-45, 0.0, 1e-45, 3.4e38, np.inf])
        return rng.choice(v, n).astype(np.float32)
    # one digit of the bit pattern varies, above or below a boundary between digits
    shift, width = {"bits0": (0, 6), "bits5": (5, 3), "bits11": (11, 3), "bits17": (17, 3), "bits24": (24, 3)}[kind]
    base = np.uint32(0x3FB10B29 & ~(((1 << width) - 1) << shift))
    b = base | (rng.integers(0, 1 << width, n).astype(np.uint32) << np.uint32(shift))
    return (b | (rng.integers(0, 2, n).astype(np.uint32) << np.uint32(31))).view(np.float32)


@pytest.mark.parametrize("kind", ["ties", "extremes", "bits0", "bits5", "bits11", "bits17", "bits24"])
@pytest.mark.parametrize("n", [1, 2, 33, 1024, 1025, 70_001])
def test_threshold_equals_the_sorted_order_statistics(kind, n):
    """Against a sort of the label-1 logits.  The order statistics are values of
    the data, so where (m - 1) q is whole the result is that value exactly;
    between two of them it is a + f (b - a) in FP32, whose difference, product
    and sum each round once: 3 * 2^-24 of the larger of |a| and |b - a|, as is
    the rounding of f."""
    rng = np.random.default_rng(n)
    z = _logits(kind, n, rng)
    for y in (np.ones(n, np.uint8), (rng.random(n) < 0.4).astype(np.uint8)):
        s = np.sort(z[y == 1])
        m = len(s)
        for q in (0.0, 1e-3, 0.37, 0.5, 1.0):
            got = mrb.mlp_threshold(torch.from_numpy(z).cuda(), torch.from_numpy(y).cuda(), q)
            if m == 0:
                assert got == 0.0
                continue
            pos = (m - 1) * q
            k = int(pos)
            a, b = s[k], s[min(k + 1, m - 1)]
            f = np.float32(pos - k)
            with np.errstate(all="ignore"):
                d = np.float32(b - a)
                want = np.float32(a + f * d)
            if not np.isfinite(want):
                assert np.array_equal(np.float32(got), want, equal_nan=True), (q, got, want)
            elif f == 0.0 or d == 0.0:
                assert np.float32(got) == want, (q, got, want)
            else:
                scale = max(abs(float(a)), abs(float(d)))
                assert abs(got - float(want)) <= 4 * 2.0 ** -24 * scale + 1.5e-45, (q, got, want)


def test_an_earlier_error_is_left_alone():
    """An error that another call of the process left pending (a device that does
    not exist) neither fails the threshold nor is taken by it."""
    import ctypes

    z = torch.linspace(-1.0, 1.0, 101, device="cuda")
    y = torch.ones(101, dtype=torch.uint8, device="cuda")
    work = torch.empty(256, dtype=torch.int64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    L, out = mrb.lib(), ctypes.c_float()
    torch.cuda.synchronize()
    assert L.cudaSetDevice(9999) != 0
    rc = L.mrb_mlp_threshold(z.data_ptr(), y.data_ptr(), 101, 0.5, work.data_ptr(), ctypes.byref(out), st)
    left = L.cudaGetLastError()
    assert rc == mrb.MRB_OK and out.value == z[50].item() and left != 0
