"""The eigensolver's FP64 helpers: the integer warp sum against the exact sum of its values, the square root and
reciprocals against CUDA's.

Bound of the sum: a value is cut at 52 + 25 (one value per lane) or 52 + 19 binades (four) below the largest one, which 32
or 128 values add up to 2^-72 or 2^-64 of the largest value; half of that again for the alignment of the limbs,
and one rounding of the result.
Bound of the roots and reciprocals (normal operands and results): the result's rounding is 2^-53 relative, that of
the product x y inside the square root leaves another 2^-54, and the series' remainders are below 2^-56.  CUDA's
square root and division are correctly rounded (2^-53), the reciprocal root formed from both is within 1.5 x 2^-52:
2^-51 covers each comparison.
"""
import ctypes
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2405_08971_gb300 import binding  # noqa: E402


def rows_of(kind, n):
    rng = np.random.default_rng(n)
    x = rng.standard_normal((64, n))
    if kind == "spread":                       # exponents over the whole range of the alignment and far below it
        x *= 2.0 ** rng.integers(-150, 1, x.shape)
    if kind == "cancelling":                   # large terms cancel; the rest lies 0 .. 400 binades below
        x *= 2.0 ** -np.arange(0, 640, 10)[:, None]
        x[:, 0], x[:, 1] = 1.0, -1.0
    if kind == "far":                          # 1, -1 and terms that lie below every limb
        x = np.full((64, n), 1e-100)
        x[:, 0], x[:, 1] = 1.0, -1.0
    if kind == "ends":
        x *= 2.0 ** np.linspace(-900, 900, 64)[:, None]
    return x


@pytest.mark.parametrize("kind", ["normal", "spread", "cancelling", "far", "ends"])
@pytest.mark.parametrize("nv,floor", [(1, 1.5 * 2.0 ** -72), (4, 1.5 * 2.0 ** -64)])
def test_warp_sum(kind, nv, floor):
    x = rows_of(kind, 32 * nv)
    t = torch.as_tensor(x, device="cuda")
    out = torch.empty(len(x), dtype=torch.float64, device="cuda")
    rc = binding.lib().cakf_probe_warp_sum(nv, len(x), ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(out.data_ptr()))
    assert rc == 0
    got = out.cpu().numpy()
    for i in range(len(x)):
        exact = math.fsum(x[i])
        assert abs(got[i] - exact) <= 2.0 ** -52 * abs(exact) + floor * np.max(np.abs(x[i])), (i, got[i], exact)


def test_roots_and_reciprocals():
    rng = np.random.default_rng(3)
    n = 200000
    x = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-1021, 1022, n) * rng.choice([-1.0, 1.0], n)
    x[:4] = 1.0, 2.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0)
    x[4:2000] = 1.0 + np.arange(1996) * 2.0 ** -52                    # around a power of two
    x[2000:4000] = rng.integers(1, 2000, 2000).astype(np.float64) ** 2    # exact roots
    t = torch.as_tensor(x, device="cuda")
    sq, rs, rc = (torch.empty_like(t) for _ in range(3))
    assert binding.lib().cakf_probe_roots(n, *(ctypes.c_void_p(a.data_ptr()) for a in (t, sq, rs, rc))) == 0
    root = torch.sqrt(torch.abs(t))
    for name, got, want in (("sqrt", sq, root), ("rsqrt", rs, 1.0 / root), ("rcp", rc, 1.0 / t)):
        err = torch.max(torch.abs(got / want - 1.0)).item()
        assert err <= 2.0 ** -51, (name, err)
