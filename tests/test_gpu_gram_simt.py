"""The plain FP32 and FP64 Gram x block kernels at the edges of their tiles: 32- and 128-row tiles, 16-column
stages split over one to eight blocks of a cluster (FP32: and two halves of a block), 1 to 9 columns per
thread or warp, and widths above 72 that take several column chunks.

Bounds as in test_gpu_gram: FP64 1e-12, FP32 2e-5 (normwise per column, against the oracle's dense product).
"""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2405_08971_gb300 as ck  # noqa: E402


@pytest.mark.parametrize("nr,nc,width", [
    (1, 1, 1), (31, 15, 8), (32, 16, 9), (33, 17, 24), (127, 500, 25), (128, 33, 40), (129, 2000, 41),
    (300, 129, 56), (2500, 64, 57), (5000, 300, 72), (40000, 40, 73), (513, 4000, 145)])
@pytest.mark.parametrize("kernel", [0, 1, 2])
def test_gram_simt_tile_edges(nr, nc, width, kernel):
    rng = np.random.default_rng(nr + nc + width)
    Xr, Xc = rng.uniform(size=(nr, 2)), rng.uniform(size=(nc, 2))
    B = rng.standard_normal((width, nc))
    ref = 1.3 * (oracle.kernel_matrix(Xr, Xc, kernel, 0.2, 1.0) @ B.T).T
    d = torch.device("cuda:0")
    t = [torch.as_tensor(a, device=d) for a in (Xr, Xc, B)]
    for precision, tol in (("fp64", 1e-12), ("fp32", 2e-5)):
        # FP32 rounds the inputs too, so its reference takes the rounded B
        want = ref if precision == "fp64" else \
            1.3 * (oracle.kernel_matrix(Xr, Xc, kernel, 0.2, 1.0) @ B.astype(np.float32).astype(np.float64).T).T
        got = ck.cakf_gram_matmul(kernel, math.log(0.2), math.log(1.3), *t, precision=precision).cpu().double().numpy()
        # relative to the size of the sum's terms: a column of one or two terms may cancel
        scale = np.abs(B).sum(axis=1)[:, None] * 1.3 / math.sqrt(nc)
        err = np.linalg.norm(got - want, axis=1) / np.maximum(np.linalg.norm(want, axis=1), 1e-3 * scale[:, 0])
        assert err.max() <= tol, (precision, err.max())
