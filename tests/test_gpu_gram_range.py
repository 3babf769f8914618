"""The plain FP32 Gram x block product where sf2 K B is in range and K B is not: sf2 belongs to the kernel value.

Bound as in test_gpu_gram for FP32: 2e-5, normwise per column.
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


@pytest.mark.parametrize("nr,nc,width", [(33, 300, 3), (5000, 300, 72)])
@pytest.mark.parametrize("kernel", [0, 1, 2])
def test_large_operands_and_a_small_variance(nr, nc, width, kernel):
    rng = np.random.default_rng(nr)
    Xr, Xc = rng.uniform(size=(nr, 2)), rng.uniform(size=(nc, 2))
    B = rng.uniform(0.5, 1.0, size=(width, nc)).astype(np.float32) * np.float32(1e37)
    t = [torch.as_tensor(a, device="cuda:0") for a in (Xr, Xc, B)]
    got = ck.cakf_gram_matmul(kernel, math.log(0.5), math.log(1e-3), *t, precision="fp32").cpu().double().numpy()
    want = 1e-3 * (oracle.kernel_matrix(Xr, Xc, kernel, 0.5, 1.0) @ B.astype(np.float64).T).T
    assert np.max(np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)) <= 2e-5
