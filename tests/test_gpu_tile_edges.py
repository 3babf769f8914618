"""The tensor-core Gram products and the factor products at the edges of their slices, stages and tiles: a single
K slice and odd numbers of them (two producer groups take alternate slices), 2 to 8 pipeline stages (widths),
tiles shared between CTAs, one row; factor products of one row, column or term, ragged K, and a TN product
whose last chunks are cut finer.

Bounds, per column normwise against the exact product: as in test_gpu_gram (split modes 1e-4, TF32 5e-3,
BF16 3e-2, the mean column 2e-5) and test_gpu_gemm (FP32 1e-5, split TF32 5e-5).
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


def rel(got, ref):
    return np.linalg.norm(got - ref, axis=1) / np.maximum(np.linalg.norm(ref, axis=1), 1e-300)


@pytest.mark.parametrize("nr,nc,width", [(1, 1, 2), (129, 31, 200), (128, 33, 305), (20001, 65, 17), (300, 97, 513),
                                         (20001, 161, 305)])
@pytest.mark.parametrize("precision,tol", [("fp16x3", 1e-4), ("tf32x3", 1e-4), ("tf32", 5e-3), ("bf16", 3e-2)])
def test_gram_slices_and_stages(nr, nc, width, precision, tol):
    rng = np.random.default_rng(nr + nc + width)
    Xr, Xc = rng.uniform(size=(nr, 3)), rng.uniform(size=(nc, 3))
    B = rng.uniform(0.1, 1.0, size=(width, nc)).astype(np.float32)
    ref = 1.3 * (oracle.kernel_matrix(Xr, Xc, 1, 0.3, 1.0) @ B.astype(np.float64).T).T
    t = [torch.as_tensor(a, device="cuda:0") for a in (Xr, Xc, B)]
    got = ck.cakf_gram_matmul(1, math.log(0.3), math.log(1.3), *t, precision=precision).cpu().double().numpy()
    e = rel(got, ref)
    assert e[:-1].max() <= tol and e[-1] <= 2e-5, (e[:-1].max(), e[-1])


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-5), ("tf32x3", 5e-5)])
@pytest.mark.parametrize("trans,M,N,K", [
    (False, 31, 1, 1), (False, 33, 8, 15), (False, 129, 9, 16), (False, 8192, 24, 33), (False, 8193, 41, 48),
    (False, 100, 65, 17), (True, 16, 1, 1), (True, 17, 5, 33), (True, 130, 300, 2049), (True, 512, 577, 65541)])
@pytest.mark.parametrize("beta", [0.0, 1.0])
def test_factor_products(trans, M, N, K, precision, tol, beta):
    rng = np.random.default_rng(M + N + K)
    A = rng.uniform(0.1, 1.0, size=(K, M)).astype(np.float32)          # column-major M x K
    B = rng.uniform(0.1, 1.0, size=(N, K)).astype(np.float32)          # column-major K x N
    C = rng.uniform(0.1, 1.0, size=(N, M)).astype(np.float32)
    t = [torch.as_tensor(np.ascontiguousarray(a), device="cuda:0") for a in (A.T if trans else A, B, C)]
    ck.cakf_factor_gemm(*t, trans_a=trans, alpha=0.7, beta=beta, precision=precision)
    ref = 0.7 * (B.astype(np.float64) @ A.astype(np.float64)) + beta * C
    assert rel(t[2].cpu().double().numpy(), ref).max() <= tol
