"""The eigensolver over the FP64 exponent range: whole matrices near both ends of it, and decoupled blocks far
below the rest of their matrix (rank-deficient Grams have them).  Every merge of the divide and conquer works in
its own power-of-two units; in the matrix's units its squares and reciprocals leave the range below 2^-430.

Bounds as in test_gpu_eig: eigenvalues, residual and orthogonality within 1e-12 relative to ||A||_2; a
block's own eigenvalues to 1e-12 of the block.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2405_08971_gb300 as ck  # noqa: E402


def matrix(kind, N):
    rng = np.random.default_rng(N)
    X = rng.standard_normal((N, N))
    if kind == "dense":
        return X + X.T
    if kind == "tridiagonal":
        return np.triu(np.tril(X + X.T, 1), -1)
    X = X * 10.0 ** -np.linspace(0, 6, N)      # a Gram matrix whose spectrum spans 12 digits
    return X.T @ X


def check(A, unit, mixed):
    """A in units of `unit`; the matrix given to the solver is unit * A."""
    N, nrm = A.shape[0], np.linalg.norm(A, 2)
    w, U = ck.cakf_eig_topk(torch.as_tensor(A * unit, device="cuda"), N, mixed=mixed)
    w, U = w.cpu().numpy() / unit, U.cpu().numpy().T
    assert np.max(np.abs(w - np.linalg.eigvalsh(A)[::-1])) <= 1e-12 * nrm
    assert np.linalg.norm((A / nrm) @ U - U * (w / nrm)) <= 1e-12 * np.sqrt(N)
    assert np.max(np.abs(U.T @ U - np.eye(N))) <= 1e-12
    return w


@pytest.mark.parametrize("exponent", [-1000, -700, -512, -490, -440, 506, 512, 700, 1000])
@pytest.mark.parametrize("kind,N", [(k, n) for k in ("dense", "tridiagonal", "gram") for n in (2, 3, 97)])
@pytest.mark.parametrize("mixed", [False, True])
def test_scales(kind, N, exponent, mixed):
    check(matrix(kind, N), 2.0 ** exponent, mixed)


@pytest.mark.parametrize("exponent", [-400, -440])
@pytest.mark.parametrize("kind,n", [("tridiagonal", 2), ("gram", 48)])
def test_a_small_block(kind, n, exponent):
    A = np.zeros((2 * n, 2 * n))
    B = matrix(kind, n) * 2.0 ** exponent
    A[:n, :n] = matrix("dense", n) + 100.0 * np.eye(n)
    A[n:, n:] = B
    w = check(A, 1.0, False)
    assert np.min(w[:n]) > 1.0
    assert np.max(np.abs(w[n:] - np.linalg.eigvalsh(B / 2.0 ** exponent)[::-1] * 2.0 ** exponent)) <= \
        1e-12 * np.linalg.norm(B / 2.0 ** exponent, 2) * 2.0 ** exponent
