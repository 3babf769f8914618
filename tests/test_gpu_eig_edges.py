"""The eigensolver at the edges of its kernels: the smallest orders, one owned column per block and up to the
orders where a block owns many (beyond the 5-entry poll batches), matrices scaled near the ends of the
FP64 range (the tridiagonalisation scales by a power of two), and columns its reflectors leave alone
(diagonal, decoupled, zero and rank-one matrices).

Bounds as in test_gpu_eig: eigenvalues, residual and orthogonality within 1e-12 relative to ||A||_2.
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
    if kind == "diagonal":
        return np.diag(rng.uniform(-1, 1, N))
    if kind == "zero":
        return np.zeros((N, N))
    if kind == "rank1":
        u = rng.standard_normal(N)
        return np.outer(u, u)
    if kind == "blocks":                       # decoupled blocks: zero columns below the subdiagonal
        A = np.zeros((N, N))
        for lo in range(0, N, 7):
            X = rng.standard_normal((min(7, N - lo),) * 2)
            A[lo:lo + 7, lo:lo + 7] = X @ X.T
        return A
    X = rng.standard_normal((N, N))
    return (X + X.T) * {"dense": 1.0, "huge": 2.0 ** 480, "tiny": 2.0 ** -480}[kind]


CASES = [("dense", N) for N in (1, 2, 3, 4, 5, 6, 31, 33, 64, 65, 152, 153, 305, 641, 1290)]
CASES += [(k, 97) for k in ("huge", "tiny", "diagonal", "zero", "rank1", "blocks")]


@pytest.mark.parametrize("kind,N", CASES)
@pytest.mark.parametrize("mixed", [False, True])
def test_eig_edges(kind, N, mixed):
    A = matrix(kind, N)
    nrm = np.linalg.norm(A, 2) or 1.0
    keep = max(1, N - N // 5)
    w_ref = np.linalg.eigvalsh(A)[::-1][:keep]
    w, U = ck.cakf_eig_topk(torch.as_tensor(A, device="cuda"), keep, mixed=mixed)
    w, U = w.cpu().numpy(), U.cpu().numpy().T
    assert np.max(np.abs(w - w_ref)) <= 1e-12 * nrm
    assert np.linalg.norm((A / nrm) @ U - U * (w / nrm)) <= 1e-12 * np.sqrt(keep)
    assert np.max(np.abs(U.T @ U - np.eye(keep))) <= 1e-12
