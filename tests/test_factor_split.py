"""The split of a long K range over the CTAs of a transposed factor product: its last chunks are cut finer where
that fills the last round of units, which needs at least one CTA per output tile.  The plan on the CPU (in a child
process: a division by zero ends it), over products with fewer and more output tiles than CTAs; on the GPU
products of more tiles than SMs, within test_gpu_gemm's bound for split TF32.
"""
import subprocess
import sys

import numpy as np
import pytest

PLAN = """
import ctypes, sys
lib = ctypes.CDLL(sys.argv[1])
lib.cakf_split_tail.argtypes = [ctypes.c_int] * 5 + [ctypes.c_size_t, ctypes.c_void_p]
out = (ctypes.c_int * 3)()
cut = 0
for slots in (148, 152, 304):
    for base in (*range(1, 40), 147, 152, 153, 157, 256, 320, 1000):
        for nk in (1, 5, 64, 128, 129, 1000, 4096, 4097):
            for want in (1, 2, 5, 6, 64):
                ks = -(-nk // min(want, nk))
                kc = -(-nk // ks)
                for cap in (kc, 4096):
                    if lib.cakf_split_tail(base, nk, ks, kc, slots, cap, out):
                        full, tail, total = out
                        cut += 1
                        # whole chunks, then shorter ones that cover the rest, none empty, within the capacity
                        rest = nk - full * ks
                        assert 0 < full < kc and 0 < tail < ks and kc <= total <= cap, (base, nk, ks, kc)
                        assert (total - full - 1) * tail < rest <= (total - full) * tail, (base, nk, ks, kc)
                        assert base <= slots
print(cut)
"""


def test_the_last_chunks_cover_the_range():
    from paper_2405_08971_gb300 import build
    r = subprocess.run([sys.executable, "-c", PLAN, build.build()], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout) > 100


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(5000, 1024, 2048), (3000, 2000, 4096), (20000, 256, 2048)])
def test_products_of_more_tiles_than_sms(M, N, K):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2405_08971_gb300 as ck
    g = torch.Generator(device="cuda:0").manual_seed(M)
    A = 0.1 + 0.9 * torch.rand((M, K), generator=g, device="cuda:0")
    B = 0.1 + 0.9 * torch.rand((N, K), generator=g, device="cuda:0")
    got = ck.cakf_factor_gemm(A, B, trans_a=True, alpha=0.7, precision="tf32x3").cpu().double().numpy()
    ref = 0.7 * (B.double().cpu().numpy() @ A.double().cpu().numpy().T)
    assert np.max(np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 5e-5
