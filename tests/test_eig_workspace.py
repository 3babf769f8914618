"""The eigensolver's workspace: a context allocates it once, for its largest order, and solves every smaller one in
it, so it may never need more for a smaller order (the exchange's replicas drop from 4 to 1 above order
1,024).  The size itself on the CPU; on the GPU a filter and smoother whose orders pass through 1,024 on the way
to 1,128, against the oracle within the FP64 mode's 1e-10.
"""
import ctypes

import numpy as np
import pytest

import oracle
import synth


def test_workspace_never_shrinks_with_the_order():
    from paper_2405_08971_gb300 import build
    size = ctypes.CDLL(build.build())._ZN4cakf19eig_workspace_bytesEi      # cakf::eig_workspace_bytes(int)
    size.restype, size.argtypes = ctypes.c_size_t, [ctypes.c_int]
    b = np.array([size(n) for n in range(1, 2049)], dtype=np.int64)
    assert np.all(np.diff(b) >= 0)


@pytest.mark.gpu
def test_orders_on_both_sides_of_the_replica_limit():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_2405_08971_gb300 as ck
    w = synth.small(n=1100, dim=2, m=140, T=9, budget_i=128, rank_r=1000, lx=0.05, seed=3)
    S = synth.gaussian_actions(w, seed=5)
    f = oracle.filter_run(w, policy="given", S_given=S)
    ms_o, vs_o, _ = oracle.smoother_run(w, f)
    ctx, mf, vf = ck.cakf_filter(ck.problem_from_workload(w, precision="fp64", policy="batch",
                                                          replay=ck.pack_actions(S, w.T)))
    ms, vs = ck.cakf_smooth(ctx)
    ctx.close()
    for a, b in ((mf, f.m), (ms, ms_o)):
        scale = max(np.linalg.norm(b[k]) for k in range(b.shape[0]))
        for k in range(b.shape[0]):
            assert np.linalg.norm(a[k] - b[k]) <= 1e-10 * (np.linalg.norm(b[k]) or scale)
    for a, b in ((vf, f.var), (vs, vs_o)):
        assert np.max(np.abs(a - b) / np.abs(b)) <= 1e-10
