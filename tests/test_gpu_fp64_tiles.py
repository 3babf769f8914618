"""The FP64 mode at the observation counts where its matvec changes tiling (every entry up to 416, 32 x 32
tiles up to 2,048, 128 x 128 above; see gram_matvec_slots), and at the ragged orders of its factor
products (32-row tiles, 1 to 4 columns per warp, K split or not), against the oracle.  The second step
has one observation fewer than the first, so both sides of a boundary run on one context's buffers.

Bound: the FP64 mode's 1e-10 on means (normwise per step) and variances (elementwise).
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2405_08971_gb300 as ck  # noqa: E402


def two_steps(m):
    w = synth.small(n=m + 37, dim=2, m=m, T=2, budget_i=min(5, m), rank_r=7, lx=0.1, seed=m)
    keep = np.ones(2 * m, dtype=bool)
    if m > 1:
        keep[m + m // 2] = False
    ptr = np.array([0, m, int(keep.sum())], dtype=np.int32)
    return w.with_(obs_ptr=ptr, obs_idx=w.obs_idx[keep], y=w.y[keep])


@pytest.mark.parametrize("m", [1, 2, 33, 257, 417, 1000, 2049])
def test_fp64_tilings_against_the_oracle(m):
    w = two_steps(m)
    f = oracle.filter_run(w)
    ms_o, vs_o, _ = oracle.smoother_run(w, f)
    ctx, mf, vf = ck.cakf_filter(ck.problem_from_workload(w, precision="fp64"))
    ms, vs = ck.cakf_smooth(ctx)
    ctx.close()
    for a, b in ((mf, f.m), (ms, ms_o)):
        scale = max(np.linalg.norm(b[k]) for k in range(b.shape[0]))
        for k in range(b.shape[0]):
            assert np.linalg.norm(a[k] - b[k]) <= 1e-10 * (np.linalg.norm(b[k]) or scale)
    for a, b in ((vf, f.var), (vs, vs_o)):
        assert np.max(np.abs(a - b) / np.abs(b)) <= 1e-10
