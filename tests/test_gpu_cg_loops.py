"""The CG iteration's kernels beyond what they load ahead: more than 64 previous directions and more than 512
factor columns, in the small FP64 row blocks (up to 2,048 observations), the 32/64-row blocks above and in FP32,
with the oracle's actions replayed (each next action is written by the update kernel), against the oracle.

Bounds: the modes' own, 1e-10 (FP64) and 1e-3 (FP32) on means (normwise per step) and variances (elementwise).
"""
import functools

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2405_08971_gb300 as ck  # noqa: E402


@functools.lru_cache(maxsize=None)
def case(m):
    T = 7 if m < 1000 else 2
    w = synth.small(n=m + 57, dim=2, m=m, T=T, budget_i=90, rank_r=640, lx=0.05, seed=m)
    return w, oracle.filter_run(w)


@pytest.mark.parametrize("m,precision", [(301, "fp64"), (301, "fp32"), (2081, "fp64")])
def test_many_directions_and_columns(m, precision):
    w, f = case(m)
    prob = ck.problem_from_workload(w, precision=precision, replay=ck.pack_actions(f.S, w.T))
    ctx, mf, vf = ck.cakf_filter(prob)
    ctx.close()
    tol = 1e-10 if precision == "fp64" else 1e-3
    scale = max(np.linalg.norm(f.m[k]) for k in range(f.m.shape[0]))
    for k in range(f.m.shape[0]):
        assert np.linalg.norm(mf[k] - f.m[k]) <= tol * (np.linalg.norm(f.m[k]) or scale)
    assert np.max(np.abs(vf - f.var) / np.abs(f.var)) <= tol
