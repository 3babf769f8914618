"""The performance cases: work that a user of the framework has it do, over the range of its sizes.

Five kinds of call, each through the public binding:

* ``gram``    K(Xr, Xc) B, the matrix-free kernel-Gram product (cakf_gram_matmul and its variant that
              allocates nothing);
* ``factor``  the tall-skinny factor products of the filter and smoother (cakf_factor_gemm);
* ``eig``     the truncation eigensolver (cakf_eig_topk), returned as the kept eigenvalues and the kept
              part U diag(w) U^T of the Gram (eigenvectors alone are defined up to sign and, in
              clusters, up to rotation);
* ``series``  a whole filter + smoother pass over a time series;
* ``fit``     one evaluation of a hyperparameter fit: filter, negative log likelihood and gradient.

Coordinates, spectra and data follow the models of ``synth`` (uniform 2-D grids, the lat-lon sphere
grid, random-Fourier-feature draws of the prior plus noise).  The FP32-based modes of ``series`` hand
their fields on as float32: the arithmetic behind them is FP32.
"""
import math

import numpy as np
import torch

import paper_2405_08971_gb300 as ck

DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # a few stations against a small set of observations, called in a latency-bound loop by a program
        # that must not allocate: launches and host work are all there is
        {"name": "gram_small", "kind": "gram", "nr": 513, "nc": 300, "width": 17, "dim": 2, "kernel": 1,
         "precision": "fp32", "noalloc": True},
        # the shape of the paper's kernel benchmark (9,600 points in 3-D, 128 columns, plus the mean
        # column) in the plain FP32 mode
        {"name": "gram_9600_fp32", "kind": "gram", "nr": 9600, "nc": 9600, "width": 129, "dim": 3, "kernel": 1,
         "precision": "fp32", "noalloc": False},
        # the filter's product K(X, X_o)[V v] on the 65,536-point sphere grid in the default mixed mode
        {"name": "gram_filter_65k", "kind": "gram", "nr": 65536, "nc": 8192, "width": 65, "dim": 3, "kernel": 1,
         "precision": "fp16x3", "noalloc": False},
        # the same product of the 2-D model in the FP64 reference mode (ragged observation count)
        {"name": "gram_2d_fp64", "kind": "gram", "nr": 4097, "nc": 2000, "width": 33, "dim": 2, "kernel": 2,
         "precision": "fp64", "noalloc": False},
        # covariance times a full-rank block (all 512 factor columns) with BF16 tiles: the widest product
        {"name": "gram_wide_bf16", "kind": "gram", "nr": 32768, "nc": 16384, "width": 513, "dim": 3, "kernel": 1,
         "precision": "bf16", "noalloc": False},
        # Truncate: the 65k factor rotated onto its kept eigenvectors
        {"name": "factor_rotate_65k", "kind": "factor", "trans": False, "M": 65536, "N": 512, "K": 576,
         "precision": "tf32x3", "update": False},
        # the smoother's projection M^T X of one tall block onto another
        {"name": "factor_project_65k", "kind": "factor", "trans": True, "M": 512, "N": 577, "K": 65536,
         "precision": "tf32x3", "update": False},
        # the low-rank correction K(X, X_o) V - M t of a small 2-D model in the plain FP32 mode, ragged
        {"name": "factor_small_fp32", "kind": "factor", "trans": False, "M": 5000, "N": 33, "K": 257,
         "precision": "fp32", "update": True},
        # the eigensolver inside every truncation of the 65k model (r = 512, i = 64)
        {"name": "eig_576_mixed", "kind": "eig", "N": 576, "keep": 512, "mixed": True},
        # the same for the 2-D model (r = 256, i = 32) in the FP64 mode
        {"name": "eig_288_fp64", "kind": "eig", "N": 288, "keep": 256, "mixed": False},
        # filter + smoother on the sphere grid in the mixed mode, actions frozen (a model evaluated
        # again with the actions of an earlier fit); ten steps reach the truncation
        {"name": "series_sphere_65k", "kind": "series", "grid": "sphere", "nx": 256, "ny": 256, "m": 8192, "T": 10,
         "budget": 64, "rank": 512, "lx": 0.1, "sn2": 0.05, "kernel": 1, "precision": "fp16x3", "policy": "cg"},
        # one evaluation of a hyperparameter fit with the actions frozen (the gradient check's 2-D model),
        # FP64: many small launches
        {"name": "fit_2d_1k_fp64", "kind": "fit", "grid": "2d", "nx": 32, "ny": 32, "m": 128, "T": 20, "budget": 32,
         "rank": 256, "lx": 0.05, "sn2": 0.01, "kernel": 2, "precision": "fp64", "policy": "cg"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gram", "gram", "gram", "factor", "factor", "eig", "eig", "series", "fit"])
    if kind == "gram":
        precision = rng.choice(["fp32", "fp16x3", "fp16x3", "bf16", "tf32", "tf32x3", "fp64"])
        nr, nc = _log_int(rng, 300, 40000), _log_int(rng, 200, 12000)
        width = _log_int(rng, 2, 300)
        if precision in ("fp64", "fp32"):     # the plain modes serve the smaller models
            nr, nc, width = min(nr, 12000), min(nc, 4000), min(width, 70)
        return {"kind": "gram", "nr": nr, "nc": nc, "width": width, "dim": rng.choice([1, 2, 3]),
                "kernel": rng.choice([0, 1, 2]), "precision": precision,
                "noalloc": nr * nc < 4e6 and rng.random() < 0.5}
    if kind == "factor":
        trans = rng.random() < 0.5
        tall = _log_int(rng, 1000, 65536)
        a, b = _log_int(rng, 16, 512), _log_int(rng, 16, 577)
        M, N, K = (a, b, tall) if trans else (tall, b, a)
        return {"kind": "factor", "trans": trans, "M": M, "N": N, "K": K,
                "precision": rng.choice(["fp32", "tf32x3", "tf32x3"]), "update": rng.random() < 0.5}
    if kind == "eig":
        N = _log_int(rng, 24, 640)
        return {"kind": "eig", "N": N, "keep": max(1, N - rng.randint(0, N // 4)), "mixed": rng.random() < 0.5}
    if kind == "series":
        side = rng.randint(24, 72)
        n = side * (side + 3)
        policy = rng.choice(["cg", "cg", "coordinate", "full"])
        m = rng.randint(max(40, n // 12), n // 4)
        budget = rng.randint(8, 24)
        if policy == "full":                  # every direction observed: the exact posterior
            m = budget = rng.randint(12, 32)
        return {"kind": "series", "grid": rng.choice(["2d", "sphere"]), "nx": side, "ny": side + 3, "m": m,
                "T": rng.randint(5, 12), "budget": budget, "rank": budget * rng.randint(2, 5), "lx": 0.15,
                "sn2": 0.05, "kernel": rng.choice([1, 2]),
                "precision": "fp64" if policy == "full" else rng.choice(["fp32", "fp16x3", "tf32x3", "fp64"]),
                "policy": policy}
    side = rng.randint(20, 40)
    n = side * side
    return {"kind": "fit", "grid": "2d", "nx": side, "ny": side, "m": rng.randint(n // 12, n // 6),
            "T": rng.randint(5, 20), "budget": rng.randint(8, 32), "rank": rng.randint(60, 200), "lx": 0.08,
            "sn2": 0.01, "kernel": rng.choice([1, 2]), "precision": "fp64", "policy": "cg"}


# ------------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _points(case, n, g):
    if case["dim"] == 3:                      # the sphere model
        x = torch.randn((n, 3), generator=g, device=DEV, dtype=F64)
        return (x / x.norm(dim=1, keepdim=True)).contiguous()
    return torch.rand((n, case["dim"]), generator=g, device=DEV, dtype=F64)


def _gram_inputs(case, seed):
    g = _gen(seed)
    Xr, Xc = _points(case, case["nr"], g), _points(case, case["nc"], g)
    # directions and solution coefficients: columns of norm about one, of different sizes
    scale = torch.exp(torch.rand((case["width"], 1), generator=g, device=DEV, dtype=F64) * 3 - 2)
    B = torch.randn((case["width"], case["nc"]), generator=g, device=DEV, dtype=F64) * scale / math.sqrt(case["nc"])
    B = B.to(F64 if case["precision"] == "fp64" else torch.float32)
    return Xr, Xc, B


def _factor_inputs(case, seed):
    g = _gen(seed)
    M, N, K = case["M"], case["N"], case["K"]

    def block(cols, rows, decay):             # a downdate factor: column norms over several decades
        s = torch.exp(-decay * torch.arange(cols, device=DEV) / max(cols, 1))
        return torch.randn((cols, rows), generator=g, device=DEV) * s[:, None]

    if case["trans"]:
        A, B = block(M, K, 6.0), block(N, K, 2.0)
    else:
        A, B = block(K, M, 6.0), torch.randn((N, K), generator=g, device=DEV) / math.sqrt(K)
    C0 = torch.randn((N, M), generator=g, device=DEV)
    return A, B, C0


def _eig_input(case, seed):
    """The Gram of [a M+, P^- W]: M+ with orthogonal columns of decaying norms, bordered by new columns."""
    g = _gen(seed)
    N = case["N"]
    i = max(1, N // 9)
    r = N - i
    d = torch.exp(-12.8 * torch.arange(r, device=DEV, dtype=F64) / r)
    d = torch.sort(d * (0.5 + torch.rand(r, generator=g, device=DEV, dtype=F64)), descending=True).values
    Wq = torch.randn((r, i), generator=g, device=DEV, dtype=F64) * 0.3     # W in the span of M+ ...
    Wp = torch.randn((3 * N - r, i), generator=g, device=DEV, dtype=F64) * 0.3    # ... and outside it
    B = d.sqrt()[:, None] * Wq
    A = torch.zeros((N, N), device=DEV, dtype=F64)
    A[:r, :r] = torch.diag(d)
    A[:r, r:] = B
    A[r:, :r] = B.T
    C = Wq.T @ Wq + Wp.T @ Wp
    A[r:, r:] = 0.5 * (C + C.T)
    return A


def _grid(case):
    nx, ny = case["nx"], case["ny"]
    if case["grid"] == "sphere":
        la = (torch.arange(nx, device=DEV, dtype=F64) + 0.5) * math.pi / nx - math.pi / 2
        lo = torch.arange(ny, device=DEV, dtype=F64) * 2 * math.pi / ny
        la, lo = torch.meshgrid(la, lo, indexing="ij")
        x = torch.stack([la.cos() * lo.cos(), la.cos() * lo.sin(), la.sin()], -1)
        return x.reshape(-1, 3).contiguous()
    gx = (torch.arange(nx, device=DEV, dtype=F64) + 0.5) / nx
    gy = (torch.arange(ny, device=DEV, dtype=F64) + 0.5) / ny
    x, y = torch.meshgrid(gx, gy, indexing="ij")
    return torch.stack([x, y], -1).reshape(-1, 2).contiguous()


def _kernel(X, Y, kernel, lx):
    """Matern correlations in 64 bits."""
    d2 = torch.zeros((X.shape[0], Y.shape[0]), device=X.device, dtype=F64)
    for c in range(X.shape[1]):
        d2 = d2 + (X[:, c][:, None] - Y[:, c][None, :]) ** 2
    s = torch.sqrt(torch.clamp(d2, min=1e-300)) * (1.0, math.sqrt(3.0), math.sqrt(5.0))[kernel] / lx
    e = torch.exp(-s)
    return e if kernel == 0 else (1 + s) * e if kernel == 1 else (1 + s + s * s / 3) * e


def _lanczos(K, sn2, r, count):
    """Orthonormal basis of the Krylov space of K + sn2 I at r (m x count)."""
    Q = torch.zeros((r.numel(), count), device=r.device, dtype=F64)
    q = r / r.norm()
    for j in range(count):
        Q[:, j] = q
        q = K @ q + sn2 * q
        for _ in range(2):
            q = q - Q[:, : j + 1] @ (Q[:, : j + 1].T @ q)
        q = q / q.norm()
    return Q


def _model(case, seed):
    """Grid, observation sets (70 % fixed stations), data and, for frozen CG actions, the actions."""
    g = _gen(seed)
    X = _grid(case)
    n, T, m = X.shape[0], case["T"], case["m"]
    lx, lt, dt, sn2, kernel = case["lx"], 1.0, 0.1, case["sn2"], case["kernel"]
    a = math.exp(-dt / lt)
    F = 512                                     # random Fourier features of the Matern spectral density
    nu = (0.5, 1.5, 2.5)[kernel]
    chi = torch.randn((F, int(2 * nu)), generator=g, device=DEV, dtype=F64).square().sum(1)
    om = torch.randn((F, X.shape[1]), generator=g, device=DEV, dtype=F64) / lx * torch.sqrt(2 * nu / chi)[:, None]
    ph = torch.rand(F, generator=g, device=DEV, dtype=F64) * 2 * math.pi
    perm = torch.randperm(n, generator=g, device=DEV)
    ns = int(0.7 * m)
    stations, others = perm[:ns], perm[ns:]
    w = torch.randn(F, generator=g, device=DEV, dtype=F64)
    t = np.arange(T + 1) * dt
    mu = None
    if case["grid"] == "2d":                    # seasonal prior mean of the 2-D models
        mu = 0.5 * torch.as_tensor(np.sin(2 * np.pi * t / 5.0), device=DEV)[:, None] * torch.cos(2 * math.pi * X[:, 0])[None]
        mu = mu.contiguous()
    idx, ys, acts = [], [], []
    for k in range(1, T + 1):
        w = a * w + math.sqrt(1 - a * a) * torch.randn(F, generator=g, device=DEV, dtype=F64)
        extra = others[torch.randperm(others.numel(), generator=g, device=DEV)[: m - ns]]
        ix = torch.sort(torch.cat([stations, extra])).values
        y = (torch.cos(X[ix] @ om.T + ph) * math.sqrt(2.0 / F)) @ w
        y = y + math.sqrt(sn2) * torch.randn(m, generator=g, device=DEV, dtype=F64)
        if mu is not None:
            y = y + mu[k, ix]
        if case["policy"] == "cg":
            acts.append(_lanczos(_kernel(X[ix], X[ix], kernel, lx), sn2, y, min(case["budget"], m)))
        idx.append(ix)
        ys.append(y)
    return {"X": X, "idx": idx, "y": ys, "mu": mu, "acts": acts, "theta": [math.log(lx), math.log(lt), 0.0, math.log(sn2)],
            "dt": dt}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gram":
        Xr, Xc, B = _gram_inputs(case, seed)
        return {"case": case, "Xr": Xr, "Xc": Xc, "B": B,
                "out": torch.empty((case["width"], case["nr"]), device=DEV, dtype=B.dtype)}
    if kind == "factor":
        A, B, C0 = _factor_inputs(case, seed)
        return {"case": case, "A": A, "B": B, "C0": C0, "C": torch.empty_like(C0)}
    if kind == "eig":
        return {"case": case, "A": _eig_input(case, seed)}
    mod = _model(case, seed)
    T, n, m = case["T"], mod["X"].shape[0], case["m"]
    replay = counts = None
    if mod["acts"]:
        replay = np.concatenate([S.T.contiguous().cpu().numpy().ravel() for S in mod["acts"]])
        counts = np.array([0] + [S.shape[1] for S in mod["acts"]], dtype=np.int32)
    problem = ck.make_problem(
        mod["X"], case["kernel"], *mod["theta"], T, mod["dt"], np.arange(T + 1, dtype=np.int32) * m,
        torch.cat(mod["idx"]).to(torch.int32), torch.cat(mod["y"]), case["budget"], case["rank"],
        precision=case["precision"], prior_mean=mod["mu"], replay_actions=replay, replay_counts=counts,
        policy="coordinate" if case["policy"] == "coordinate" else "cg")
    outs = [torch.empty((T + 1, n), device=DEV, dtype=F64) for _ in range(4)]
    return {"case": case, "problem": problem, "ctx": ck.Context(), "outs": outs}


# ------------------------------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gram":
        call = ck.cakf_gram_matmul_noalloc if case["noalloc"] else ck.cakf_gram_matmul
        return call(case["kernel"], math.log(0.1), 0.0, state["Xr"], state["Xc"], state["B"], out=state["out"],
                    precision=case["precision"])
    if kind == "factor":
        if case["update"]:
            C = state["C"].copy_(state["C0"])
            return ck.cakf_factor_gemm(state["A"], state["B"], C, trans_a=case["trans"], alpha=-1.0, beta=1.0,
                                       precision=case["precision"])
        return ck.cakf_factor_gemm(state["A"], state["B"], state["C"], trans_a=case["trans"],
                                   precision=case["precision"])
    if kind == "eig":
        w, U = ck.cakf_eig_topk(state["A"], case["keep"], mixed=case["mixed"])
        return {"w": w, "kept": (U.T * w) @ U}
    st = torch.cuda.current_stream().cuda_stream
    fm, fv, sm, sv = state["outs"]
    if kind == "series":
        ctx, _, _ = ck.cakf_filter(state["problem"], state["ctx"], fm, fv, stream=st)
        ck.cakf_smooth(ctx, sm, sv, stream=st)
        out = {"filter_mean": fm, "filter_var": fv, "smoother_mean": sm, "smoother_var": sv}
        return out if case["precision"] == "fp64" else {k: v.float() for k, v in out.items()}
    ctx, _, _ = ck.cakf_filter(state["problem"], state["ctx"], fm, fv, stream=st)
    nll = ck.cakf_nll(ctx)
    return {"nll": nll, "grad": ck.cakf_nll_backward(ctx), "filter_mean": fm, "filter_var": fv}


# ------------------------------------------------------------------------------------- work
def work(case):
    """What a pass cannot do without: each input read once, each output written once; the arithmetic of
    the definition (a kernel value counted as 3 dim + 6 operations)."""
    kind = case["kind"]
    if kind == "gram":
        nr, nc, w, dim = case["nr"], case["nc"], case["width"], case["dim"]
        es = 8 if case["precision"] == "fp64" else 4
        return {"bytes": (nr + nc) * dim * 8 + w * (nr + nc) * es, "flops": nr * nc * (2.0 * w + 3 * dim + 6)}
    if kind == "factor":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 4 * (M * K + K * N + M * N * (2 if case["update"] else 1)), "flops": 2.0 * M * N * K}
    if kind == "eig":
        N, keep = case["N"], case["keep"]
        return {"bytes": 8 * (2 * N * N + keep),
                "flops": 4.0 / 3.0 * N ** 3 + 2.0 * N * N * keep + 2.0 * N * N * keep}
    n, m, T, i, r = case["nx"] * case["ny"], case["m"], case["T"], case["budget"], case["rank"]
    dim = 3 if case["grid"] == "sphere" else 2
    ev = 3 * dim + 6
    flops = 0.0
    cols = 0
    for _ in range(T):
        N = cols + i
        keep = min(r, N)
        flops += 0.5 * m * m * ev + 2.0 * m * m * i + n * m * (ev + 2.0 * (i + 1)) + 4.0 * n * cols * (i + 1)
        trunc = 4.0 / 3.0 * N ** 3 + 2.0 * n * N * keep
        flops += trunc
        if kind == "series":                    # the smoother's step: projection, combination, truncation
            flops += 4.0 * n * cols * (keep + 1) + 2.0 * n * i * (keep + 1) + 2.0 * trunc
        else:                                   # four tangents of the step
            flops += n * m * (ev + 2.0 * (i + 1)) + 4 * (4.0 * n * cols * (i + 1) + 2.0 * n * N * keep)
        cols = keep
    outs = 4 if kind == "series" else 2
    return {"bytes": n * dim * 8 + T * m * 12 + outs * (T + 1) * n * 8, "flops": flops}


# ------------------------------------------------------------------------------------- 64 bits
def _exact_gram(case, seed):
    Xr, Xc, B = _gram_inputs(case, seed)
    B = B.to(F64).T.contiguous()
    out = torch.empty((case["nr"], case["width"]), device=DEV, dtype=F64)
    step = max(1, (1 << 27) // case["nc"])
    for r in range(0, case["nr"], step):
        out[r:r + step] = _kernel(Xr[r:r + step], Xc, case["kernel"], 0.1) @ B
    return out.T.contiguous()


def _exact_filter(case, mod, theta):
    """The filter in 64 bits with the whole observation Gram in memory; the truncation rotations are held
    fixed for derivatives.  Per step: means, variances, the factors the smoother needs; and the negative
    log likelihood."""
    X, dt, r = mod["X"], mod["dt"], case["rank"]
    lx, lt, sf2, sn2 = torch.exp(theta)
    a = torch.exp(-dt / lt)
    n, mu = X.shape[0], mod["mu"]
    zero = torch.zeros(n, device=DEV, dtype=F64)
    mean = mu[0] if mu is not None else zero
    M = torch.zeros((n, 0), device=DEV, dtype=F64)
    means, varis, steps = [mean], [sf2 * torch.ones(n, device=DEV, dtype=F64)], [None]
    nll = torch.zeros((), device=DEV, dtype=F64)
    for k in range(1, case["T"] + 1):
        ix, y = mod["idx"][k - 1], mod["y"][k - 1]
        m = ix.numel()
        mp = a * mean + (mu[k] - a * mu[k - 1] if mu is not None else 0.0)
        Mp = a * M
        Mo = Mp[ix]
        G = sf2 * _kernel(X[ix], X[ix], case["kernel"], lx) + sn2 * torch.eye(m, device=DEV, dtype=F64) - Mo @ Mo.T
        r0 = y - mp[ix]
        i = min(case["budget"], m)
        if mod["acts"]:                         # "cg": the actions of CG on the prior, frozen
            S = mod["acts"][k - 1]
        elif case["policy"] == "coordinate":
            S = torch.zeros((m, i), device=DEV, dtype=F64)
            q = torch.arange(i, device=DEV)
            S[((q.to(F64) + 0.5) * m / i).to(torch.int64), q] = 1.0
        else:                                   # "full": the actions span all of the observations
            S = torch.eye(m, device=DEV, dtype=F64)
        S = torch.linalg.qr(S).Q                # the same span, well conditioned
        Gh = S.T @ G @ S
        Gh = 0.5 * (Gh + Gh.T)
        L = torch.linalg.cholesky(Gh)
        V = torch.linalg.solve_triangular(L, S.T, upper=False).T
        c = V.T @ r0
        nll = nll + 0.5 * i * math.log(2 * math.pi) + torch.log(torch.diagonal(L)).sum() + 0.5 * (c * c).sum()
        Vv = torch.cat([V, (V @ c)[:, None]], 1)
        rows = max(1, (1 << 27) // m)
        KV = torch.cat([sf2 * _kernel(X[q:q + rows], X[ix], case["kernel"], lx) @ Vv for q in range(0, n, rows)], 0)
        PV = KV - Mp @ (Mo.T @ Vv)
        mean = mp + PV[:, i]
        full = torch.cat([Mp, PV[:, :i]], 1)
        means.append(mean)
        varis.append(sf2 - (full * full).sum(1))
        steps.append({"M": Mp, "PV": PV[:, :i], "KV": KV, "Vv": Vv, "ix": ix})
        if r > 0 and full.shape[1] > r:
            with torch.no_grad():
                U = torch.linalg.eigh(full.T @ full).eigenvectors[:, -r:]
            full = full @ U
        M = full
    return means, varis, steps, nll, a


def _exact_smoother(case, fm, fv, steps, a):
    T, r = case["T"], case["rank"]
    n = fm[0].numel()

    def spread(ix, block):                      # H^T block
        out = torch.zeros((n, block.shape[1]), device=DEV, dtype=F64)
        out[ix] = block
        return out

    ms, vs = list(fm), list(fv)
    W, KW = spread(steps[T]["ix"], steps[T]["Vv"]), steps[T]["KV"]     # last column: the vector message
    for k in range(T - 1, -1, -1):
        X, Y = a * W, a * KW
        if k == 0:
            ms[0], vs[0] = fm[0] + Y[:, -1], fv[0] - (Y[:, :-1] ** 2).sum(1)
            break
        s = steps[k]
        ix, V, v = s["ix"], s["Vv"][:, :-1], s["Vv"][:, -1:]
        P = Y - s["M"] @ (s["M"].T @ X)
        Z = V.T @ P[ix]
        P = P - s["PV"] @ Z
        ms[k], vs[k] = fm[k] + P[:, -1], fv[k] - (P[:, :-1] ** 2).sum(1)
        W = torch.cat([spread(ix, V), X - spread(ix, V @ Z)], 1)
        KW = torch.cat([s["KV"][:, :-1], Y - s["KV"][:, :-1] @ Z], 1)
        W[ix, -1] += v[:, 0]
        KW[:, -1] += s["KV"][:, -1]
        if r > 0 and W.shape[1] - 1 > r:
            U = torch.linalg.eigh(W[:, :-1].T @ W[:, :-1]).eigenvectors[:, -r:]
            W = torch.cat([W[:, :-1] @ U, W[:, -1:]], 1)
            KW = torch.cat([KW[:, :-1] @ U, KW[:, -1:]], 1)
    return ms, vs


def exact(case, seed):
    kind = case["kind"]
    if kind == "gram":
        return _exact_gram(case, seed)
    if kind == "factor":
        A, B, C0 = (t.to(F64) for t in _factor_inputs(case, seed))
        prod = B @ (A.T if case["trans"] else A)
        return C0 - prod if case["update"] else prod
    if kind == "eig":
        w, U = torch.linalg.eigh(_eig_input(case, seed))
        w, U = w[-case["keep"]:].flip(0), U[:, -case["keep"]:].flip(1)
        return {"w": w, "kept": (U * w) @ U.T}
    mod = _model(case, seed)
    theta = torch.tensor(mod["theta"], device=DEV, dtype=F64, requires_grad=kind == "fit")
    if kind == "series":
        with torch.no_grad():
            fm, fv, steps, _, a = _exact_filter(case, mod, theta)
            sm, sv = _exact_smoother(case, fm, fv, steps, a)
            return {"filter_mean": torch.stack(fm), "filter_var": torch.stack(fv),
                    "smoother_mean": torch.stack(sm), "smoother_var": torch.stack(sv)}
    fm, fv, _, nll, _ = _exact_filter(case, mod, theta)
    (grad,) = torch.autograd.grad(nll, theta)
    return {"nll": float(nll), "grad": grad.cpu().numpy(), "filter_mean": torch.stack(fm).detach(),
            "filter_var": torch.stack(fv).detach()}
