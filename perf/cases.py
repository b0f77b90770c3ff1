"""Performance cases: the calls a user of this library makes, at the sizes they make them.

Each case is one call (or the few calls that belong together) of the Python
binding on inputs like those of the library's own workloads: Kronecker-
structured matrices with sorted diagonals and random couplings, orthonormal
Lanczos bases, band matrices T of a real Lanczos run, the learned-pivot
network's training step, and whole solves.
"""
import math
import types

import numpy as np
import torch

import paper_2210_15763_gb300 as bbl

DEV = "cuda"


# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------
def listed():
    return [
        # S1 on the plain FP64 form's matrix (n = 2e4, ~100 nonzeros per row): the
        # smallest product of a solve, where the launch and the latency count.
        dict(name="spmm_csr_f64_n2e4", kind="spmm", nP=200, nN=100, K=4, c=4.75, b=4, dtype="f64", fmt="csr", sigma=0),
        # S1 of the FP32 stage on a stored matrix of the headline family (~282
        # nonzeros per row), in the format the autotuner picks for it.
        dict(name="spmm_sell_f32_n1e6", kind="spmm", nP=1000, nN=1000, K=12, c=4.8, b=8, dtype="f32", fmt="sell", sigma=1024),
        # S1 without a stored matrix: the factored operator of the headline family.
        dict(name="kron_f32_n2e6", kind="kron", nP=2000, nN=1000, K=12, c=4.8, b=8, dtype="f32"),
        # S2 of the plain FP64 form in the middle of a run.
        dict(name="reorth_f64_n2e5", kind="reorth", n=200000, b=8, blocks=50, dtype="f64"),
        # S2 in FP32 near the end of a run of the headline family.
        dict(name="reorth_f32_n1e6", kind="reorth", n=1000003, b=8, blocks=90, dtype="f32"),
        # First Gram-Schmidt pass of the FP32 stage: coefficients and update from the FP16 copy.
        dict(name="first_pass_f16_n1e6", kind="f16", n=1000003, blocks=90),
        # S3: the block normalisation at the headline's n.
        dict(name="cholqr2_f32_n2e6", kind="cholqr2", n=2000000, b=8, dtype="f32"),
        # S4: the lowest pairs of T late in a run (91 blocks of 8).
        dict(name="ritz_m728", kind="ritz", p=8, blocks=91, nev=8),
        # The learned pivot's training step (48 solves, hidden 128, 64 x 8 coefficients).
        dict(name="mlp_step_h128", kind="mlp", hidden=128, out=512, batch=48),
        # Many uneven problems at once (b = nev = 4, FP32 storage, FP64 polish).
        dict(name="batch_24", kind="batch", count=24, n_lo=2000, n_hi=20000, b=4),
        # A whole solve of the plain FP64 form, from a random pivot.
        dict(name="solve_f64_n2e4", kind="solve", nP=200, nN=100, K=4, c=4.75, b=4, dtype="f64"),
        # The headline step at a quarter of its size: bootstrapped pivot, FP32 stage, float-float polish.
        dict(name="solve_mixed_n5e5", kind="solve", nP=1000, nN=500, K=12, c=4.8, b=8, dtype="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmm", "spmm", "kron", "reorth", "reorth", "reorth", "f16", "cholqr2", "cholqr2", "ritz", "mlp", "batch",
                       "solve"])
    if kind == "spmm":
        nP = _log(rng, 40, 1000)
        nN = _log(rng, 40, 1000)
        return dict(kind="spmm", nP=nP, nN=nN, K=rng.choice([4, 8, 12]), c=round(rng.uniform(3.0, 4.8), 2),
                    b=rng.choice([1, 2, 4, 4, 8, 8, 8, 16, 3, 6]), dtype=rng.choice(["f64", "f32"]),
                    fmt=rng.choice(["csr", "sell"]), sigma=256)
    if kind == "kron":
        return dict(kind="kron", nP=_log(rng, 60, 2000), nN=_log(rng, 60, 1000), K=rng.choice([4, 8, 12]),
                    c=round(rng.uniform(3.0, 4.8), 2), b=rng.choice([4, 8, 8, 16]), dtype=rng.choice(["f32", "f32", "f64"]))
    if kind == "reorth":
        dtype = rng.choice(["f64", "f32"])
        b = rng.choice([1, 2, 4, 4, 8, 8, 8, 16, 5])
        n = _log(rng, 3000, 1000000)
        most = min((8.0e7 if dtype == "f64" else 7.2e8) / n / b, 800 / b)
        if dtype == "f64":  # making the basis takes 2 n m^2 FP64 operations, twice
            most = min(most, math.sqrt(1.0e11 / n) / b)
        return dict(kind="reorth", n=n, b=b, blocks=_log(rng, 2, max(2.0, min(most, n / (4 * b)))), dtype=dtype)
    if kind == "f16":
        n = _log(rng, 5000, 1000000)
        return dict(kind="f16", n=n, blocks=_log(rng, 4, min(100, n / 32)))
    if kind == "cholqr2":
        return dict(kind="cholqr2", n=_log(rng, 2000, 2000000), b=rng.choice([1, 2, 4, 4, 8, 8, 8, 16, 3]),
                    dtype=rng.choice(["f64", "f32"]))
    if kind == "ritz":
        p = rng.choice([1, 2, 4, 8, 8, 16])
        return dict(kind="ritz", p=p, blocks=_log(rng, 6, 800 / p), nev=min(16, rng.choice([p, 8, 4])))
    if kind == "mlp":
        return dict(kind="mlp", hidden=_log(rng, 16, 256), out=_log(rng, 32, 1024), batch=_log(rng, 6, 128))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 24), n_lo=1000, n_hi=_log(rng, 4000, 20000), b=rng.choice([2, 4, 8]))
    if rng.random() < 0.5:
        nP = _log(rng, 50, 250)
        return dict(kind="solve", nP=nP, nN=_log(rng, 40, 120), K=4, c=4.75, b=rng.choice([2, 4, 8]), dtype="f64")
    return dict(kind="solve", nP=_log(rng, 200, 900), nN=_log(rng, 150, 500), K=rng.choice([8, 12]),
                c=round(rng.uniform(3.5, 4.8), 2), b=8, dtype="f32")


# --------------------------------------------------------------------------
# Matrices: H = Hp (x) I + I (x) Hn + sum_k Cp_k (x) Cn_k
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + 17)
    return g


def _grid(x):
    # multiples of 2^-10: sums of a few products are exact, whatever their order
    return torch.round(x * 1024.0) / 1024.0


def _factor(g, N, per_row, sigma, diag):
    """Symmetric sparse N x N factor (rows, cols, values sorted by row and column)."""
    pairs = int(round(N * max(per_row, 0.0) / 2))
    i = torch.randint(0, N, (pairs,), generator=g, device=DEV)
    j = torch.randint(0, N, (pairs,), generator=g, device=DEV)
    lo, hi = torch.minimum(i, j), torch.maximum(i, j)
    key = torch.unique((lo * N + hi)[lo != hi])
    v = _grid(torch.randn(key.numel(), generator=g, device=DEV, dtype=torch.float64) * sigma)
    lo, hi, d = key // N, key % N, torch.arange(N, device=DEV)
    rows, cols, vals = torch.cat([lo, hi, d]), torch.cat([hi, lo, d]), torch.cat([v, v, _grid(diag)])
    o = torch.argsort(rows * N + cols)
    return rows[o], cols[o], vals[o]


def _factors(case, seed):
    """(Hp, Hn, [Cp_k], [Cn_k])."""
    g = _gen(seed)
    out = []
    for N in (case["nP"], case["nN"]):
        d = torch.sort(torch.rand(N, generator=g, device=DEV, dtype=torch.float64) * 20.0).values
        out.append(_factor(g, N, min(10.0, N / 4), 1.0, d))
    cp, cn = [], []
    for _ in range(case["K"]):
        for N, to in ((case["nP"], cp), (case["nN"], cn)):
            d = torch.randn(N, generator=g, device=DEV, dtype=torch.float64) * 0.5
            to.append(_factor(g, N, min(case["c"] - 1.0, N / 4), 0.5, d))
    return out[0], out[1], cp, cn


def _csr(n, rows, cols, vals, **kw):
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return types.SimpleNamespace(n=n, row_ptr=rp, col=cols.to(torch.int32), val=vals, **kw)


def _matrix(case, seed, dtype):
    """The stored matrix as CSR on the GPU; FP64 values are in units that no FP32 number holds."""
    nP, nN = case["nP"], case["nN"]
    n = nP * nN
    hp, hn, cp, cn = _factors(case, seed)
    q = torch.arange(nN, device=DEV)
    p = torch.arange(nP, device=DEV)
    one = ((q, q, torch.ones(nN, dtype=torch.float64, device=DEV)), (p, p, torch.ones(nP, dtype=torch.float64, device=DEV)))
    keys, vals = [], []
    for (ar, ac, av), (br, bc, bv) in [(hp, one[0]), (one[1], hn)] + list(zip(cp, cn)):
        keys.append(((ar[:, None] * nN + br[None, :]) * n + (ac[:, None] * nN + bc[None, :])).reshape(-1))
        vals.append((av[:, None] * bv[None, :]).reshape(-1))
    key, o = torch.sort(torch.cat(keys))
    val = torch.cat(vals)[o]
    del keys, vals, o
    key, inv = torch.unique_consecutive(key, return_inverse=True)
    val = torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, inv, val)
    del inv
    val = val.to(torch.float32) if dtype == "f32" else val * 0.9371
    return _csr(n, key // n, key % n, val)


def _host(c):
    return types.SimpleNamespace(n=c.n, row_ptr=c.row_ptr.cpu().numpy(), col=c.col.cpu().numpy(), val=c.val.cpu().numpy())


def _times(c, X):
    """H X in FP64 by torch."""
    with _quiet():
        A = torch.sparse_csr_tensor(c.row_ptr, c.col.to(torch.int64), c.val.to(torch.float64), size=(c.n, c.n))
        return A @ X


class _quiet:
    def __enter__(self):
        import warnings
        self.w = warnings.catch_warnings()
        self.w.__enter__()
        warnings.simplefilter("ignore")

    def __exit__(self, *a):
        self.w.__exit__(*a)


def _nnz_per_row(case):
    return 21.0 + case["K"] * case["c"] ** 2


# --------------------------------------------------------------------------
# Bases, blocks and band matrices
# --------------------------------------------------------------------------
def _basis(g, n, m, b, dtype):
    """Orthonormal columns (to rounding) as blocks (m/b, n, b), by Cholesky QR."""
    t = torch.float64 if dtype == "f64" else torch.float32
    X = torch.randn(n, m, generator=g, device=DEV, dtype=t) / math.sqrt(n)
    for _ in range(2 if dtype == "f32" else 1):
        R = torch.linalg.cholesky((X.T @ X).double(), upper=True)
        X = X @ torch.linalg.inv(R).to(t)
    return X.reshape(n, m // b, b).permute(1, 0, 2).contiguous()


def _new_block(g, basis, b):
    """W = H V_j as Gram-Schmidt meets it: mostly in the newest two blocks, the rest new."""
    W = torch.randn(basis.shape[1], b, generator=g, device=DEV, dtype=basis.dtype) / math.sqrt(basis.shape[1])
    for q in basis[-2:]:
        W = W + 3.0 * (q @ torch.randn(b, b, generator=g, device=DEV, dtype=basis.dtype))
    return (5.0 * W).contiguous()


def _lanczos(times, n, b, blocks, g, tol=None, nev=0):
    """Plain FP64 block Lanczos with full reorthogonalisation: (T, basis) of at most `blocks` blocks."""
    Q, _ = torch.linalg.qr(torch.randn(n, b, generator=g, device=DEV, dtype=torch.float64))
    V = torch.zeros(n, blocks * b, dtype=torch.float64, device=DEV)
    T = torch.zeros(blocks * b + b, blocks * b + b, dtype=torch.float64, device=DEV)
    V[:, :b] = Q
    for j in range(blocks):
        m = (j + 1) * b
        W = times(V[:, j * b:m])
        B = V[:, :m]
        C = B.T @ W
        W = W - B @ C
        C2 = B.T @ W
        W = W - B @ C2
        A = (C + C2)[j * b:]
        T[j * b:m, j * b:m] = 0.5 * (A + A.T)
        Q, R = torch.linalg.qr(W)
        s = torch.sign(torch.diagonal(R))
        R = s[:, None] * R
        T[m:m + b, j * b:m] = R
        T[j * b:m, m:m + b] = R.T
        if tol is not None and (j % 8 == 7 or j == blocks - 1):
            w, S = np.linalg.eigh(T[:m, :m].cpu().numpy())
            est = np.linalg.norm(R.cpu().numpy() @ S[-b:, :nev], axis=0)
            if np.all(est <= tol * max(1.0, abs(w[0]), abs(w[-1]))):
                return w[:nev]
        if j + 1 < blocks:
            V[:, m:m + b] = Q * s
    return None if tol is not None else T[:blocks * b, :blocks * b]


def _band(case, seed):
    """T of a block Lanczos run on a diagonal operator with a spectrum like the matrices' (lower band storage)."""
    p, m = case["p"], case["p"] * case["blocks"]
    g = _gen(seed)
    n = 3000 + 4 * m
    d = torch.randn(n, generator=g, device=DEV, dtype=torch.float64) * 6.0 + torch.rand(n, generator=g, device=DEV,
                                                                                        dtype=torch.float64) * 30.0
    T = _lanczos(lambda X: d[:, None] * X, n, p, case["blocks"], g)
    return torch.stack([torch.cat([torch.zeros(k, dtype=T.dtype, device=DEV), torch.diagonal(T, -k)]) for k in range(p + 1)],
                       1).contiguous(), T


def _spawn(seed, i):
    return 7919 * int(seed) + 31 * i + 5


def _batch_cases(case, seed):
    r = np.random.default_rng([int(seed), 3])
    out = []
    for _ in range(case["count"]):
        n = math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))
        nP = max(8, int(round(math.sqrt(2.0 * n))))
        out.append(dict(nP=nP, nN=max(4, int(round(n / nP))), K=4, c=math.sqrt((r.uniform(50.0, 150.0) - 21.0) / 4)))
    return out


# --------------------------------------------------------------------------
# prepare / run
# --------------------------------------------------------------------------
def _mlp_inputs(case, seed):
    r = np.random.default_rng([int(seed), 5])
    H, O, N = case["hidden"], case["out"], case["batch"]
    parts = []
    for o, i in ((H, 1), (H, H), (O, H)):
        parts += [r.uniform(-1, 1, o * i) / math.sqrt(i), r.uniform(-0.05, 0.05, o)]
    params = np.concatenate(parts).astype(np.float32)
    g = r.uniform(0.0, 1.0, N)
    t = np.cos(np.outer(g, r.uniform(0.0, 3.0, O)) + r.uniform(0.0, 6.3, O)) * r.uniform(0.05, 0.9, O)
    return params, g.astype(np.float32), t.astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    g = _gen(seed + 500009)
    t = {"f64": torch.float64, "f32": torch.float32}.get(case.get("dtype"))
    storage = {"f64": "fp64", "f32": "fp32"}.get(case.get("dtype"))
    if kind == "spmm":
        s["M"] = bbl.Matrix(_matrix(case, seed, case["dtype"]), storage=storage, fmt=case["fmt"], sell_sigma=case["sigma"])
        s["V"] = torch.randn(s["M"].n, case["b"], generator=g, device=DEV, dtype=t)
    elif kind == "kron":
        hp, hn, cp, cn = _factors(case, seed)
        h = lambda f, N: _host(_csr(N, *f))  # noqa: E731
        nP, nN = case["nP"], case["nN"]
        s["M"] = bbl.KronMatrix(types.SimpleNamespace(Hp=h(hp, nP), Hn=h(hn, nN), Cp=[h(f, nP) for f in cp], Cn=[h(f, nN) for f in cn]),
                                storage=storage)
        s["V"] = torch.randn(nP * nN, case["b"], generator=g, device=DEV, dtype=t)
    elif kind == "reorth":
        s["Q"] = _basis(g, case["n"], case["blocks"] * case["b"], case["b"], case["dtype"])
        s["W"] = _new_block(g, s["Q"], case["b"])
    elif kind == "f16":
        s["Q"] = _basis(g, case["n"], case["blocks"] * 8, 8, "f32")
        s["Q16"] = s["Q"].to(torch.float16)
        s["W"] = _new_block(g, s["Q"], 8)
    elif kind == "cholqr2":
        W = torch.randn(case["n"], case["b"], generator=g, device=DEV, dtype=t)
        s["W"] = W @ (torch.eye(case["b"], device=DEV, dtype=t) + 0.3 * torch.randn(case["b"], case["b"], generator=g, device=DEV, dtype=t))
    elif kind == "ritz":
        s["T"], _ = _band(case, seed)
    elif kind == "mlp":
        params, x, y = _mlp_inputs(case, seed)
        s["net"] = bbl.MLP(case["hidden"], case["out"])
        s["net"].set_params(params)
        s["x"], s["y"] = torch.from_numpy(x).to(DEV), torch.from_numpy(y).to(DEV)
    elif kind == "batch":
        mats = [_host(_matrix(c, _spawn(seed, i), "f32")) for i, c in enumerate(_batch_cases(case, seed))]
        s["B"] = bbl.Batch(mats, storage="fp32", fmt="sell", sell_sigma=256)
    else:
        fmt = "csr" if case["dtype"] == "f64" else "sell"
        s["M"] = bbl.Matrix(_matrix(case, seed, case["dtype"]), storage=storage, fmt=fmt, sell_sigma=0 if fmt == "csr" else 1024)
        if case["dtype"] == "f64":
            s["P"] = bbl.pivot_random(s["M"].n, case["b"], int(seed))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("spmm", "kron"):
        return bbl.spmm(s["M"], s["V"])
    if kind == "reorth":
        W = s["W"].clone()  # the new block of this iteration
        C = bbl.block_reorth(s["Q"], W)
        return {"W": W, "C": C}
    if kind == "f16":
        W = s["W"].clone()
        C = bbl.block_gram_f16(s["Q16"], W)
        bbl.block_update_f16old(s["Q16"], s["Q"], W, C)
        return {"W": W, "C": C}
    if kind == "cholqr2":
        Q = s["W"].clone()
        B, defl = bbl.cholqr2(Q)
        return {"Q": Q, "B": B, "defl": defl}
    if kind == "ritz":
        theta, S = bbl.ritz_banded(s["T"], case["nev"])
        return {"theta": theta, "S": S}
    if kind == "mlp":
        loss = s["net"].loss_grad(s["x"], s["y"])
        s["net"].adam_step(1e-3)
        params, grads = s["net"].get_params()
        return {"loss": loss, "grads": grads, "params": params}
    if kind == "batch":
        evals, _, _, status, _ = s["B"].solve(case["b"], case["b"], tol=1e-9, max_vectors=400)
        return {"evals": evals, "status": status}
    if case["dtype"] == "f64":  # energies and vectors to near working precision
        r = bbl.solve(s["M"], case["b"], case["b"], pivot=s["P"], tol=1e-12)
        return {"evals": r.evals, "evecs": r.evecs}
    P = bbl.pivot_bootstrap(s["M"], max(64, s["M"].n // 100), case["b"], sub_tol=1e-4)
    r = bbl.solve(s["M"], case["b"], case["b"], pivot=P, tol=1e-8, stage1_tol=3e-7, evecs=None)  # the energies
    return {"evals": r.evals}


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    e = 8.0 if case.get("dtype") == "f64" else 4.0
    if kind in ("spmm", "solve"):
        n = case["nP"] * case["nN"]
        nnz = n * _nnz_per_row(case)
        b = case["b"]
        if kind == "spmm":
            return dict(bytes=nnz * (e + 4) + 8 * (n + 1) + 2 * n * b * e, flops=2 * nnz * b)
        # about 80 (FP64, small) to 100 block steps: a product, and the new block against all earlier ones twice
        J = 100
        return dict(bytes=J * (nnz * (e + 4) + 8 * (n + 1) + 2 * n * b * e) + 2 * n * b * e * J * J / 2,
                    flops=J * 2 * nnz * b + 8 * n * b * b * J * J / 2)
    if kind == "kron":
        n = case["nP"] * case["nN"]
        f = (case["nP"] + case["nN"]) * (11 + case["K"] * case["c"])
        return dict(bytes=f * (e + 4) + 2 * n * case["b"] * e, flops=2 * n * case["b"] * (22 + 2 * case["K"] * case["c"]))
    if kind == "reorth":
        n, b, m = case["n"], case["b"], case["blocks"] * case["b"]
        return dict(bytes=n * m * e + 2 * n * b * e + 16 * m * b, flops=8 * n * m * b)
    if kind == "f16":
        n, m = case["n"], case["blocks"] * 8
        return dict(bytes=n * m * 2 + n * 16 * 4 + 2 * n * 8 * 4 + 8 * m * 8, flops=4 * n * m * 8)
    if kind == "cholqr2":
        n, b = case["n"], case["b"]
        return dict(bytes=2 * n * b * e, flops=4 * n * b * b)
    if kind == "ritz":
        m, p, nev = case["p"] * case["blocks"], case["p"], case["nev"]
        return dict(bytes=8 * m * (p + 1) + 8 * m * nev, flops=nev * m * (30 * p * p + 30 * p))
    if kind == "mlp":
        H, O, N = case["hidden"], case["out"], case["batch"]
        npar = 3 * H + H * H + O * H + O
        return dict(bytes=4 * npar * 8 + 4 * N * O, flops=6 * N * npar)
    rows = case["count"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
    return dict(bytes=60 * rows * 100 * 8, flops=60 * 2 * rows * 100 * case["b"] + 8 * rows * case["b"] ** 2 * 60 * 60 / 2)


# --------------------------------------------------------------------------
# The same results in 64 bits
# --------------------------------------------------------------------------
def _lowest(c, nev, b, tol):
    with _quiet():
        A = torch.sparse_csr_tensor(c.row_ptr, c.col.to(torch.int64), c.val.to(torch.float64), size=(c.n, c.n))
    return _lanczos(lambda X: A @ X, c.n, b, min(400, c.n // (2 * b)), _gen(99), tol=tol, nev=nev)


def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))


def _mlp_exact(case, seed):
    params, x, y = (torch.from_numpy(v).to(DEV).double() for v in _mlp_inputs(case, seed))
    H, O, N = case["hidden"], case["out"], case["batch"]
    sizes, shapes = [H, H, H * H, H, O * H, O], [(H, 1), None, (H, H), None, (O, H), None]
    leaf, used = [], []
    for v, sh in zip(torch.split(params, sizes), shapes):
        u = v.float().bfloat16().double().reshape(sh) if sh else v  # the weights are used in BF16
        leaf.append(u.clone().requires_grad_(True))
    h = _gelu(x[:, None] @ leaf[0].T + leaf[1])
    h = _gelu(h @ leaf[2].T + leaf[3])
    out = h @ leaf[4].T + leaf[5]
    loss = ((out - y) ** 2).mean()
    loss.backward()
    grads = torch.cat([v.grad.reshape(-1) for v in leaf])
    m, v = 0.1 * grads, 0.001 * grads * grads
    new = params - 1e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return {"loss": float(loss), "grads": grads.cpu().numpy(), "params": new.detach().cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _mlp_exact(case, seed)
    if kind == "ritz":
        band, T = _band(case, seed)
        w, S = np.linalg.eigh(T.cpu().numpy())
        w, S = w[:case["nev"]], S[:, :case["nev"]]
        k = np.argmax(np.abs(S), axis=0)
        return {"theta": w.copy(), "S": S * np.sign(S[k, np.arange(S.shape[1])])}
    if kind == "batch":
        ev = [_lowest(_matrix(c, _spawn(seed, i), "f32"), case["b"], case["b"], 1e-10) for i, c in enumerate(_batch_cases(case, seed))]
        return {"evals": None if any(v is None for v in ev) else np.stack(ev), "status": None}
    if kind == "solve":
        return {"evals": _lowest(_matrix(case, seed, case["dtype"]), case["b"], case["b"], 1e-10), "evecs": None}
    g = _gen(seed + 500009)
    if kind == "spmm":
        c = _matrix(case, seed, case["dtype"])
        t = torch.float64 if case["dtype"] == "f64" else torch.float32
        return _times(c, torch.randn(c.n, case["b"], generator=g, device=DEV, dtype=t).double())
    if kind == "kron":
        nP, nN, b = case["nP"], case["nN"], case["b"]
        hp, hn, cp, cn = _factors(case, seed)
        t = torch.float64 if case["dtype"] == "f64" else torch.float32
        V = torch.randn(nP * nN, b, generator=g, device=DEV, dtype=t).double().reshape(nP, nN * b)
        dense = lambda f, N: torch.zeros(N, N, dtype=torch.float64, device=DEV).index_put_((f[0], f[1]), f[2])  # noqa: E731
        right = lambda f, X: torch.matmul(dense(f, nN), X.reshape(nP, nN, b)).reshape(nP, nN * b)  # noqa: E731
        W = dense(hp, nP) @ V + right(hn, V)
        for a, c in zip(cp, cn):
            W = W + right(c, dense(a, nP) @ V)
        return W.reshape(nP * nN, b)
    if kind == "cholqr2":
        W = prepare(case, seed)["W"].double()
        for k in range(2):
            R = torch.linalg.cholesky(W.T @ W, upper=True)
            W = W @ torch.linalg.inv(R)
            B = R if k == 0 else R @ B
        return {"Q": W, "B": B, "defl": None}
    if kind in ("reorth", "f16"):
        s = prepare(case, seed)
        b = s["W"].shape[1]
        W = s["W"].double()
        Q = s["Q"].permute(1, 0, 2).reshape(s["W"].shape[0], -1).double()
        if kind == "f16":
            C = Q.T @ W  # the FP16 copy stands for the basis
            return {"W": W - Q @ C, "C": C}
        C1 = Q.T @ W
        W = W - Q @ C1
        C2 = Q.T @ W
        return {"W": W - Q @ C2, "C": torch.stack([C1, C2])}
    return None
