"""The workloads this framework's speed is judged by.

Each case is one thing a user has the framework do, through the functions of
``paper_1509_09313_gb300``: whole factorisations on a handle, the paper's three
local tasks (Gram, MM, NLS) on their own, the MU and HALS updates, the sparse
product, and one gradient of the learned starting partitions. ``listed()`` has
the fixed cases, ``draw()`` makes more of the same ranges, ``prepare()`` /
``run()`` / ``work()`` / ``exact()`` serve both. A case is a plain dict whose
``kind`` names one of the families below.
"""
from __future__ import annotations

import math

import torch

import paper_1509_09313_gb300 as nmf

DEVICE = "cuda"

# Largest sizes of a family: no drawn case costs more than the largest listed one.
MN_MAX = 24000 * 16000      # elements of a dense A
NLS_MAX = 1000000 * 100     # right-hand sides x k of one batched NLS call
NNZ_MAX = 10000000          # position draws of a sparse matrix


def listed():
    return [
        # A whole small factorisation (bench.py's 2000 x 1000, k = 10, plain FP32): five
        # warm-started iterations from a random start, factors and objective read back.
        # Launches and small kernels count here.
        {"name": "anls_small", "kind": "anls", "input": "dense", "m": 2000, "n": 1000, "k": 10,
         "precision": "fp32", "solver": "bpp", "start": "warm", "iters": 5, "sigma": 0.01,
         "near": False},
        # A dense factorisation in the default tensor-core precision (bench.py's
        # dense-medium, 1.5 GB of A), resumed from factors on their way to the solution, as
        # most of a run's iterations are: the framework's main path.
        {"name": "anls_dense", "kind": "anls", "input": "dense", "m": 24000, "n": 16000, "k": 50,
         "precision": "bf16x3", "solver": "bpp", "start": "warm", "iters": 3, "sigma": 0.05,
         "near": True},
        # A whole sparse factorisation (bench.py's sparse-medium), where the batched NLS
        # solves are nearly all the time.
        {"name": "anls_sparse", "kind": "anls", "input": "csr", "m": 200000, "n": 100000,
         "k": 50, "draws": 2000000, "precision": "fp32", "solver": "bpp", "start": "warm",
         "iters": 3},
        # One half-step from its parts (Gram, product, NLS) as a program that distributes
        # the matrix itself would call them, on a ragged block of A: the H update, tensor cores.
        {"name": "half_step_ragged", "kind": "half", "m": 6007, "n": 3004, "k": 33,
         "trans": True, "precision": "bf16x3"},
        # One call on a few right-hand sides, everything it reports: a latency-bound user.
        {"name": "nls_small", "kind": "nls", "k": 20, "nrhs": 500, "mean": 0.05, "spread": 0.0,
         "warm": False, "outputs": True},
        # The H update of a dense run's first iterations (16000 columns): W's columns are still
        # nearly parallel, so the solves run in FP64.
        {"name": "nls_early", "kind": "nls", "k": 50, "nrhs": 16000, "mean": 0.05,
         "spread": 0.02, "warm": True, "outputs": False},
        # bench.py's stress batch with solutions of mixed signs: exchanges, systems of all sizes.
        {"name": "nls_mixed", "kind": "nls", "k": 100, "nrhs": 1000000, "mean": 0.05,
         "spread": 0.0, "warm": False, "outputs": False},
        # bench.py's stress batch: every solution positive, one full exchange each.
        {"name": "nls_positive", "kind": "nls", "k": 100, "nrhs": 1000000, "mean": 0.5,
         "spread": 0.0, "warm": False, "outputs": False},
        # The other local updates (HALS here, MU among the drawn cases) on the W rows of the
        # 96000 x 64000 workload.
        {"name": "update_hals", "kind": "update", "solver": "hals", "rows": 96000, "k": 50},
        # The plain FP32 product of a dense half-step, A H^T.
        {"name": "mm_fp32", "kind": "mm", "m": 24000, "n": 16000, "k": 50, "trans": False,
         "precision": "fp32"},
        # The sparse product with a factor larger than the L2 cache.
        {"name": "spmm", "kind": "spmm", "rows": 1000000, "cols": 1000000, "draws": 10000000,
         "k": 50},
        # One training gradient of the network that proposes starting partitions (its
        # default batch and width).
        {"name": "mlp_gradient", "kind": "mlp", "nrhs": 8192, "k": 50, "hidden": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["anls", "anls", "half", "nls", "nls", "nls", "update", "update", "mm", "mm",
                       "spmm", "mlp"])
    if kind == "anls":
        if rng.random() < 0.5:
            near = rng.random() < 0.7
            k = rng.randint(4, 64 if near else 12)
            precision = rng.choice(["fp32", "bf16x3"])
            m = _log(rng, 30 * k, 24000)
            n = _log(rng, 30 * k, 12000)
            if precision == "bf16x3":
                n = (n + 3) // 4 * 4           # TMA: a row stride of whole 16-byte pieces
            return {"kind": kind, "input": "dense", "m": m, "n": n, "k": k,
                    "precision": precision, "solver": rng.choice(["bpp", "bpp", "mu", "hals"]),
                    "start": rng.choice(["warm", "cold"]),
                    "iters": rng.randint(2, 3) if near else rng.randint(5, 8),
                    "sigma": 0.05, "near": near}
        m, n = _log(rng, 20000, 200000), _log(rng, 20000, 100000)
        return {"kind": kind, "input": "csr", "m": m, "n": n, "k": rng.randint(4, 50),
                "draws": 10 * m, "precision": "fp32", "solver": "bpp",
                "start": rng.choice(["warm", "cold"]), "iters": rng.randint(2, 3)}
    if kind == "half":
        k = rng.randint(4, 100)
        precision = rng.choice(["fp32", "bf16x3"])
        m, n = _log(rng, 30 * k, 12000), _log(rng, 30 * k, 12000)
        if precision == "bf16x3":
            n = (n + 3) // 4 * 4
        return {"kind": kind, "m": m, "n": n, "k": k, "trans": rng.random() < 0.5,
                "precision": precision}
    if kind == "nls":
        k = rng.randint(4, 128)
        outputs, early = rng.random() < 0.3, rng.random() < 0.2
        most = 2000 if outputs else 16000 if early else NLS_MAX // 128
        return {"kind": kind, "k": k, "nrhs": _log(rng, 100, most),
                "mean": rng.choice([0.02, 0.05, 0.1, 0.5]), "spread": 0.02 if early else 0.0,
                "warm": rng.random() < 0.5, "outputs": outputs}
    if kind == "update":
        return {"kind": kind, "solver": rng.choice(["mu", "hals"]),
                "rows": _log(rng, 1000, 1000000), "k": rng.randint(4, 100)}
    if kind == "mm":
        k = rng.randint(4, 100)
        precision = rng.choice(["fp32", "fp32", "bf16x3"])
        m = _log(rng, 500, 24000)
        n = _log(rng, 500, min(16000, MN_MAX // m))
        if precision == "bf16x3":
            n = (n + 3) // 4 * 4
        return {"kind": kind, "m": m, "n": n, "k": k, "trans": rng.random() < 0.5,
                "precision": precision}
    if kind == "spmm":
        return {"kind": kind, "rows": _log(rng, 5000, 1000000), "cols": _log(rng, 5000, 1000000),
                "draws": _log(rng, 50000, NNZ_MAX), "k": rng.randint(4, 64)}
    return {"kind": kind, "nrhs": _log(rng, 500, 8192), "k": rng.randint(8, 50), "hidden": 256}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed) * 7919 + 12345)
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEVICE, dtype=torch.float32)


def _randn(g, *shape, dtype=torch.float32):
    return torch.randn(shape, generator=g, device=DEVICE, dtype=dtype)


def _dense(g, m, n, k, sigma):
    """A = W0 H0 + |N(0, sigma^2)|, W0 and H0 uniform: the paper's dense synthetic recipe.
    Returns (A, W0, H0)."""
    w0, h0 = _rand(g, m, k), _rand(g, k, n)
    a = torch.empty((m, n), dtype=torch.float32, device=DEVICE)
    step = max(1, (1 << 27) // n)
    for r in range(0, m, step):
        e = min(m, r + step)
        a[r:e] = w0[r:e] @ h0 + (sigma * _randn(g, e - r, n)).abs_()
    return a, w0, h0


def _csr(g, rows, cols, draws):
    """Uniform positions (duplicates merged), values in (0, 1]: the paper's sparse recipe."""
    key = torch.randint(rows * cols, (draws,), generator=g, device=DEVICE, dtype=torch.int64)
    key = torch.unique(key)
    r = key // cols
    colidx = (key - r * cols).to(torch.int32)
    rowptr = torch.zeros(rows + 1, dtype=torch.int64, device=DEVICE)
    rowptr[1:] = torch.cumsum(torch.bincount(r, minlength=rows), 0)
    vals = 1.0 - _rand(g, key.numel())
    return rowptr, colidx, vals


def _gram_and_rhs(g, k, nrhs, mean, spread):
    """The stress recipe: G = W^T W of W uniform with 30% zeros (or, with a spread, of
    W = 1 + N(0, spread^2): nearly parallel columns), and right-hand sides distributed
    like W^T a with a = u + mean - 1/2, u uniform in [0, 1)."""
    rows = 2000 * k
    if spread:
        w = 1.0 + spread * _randn(g, rows, k, dtype=torch.float64)
    else:
        w = (_rand(g, rows, k) * (_rand(g, rows, k) >= 0.3)).double()
    gram = w.T @ w
    low = torch.linalg.cholesky(gram.cpu()).to(DEVICE)
    lead = mean * w.sum(0)
    b = torch.empty((nrhs, k), dtype=torch.float32, device=DEVICE)
    step = 250000
    for r in range(0, nrhs, step):
        e = min(nrhs, r + step)
        b[r:e] = (lead + _randn(g, e - r, k, dtype=torch.float64) @ low.T / math.sqrt(12.0)).float()
    return gram.contiguous(), b


def _pack(passive):
    """Boolean rows to the library's 64-bit words."""
    return nmf.bool_to_passive(passive).contiguous()


def _inputs(case, seed):
    """The tensors a case starts from (the same for run() and exact())."""
    g, kind = _gen(seed), case["kind"]
    k = case["k"]
    if kind == "anls":
        m, n = case["m"], case["n"]
        if case["input"] == "csr":
            return {"A": _csr(g, m, n, case["draws"]), "W0": _rand(g, m, k),
                    "Ht0": _rand(g, n, k)}
        a, w0, h0 = _dense(g, m, n, k, case["sigma"])
        w, ht = _rand(g, m, k), _rand(g, n, k)
        if case["near"]:
            w, ht = 0.7 * w0 + 0.3 * w, 0.7 * h0.T + 0.3 * ht
        return {"A": a, "W0": w.contiguous(), "Ht0": ht.contiguous()}
    if kind in ("half", "mm"):
        m, n = case["m"], case["n"]
        return {"A": _dense(g, m, n, k, 0.05)[0], "F": _rand(g, m if case["trans"] else n, k)}
    if kind == "nls":
        gram, b = _gram_and_rhs(g, k, case["nrhs"], case["mean"], case["spread"])
        # A warm start: the signs of the unconstrained solution, as a previous nearby
        # solve would leave them.
        pin = None
        if case["warm"]:
            pin = b.double() @ torch.linalg.inv(gram.cpu()).to(DEVICE) > 0
        return {"G": gram, "B": b, "pin": pin}
    if kind == "update":
        # The first iterations of W >= 0, W H ~ A: G = H H^T, R = A H^T.
        rows = case["rows"]
        h = _rand(g, 2000, k).double()
        gram = (h.T @ h).contiguous()
        true = _rand(g, rows, k) * (_rand(g, rows, k) >= 0.1)
        r = (true @ gram.float()) * (1.0 + 0.01 * _rand(g, rows, k))
        return {"G": gram, "R": r.contiguous(), "X": _rand(g, rows, k)}
    if kind == "spmm":
        return {"S": _csr(g, case["rows"], case["cols"], case["draws"]),
                "F": _rand(g, case["cols"], k)}
    # mlp: features as the network sees them (scaled gradient, log diagonal, scaled
    # iterate), labels of mixed signs, Glorot-uniform weights.
    nrhs, hid = case["nrhs"], case["hidden"]
    feat = torch.cat([0.3 * _randn(g, nrhs, k), (0.1 * _randn(g, 1, k)).expand(nrhs, k),
                      _rand(g, nrhs, k)], dim=1).contiguous()
    parts = []
    for rows, cols in ((hid, 3 * k), (hid, 1), (hid, hid), (hid, 1), (k, hid), (k, 1)):
        lim = math.sqrt(6.0 / (rows + cols)) if cols > 1 else 0.05
        parts.append((2.0 * _rand(g, rows * cols) - 1.0) * lim)
    label = feat[:, :k] + 0.2 * _randn(g, nrhs, k) < 0.1
    return {"F": feat, "params": torch.cat(parts), "label": label}


class _State:
    pass


def prepare(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    s = _State()
    s.case = case
    if kind == "anls":
        s.W0, s.Ht0 = x["W0"], x["Ht0"]
        shape = (case["m"], case["n"]) if case["input"] == "csr" else None
        s.handle = nmf.nmf_init(x["A"], s.W0, s.Ht0, precision=case["precision"],
                                start=case["start"], solver=case["solver"], shape=shape)
    elif kind == "mlp":
        s.F, s.passive = x["F"], _pack(x["label"])
        s.net = nmf.nmf_mlp_create(case["k"], case["hidden"], x["params"])
    else:
        for name, v in x.items():
            setattr(s, name, v)
        if kind == "nls":
            s.pin = None if x["pin"] is None else _pack(x["pin"])
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "anls":
        # A factorisation from a given start: iterate, then read the factors and the
        # objective of every iteration.
        h = s.handle
        h.nmf_set_factors(s.W0, s.Ht0)
        h.nmf_iterate(case["iters"])
        status = h.nmf_sync()
        w, ht = h.nmf_get_factors()
        return {"W": w, "Ht": ht, "f": h.nmf_objective_history(case["iters"]), "status": status}
    if kind == "half":
        gram = nmf.nmf_gram(s.F)
        v = nmf.nmf_mm_dense(s.A, s.F, case["trans"], case["precision"])
        r = nmf.nmf_nls_bpp(gram, v, outputs=False)
        return {"V": v, "X": r["X"], "worst": r["worst"]}
    if kind == "nls":
        r = nmf.nmf_nls_bpp(s.G, s.B, passive_in=s.pin, outputs=case["outputs"])
        return {name: v for name, v in r.items() if v is not None}
    if kind == "update":
        fn = nmf.nmf_update_mu if case["solver"] == "mu" else nmf.nmf_update_hals
        return fn(s.G, s.R, s.X)
    if kind == "mm":
        return nmf.nmf_mm_dense(s.A, s.F, case["trans"], case["precision"])
    if kind == "spmm":
        return nmf.nmf_mm_csr(*s.S, case["cols"], s.F)
    grad, loss = s.net.nmf_mlp_gradient(s.F, s.passive)
    return {"grad": grad, "loss": loss.float()}


def work(case):
    """Bytes: each input read once and each output written once (a factorisation reads A
    for each of its two products an iteration). Flops: the products and, per right-hand
    side of an NLS, one solve with its passive set taken as half of k."""
    kind, k = case["kind"], case["k"]

    def nls_flops(rhs):
        f = k / 2
        return rhs * (f ** 3 / 3 + 2 * f * k)

    if kind == "anls":
        m, n, it = case["m"], case["n"], case["iters"]
        size = 8.0 * case["draws"] if case["input"] == "csr" else 4.0 * m * n
        mul = (2.0 * case["draws"] if case["input"] == "csr" else 2.0 * m * n) * k
        local = nls_flops(m + n) if case["solver"] == "bpp" else 2.0 * (m + n) * k * k
        return {"bytes": it * (2 * size + 8.0 * (m + n) * k),
                "flops": it * (2 * mul + 2.0 * (m + n) * k * k + local)}
    if kind in ("half", "mm"):
        m, n = case["m"], case["n"]
        p, q = (n, m) if case["trans"] else (m, n)
        b, f = 4.0 * m * n + 4.0 * (m + n) * k, 2.0 * m * n * k
        if kind == "half":
            b, f = b + 4.0 * p * k, f + 2.0 * q * k * k + nls_flops(p)
        return {"bytes": b, "flops": f}
    if kind == "nls":
        return {"bytes": 8.0 * case["nrhs"] * k + 8.0 * k * k, "flops": nls_flops(case["nrhs"])}
    if kind == "update":
        return {"bytes": 12.0 * case["rows"] * k + 8.0 * k * k,
                "flops": 2.0 * case["rows"] * k * k}
    if kind == "spmm":
        return {"bytes": 8.0 * case["draws"] + 8.0 * case["rows"]
                + 4.0 * (case["rows"] + case["cols"]) * k, "flops": 2.0 * case["draws"] * k}
    hid = case["hidden"]
    weights = 3.0 * k * hid + hid * hid + hid * k
    return {"bytes": 12.0 * case["nrhs"] * k + 8.0 * weights,
            "flops": 6.0 * case["nrhs"] * weights - 2.0 * case["nrhs"] * 3 * k * hid}


# ---------------------------------------------------------------- 64 bits
def _nls64(gram, b, passive=None):
    """argmin_{x >= 0} 0.5 x^T G x - b^T x for each row of b, in FP64: block principal
    pivoting with masked Cholesky solves. Returns (X, passive, rounds)."""
    nrhs, k = b.shape
    x_all = torch.zeros((nrhs, k), dtype=torch.float64, device=b.device)
    p_all = torch.zeros((nrhs, k), dtype=torch.bool, device=b.device)
    r_all = torch.zeros(nrhs, dtype=torch.int32, device=b.device)
    low = torch.linalg.cholesky(gram)
    eye = torch.eye(k, dtype=torch.float64, device=b.device)
    chunk = max(1, int(1.5e9 // (8 * k * k)))

    def candidate(f, rhs):
        x = torch.zeros_like(rhs)
        whole = f.all(1)
        if bool(whole.any()):
            x[whole] = torch.cholesky_solve(rhs[whole].T, low).T
        part = torch.nonzero(~whole & f.any(1)).squeeze(1)
        for c in part.split(chunk):
            fc = f[c].double()
            mat = gram * fc[:, :, None] * fc[:, None, :] + eye * (1.0 - fc)[:, :, None]
            fac = torch.linalg.cholesky_ex(mat)[0]
            x[c] = torch.cholesky_solve((rhs[c] * fc)[:, :, None], fac).squeeze(2) * fc
        return x

    live = torch.arange(nrhs, device=b.device)
    f = passive.clone() if passive is not None else torch.zeros_like(p_all)
    alpha = torch.full((nrhs,), 3, device=b.device)
    beta = torch.full((nrhs,), k + 1, device=b.device)
    for rounds in range(200):
        rhs = b[live]
        x = candidate(f, rhs)
        y = x @ gram - rhs
        bad = torch.where(f, x < 0, y < 0)
        count = bad.sum(1)
        done = count == 0
        at = live[done]
        x_all[at], p_all[at], r_all[at] = x[done], f[done], rounds
        keep = ~done
        live, f, bad, count = live[keep], f[keep], bad[keep], count[keep]
        alpha, beta = alpha[keep], beta[keep]
        if live.numel() == 0:
            break
        drop = count < beta
        full = drop | (alpha >= 1)
        alpha = torch.where(drop, torch.full_like(alpha, 3), alpha - full.long())
        beta = torch.where(drop, count, beta)
        top = k - 1 - bad.flip(1).to(torch.int8).argmax(1)
        single = torch.zeros_like(bad)
        single[torch.arange(live.numel(), device=b.device), top] = True
        f = f ^ torch.where(full[:, None], bad, single)
    return x_all, p_all, r_all


def _update64(solver, gram, r, x):
    x = x.double()
    r = r.double()
    if solver == "mu":
        den = x @ gram
        return torch.where(den > 0, x * r / den, x)
    x = x.T.contiguous()
    for i in range(gram.shape[0]):
        rest = gram[i] @ x - gram[i, i] * x[i]
        x[i] = ((r[:, i] - rest) / gram[i, i]).clamp_min(0.0)
    return x.T.contiguous()


def _csr64(s, rows, cols, f):
    rowptr, colidx, vals = s
    row = torch.repeat_interleave(torch.arange(rows, device=f.device), rowptr.diff())
    out = torch.zeros((rows, f.shape[1]), dtype=torch.float64, device=f.device)
    for c in torch.arange(vals.numel(), device=f.device).split(4000000):
        out.index_add_(0, row[c], vals[c].double()[:, None] * f[colidx[c].long()])
    return out


def _product64(a, f, trans):
    step = max(1, (1 << 27) // a.shape[1])
    if not trans:
        return torch.cat([blk.double() @ f for blk in a.split(step)])
    out = torch.zeros((a.shape[1], f.shape[1]), dtype=torch.float64, device=f.device)
    for blk, fb in zip(a.split(step), f.split(step)):
        out += blk.double().T @ fb
    return out


def exact(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "anls":
        a, m, n, solver = x["A"], case["m"], case["n"], case["solver"]
        w, ht, hist = x["W0"].double(), x["Ht0"].double(), []
        if case["input"] == "csr":
            rowptr, colidx, vals = a
            row = torch.repeat_interleave(torch.arange(m, device=DEVICE), rowptr.diff())
            order = torch.argsort(colidx.long() * m + row)
            t_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
            t_ptr[1:] = torch.cumsum(torch.bincount(colidx.long(), minlength=n), 0)
            t = (t_ptr, row[order].to(torch.int32), vals[order])
            sq = vals.double().square().sum()
        for _ in range(case["iters"]):
            for side in ("W", "H"):
                fixed = ht if side == "W" else w
                if case["input"] == "csr":
                    v = _csr64(a, m, n, ht) if side == "W" else _csr64(t, n, m, w)
                else:
                    v = _product64(a, fixed, side == "H")
                gram = fixed.T @ fixed
                if solver == "bpp":
                    new = _nls64(gram, v)[0]
                else:
                    new = _update64(solver, gram, v, w if side == "W" else ht)
                if side == "W":
                    w = new
                else:
                    ht = new
            if case["input"] == "csr":
                f = sq - 2.0 * (ht * v).sum() + (gram * (ht.T @ ht)).sum()
            else:
                step = max(1, (1 << 27) // n)
                f = sum((blk.double() - wb @ ht.T).square().sum()
                        for blk, wb in zip(a.split(step), w.split(step)))
            hist.append(float(f))
        return {"W": w, "Ht": ht, "f": hist, "status": 0}
    if kind in ("half", "mm"):
        fac = x["F"].double()
        v = _product64(x["A"], fac, case["trans"])
        if kind == "mm":
            return v
        return {"V": v, "X": _nls64(fac.T @ fac, v)[0], "worst": 0}
    if kind == "nls":
        sol = _nls64(x["G"], x["B"].double(), x["pin"])[0]
        out = {"X": sol, "worst": 0}
        if case["outputs"]:
            out.update(passive=None, rounds=None, status=None)
        return out
    if kind == "update":
        return _update64(case["solver"], x["G"], x["R"], x["X"])
    if kind == "spmm":
        return _csr64(x["S"], case["rows"], case["cols"], x["F"].double())
    k, hid = case["k"], case["hidden"]
    shapes = ((hid, 3 * k), (hid, 1), (hid, hid), (hid, 1), (k, hid), (k, 1))
    parts = x["params"].split([r * c for r, c in shapes])
    q = [(p if c == 1 else p.bfloat16().double().reshape(r, c)).double().requires_grad_()
         for p, (r, c) in zip(parts, shapes)]
    z = torch.relu(x["F"].double() @ q[0].T + q[1])
    z = torch.relu(z @ q[2].T + q[3])
    z = z @ q[4].T + q[5]
    loss = torch.nn.functional.binary_cross_entropy_with_logits(z, x["label"].double())
    loss.backward()
    return {"grad": torch.cat([p.grad.reshape(-1) for p in q]), "loss": loss.detach().reshape(1)}
