"""The work a user of the library has it do, as cases with sizes, inputs and
64-bit references: sketches of a vector, basis products on the tensor cores,
randomized QR of a block, restarts of the eigensolver on regular, irregular
and mixed-precision problems, a batch of uneven problems in one persistent
launch, and the start-vector network forward and backward.

``listed()`` gives the fixed cases, ``draw(rng)`` more of the same ranges.
``prepare`` makes what a program holds before the call (inputs and handles),
``run`` is one pass through the public entry points, ``exact`` the same
outputs in plain 64-bit torch or numpy.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_05400_gb300 import inputs, rks

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: the sketch of one short vector (latency counts)
        dict(name="sketch_20k", kind="sketch", n=20_000, d=80, zeta=4),
        # the sketch of a vector of the 160^3 problem
        dict(name="sketch_4m", kind="sketch", n=4_096_000, d=600, zeta=8),
        # the restart product of a 1000 x 1000 problem (80 columns, 20 kept), double-float
        dict(name="product_df_1m", kind="product", prec="df", n=1_000_000, nin=80, nout=21),
        # the restart product of the 160^3 problem, FP32 basis
        dict(name="product_f32_4m", kind="product", prec="f32", n=4_096_000, nin=150, nout=51),
        # randomized Gram-Schmidt of a tall block
        dict(name="qr_rgs_1m", kind="qr", method="rgs", n=1_000_000, s=80, d=320, zeta=8),
        # randomized Cholesky QR of a narrow block with ragged rows
        dict(name="qr_rcholqr_50k", kind="qr", method="rcholqr", n=50_021, s=24, d=96, zeta=8),
        # the first restarts on a small tridiagonal problem (Table 1 of the
        # paper): kernels of microseconds, launches and host steps count
        dict(name="solve_tridiag_2k", kind="solve", op="tridiag", n=2000, k=10, p=30, d=80, zeta=4, which="LM",
             prec="df", keep=10, restarts=3),
        # the first restart of the 1000 x 1000 convection-diffusion problem
        dict(name="solve_2d_1m", kind="solve", op="conv2d", nx=1000, ny=1000, k=20, p=60, d=320, zeta=8, which="LR",
             prec="df", keep=20, restarts=1),
        # rows of 1 to 10^4 entries: the matrices of large sparse collections
        dict(name="solve_powerlaw_100k", kind="solve", op="powerlaw", n=100_003, k=8, p=32, d=128, zeta=8, which="LR",
             prec="df", keep=8, restarts=1),
        # the largest eigenvalues of the 160^3 problem to a few digits in mixed
        # precision (the bound an explicit time step needs): the FP32 basis
        dict(name="solve_3d_mixed_4m", kind="solve", op="conv3d", nx=160, ny=160, nz=160, k=6, p=24, d=96, zeta=8,
             which="LM", prec="mixed", keep=6, restarts=2),
        # half of the batch of 256 uneven 2D problems, two restarts each
        dict(name="batch_128", kind="batch", count=128, lo=70, hi=450, k=8, p=24, d=64, zeta=8, keep=12, restarts=2,
             sizes=1000),
        # gradients of a minibatch of the start-vector network on the 512 x 512 family
        dict(name="network_grad_512", kind="network", mode="grad", H=512, W=512, q=16, batch=2),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sketch", "product", "qr", "solve", "solve", "solve", "batch", "network"])
    if kind == "sketch":
        zeta = rng.choice([4, 8])
        return dict(kind=kind, n=_logint(rng, 2000, 4_096_000), d=_logint(rng, 64, 600), zeta=zeta)
    if kind == "product":
        prec = rng.choice(["df", "f32"])
        nin = rng.randint(24, 150)
        return dict(kind=kind, prec=prec, n=_logint(rng, 10_000, 2_000_000), nin=nin,
                    nout=rng.randint(4, min(51, nin - 2)))
    if kind == "qr":
        s = rng.randint(8, 80)
        return dict(kind=kind, method=rng.choice(["rgs", "whiten", "rcholqr", "rhqr"]), s=s,
                    n=_logint(rng, 20_000, 1_000_000), d=rng.randint(3 * s, 4 * s) + 8, zeta=8)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(16, 96), lo=70, hi=rng.randint(150, 450), k=8, p=24, d=64, zeta=8,
                    keep=12, restarts=rng.randint(1, 2), sizes=rng.randint(1, 10_000))
    if kind == "network":
        return dict(kind=kind, mode=rng.choice(["forward", "grad"]), H=8 * rng.randint(8, 64), W=8 * rng.randint(8, 64),
                    q=rng.randint(4, 16), batch=rng.randint(1, 2))
    op = rng.choice(["tridiag", "conv2d", "conv2d", "conv3d", "powerlaw", "wide"])
    if op == "tridiag":
        return dict(kind=kind, op=op, n=_logint(rng, 1000, 100_000), k=10, p=30, d=80, zeta=rng.choice([4, 8]),
                    which="LM", prec=rng.choice(["df", "fp64"]), keep=10, restarts=rng.randint(1, 3))
    if op == "conv2d":
        k = rng.choice([8, 16, 20])
        return dict(kind=kind, op=op, nx=rng.randint(70, 900), ny=rng.randint(70, 900), k=k, p=3 * k,
                    d=rng.randint(8 * k, 16 * k), zeta=8, which="LR", prec=rng.choice(["df", "df", "fp64"]), keep=k,
                    restarts=rng.randint(1, 2))
    if op == "conv3d":
        shape = {a: rng.randint(30, 100) for a in ("nx", "ny", "nz")}
        if rng.random() < 0.5:
            return dict(kind=kind, op=op, **shape, k=6, p=24, d=96, zeta=8, which="LM", prec="mixed", keep=6,
                        restarts=2)
        k = rng.choice([8, 16])
        return dict(kind=kind, op=op, **shape, k=k, p=3 * k, d=12 * k, zeta=8, which="LR", prec="df", keep=k,
                    restarts=1)
    n = _logint(rng, 20_000, 300_000)
    return dict(kind=kind, op=op, n=n, k=8, p=32, d=128, zeta=8, which="LR", prec=rng.choice(["df", "df", "fp64"]),
                keep=8, restarts=1)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _stencil(shape, nu, b):
    """CSR (int32, float64) of div(nu grad u) - b . grad u on the unit box,
    Dirichlet, first-order upwind: ``shape`` and ``nu`` with x last, ``b`` and
    the unknowns with x first."""
    dims = len(shape)
    strides = [1]
    for a in range(1, dims):
        strides.append(strides[-1] * shape[dims - a])
    n = nu.numel()
    p = torch.arange(n, device=DEV)
    lows, highs = [], []
    diag = torch.zeros(n, dtype=torch.float64, device=DEV)
    for a in range(dims):
        ax, sz = dims - 1 - a, shape[dims - 1 - a]
        h = 1.0 / (sz + 1)
        x = (p // strides[a]) % sz
        f = 2.0 * nu.narrow(ax, 1, sz - 1) * nu.narrow(ax, 0, sz - 1)
        f = f / (nu.narrow(ax, 1, sz - 1) + nu.narrow(ax, 0, sz - 1))
        lo = torch.cat([nu.narrow(ax, 0, 1), f], dim=ax).reshape(-1)
        hi = torch.cat([f, nu.narrow(ax, sz - 1, 1)], dim=ax).reshape(-1)
        lows.append((-strides[a], lo / h**2 + b[a] / h, x > 0))
        highs.append((strides[a], hi / h**2, x < sz - 1))
        diag -= (lo + hi) / h**2 + b[a] / h
    parts = lows[::-1] + [(0, diag, torch.ones(n, dtype=torch.bool, device=DEV))] + highs   # increasing columns
    keep = torch.stack([m for _, _, m in parts], dim=1)
    cols = torch.stack([p + o for o, _, _ in parts], dim=1)[keep]
    vals = torch.stack([v for _, v, _ in parts], dim=1)[keep]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(keep.sum(dim=1), 0)
    return rowptr.int(), cols.int(), vals


def _random_rows(n, g, lens):
    """Rows of ``lens`` entries at random columns (N(0,1) / (2 sqrt(len))) and a diagonal in [0, 2)."""
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), lens)
    cols = torch.randint(0, n, (rows.numel(),), generator=g, device=DEV)
    key = torch.unique(rows * n + cols)
    key = key[key // n != key % n]
    rows = key // n
    vals = _randn(g, key.numel()) * (0.5 / lens[rows].double().sqrt())
    diag = 2.0 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    key = torch.cat([key, torch.arange(n, device=DEV) * (n + 1)])
    vals = torch.cat([vals, diag])
    order = torch.argsort(key)
    key, vals = key[order], vals[order]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return rowptr.int(), (key % n).int(), vals


def _operator(case, g):
    op = case["op"]
    if op == "conv2d":
        nu = torch.exp(_randn(g, case["ny"], case["nx"]) * 0.25)
        return _stencil((case["ny"], case["nx"]), nu, (20.0, 10.0))
    if op == "conv3d":
        shape = (case["nz"], case["ny"], case["nx"])
        rp, ci, v = _stencil(shape, torch.exp(_randn(g, *shape)), (10.0, 5.0, 2.0))
        return rp, ci, v.float()
    n = case["n"]
    if op == "tridiag":
        t = torch.linspace(2.0, 10.0, n, dtype=torch.float64, device=DEV)
        band = torch.stack([_randn(g, n) / 100.0, torch.exp(t / 10.0), _randn(g, n) / 100.0], dim=1)
        cols = torch.arange(n, device=DEV)[:, None] + torch.arange(-1, 2, device=DEV)[None, :]
        keep = (cols >= 0) & (cols < n)
        rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        rowptr[1:] = torch.cumsum(keep.sum(dim=1), 0)
        return rowptr.int(), cols[keep].int(), band[keep]
    if op == "powerlaw":
        u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64).clamp_min(1e-300)
        lens = torch.clamp((u ** (-1.0 / 1.2)).floor(), 1, 10_000).long()
        return _random_rows(n, g, lens)
    lens = torch.randint(32, 49, (n,), generator=g, device=DEV)
    return _random_rows(n, g, lens)


def _solve_opts(case):
    """Convergence settings: residuals of 1e-2 (mixed precision, a fixed
    number of restarts) or 1e-8 on the ||A||_1 scale for the
    convection-diffusion operators, |b^T y| <= 1e-10 |lambda| otherwise."""
    if case["prec"] == "mixed":
        return dict(tol=1e-6, conv="norm1", verify=1e-2)
    if case["op"] in ("conv2d", "conv3d"):
        return dict(tol=0.25e-8, eta_lock=0.125e-8, conv="norm1", verify=1e-8)
    return dict(tol=1e-10, conv="eig")


def _batch_problems(case, seed):
    """(nx, ny, b, nu) of every problem: sides and convection from the case's own sizes, diffusivities from the seed."""
    g = _gen(seed)
    r = np.random.RandomState(case["sizes"])
    out = []
    for _ in range(case["count"]):
        nx, ny = (int(v) for v in r.randint(case["lo"], case["hi"] + 1, 2))
        b = tuple(float(v) for v in 30.0 * r.rand(2))
        out.append((nx, ny, b, torch.exp(_randn(g, ny, nx))))
    return out


def _network_inputs(case, seed):
    """Smooth log-diffusivity fields, constant convections, and orthonormal columns Q (q x H W)."""
    g = _gen(seed)
    H, W, q = case["H"], case["W"], case["q"]
    xs, qs = [], []
    for _ in range(case["batch"]):
        f = _randn(g, 1, 1, H // 8, W // 8, dtype=torch.float32)
        f = torch.nn.functional.interpolate(f, size=(H, W), mode="bicubic", align_corners=False)[0, 0]
        x = torch.empty(3, H, W, dtype=torch.float32, device=DEV)
        x[0], x[1:] = f, torch.rand(2, 1, 1, generator=g, device=DEV)
        y = (torch.arange(H, device=DEV, dtype=torch.float64) + 1.0)[:, None] / (H + 1)
        z = (torch.arange(W, device=DEV, dtype=torch.float64) + 1.0)[None, :] / (W + 1)
        modes = [torch.sin((1 + j // 4) * math.pi * y) * torch.sin((1 + j % 4) * math.pi * z) for j in range(q)]
        modes = torch.stack(modes).reshape(q, -1) * (2.0 / math.sqrt((H + 1) * (W + 1)))   # orthonormal
        R = np.linalg.qr(np.random.RandomState((int(seed) + len(xs)) % 2**31).randn(q, q))[0]
        xs.append(x)
        qs.append((torch.from_numpy(R).to(DEV) @ modes).float().contiguous())
    return xs, qs


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    if kind == "sketch":
        return dict(case=case, x=_randn(g, case["n"]), seed=int(seed) % 1000)
    if kind == "product":
        n, nin, nout = case["n"], case["nin"], case["nout"]
        ldu = (n + 31) // 32 * 32
        dt = torch.float32 if case["prec"] == "f32" else torch.float64
        U = torch.zeros(nin, ldu, dtype=dt, device=DEV)
        U[:, :n] = _randn(g, nin, n, dtype=dt)
        Q = np.linalg.qr(np.random.RandomState(int(seed) % 2**31).randn(nin, nin))[0][:, :nout]
        return dict(case=case, U=U, Q=Q, ldu=ldu, out=torch.zeros(nout, ldu, dtype=dt, device=DEV))
    if kind == "qr":
        K = _randn(g, case["s"], case["n"])
        K[1:] += 0.5 * K[:-1].clone()                 # neighbouring columns are correlated
        return dict(case=case, K=K, Q=torch.empty_like(K), seed=int(seed) % 1000)
    if kind == "solve":
        rp, ci, v = _operator(case, g)
        n = rp.numel() - 1
        u1 = _randn(g, n)
        torch.cuda.synchronize()
        s = rks.Solver(n, rp, ci, v, case["k"], case["p"], case["d"], which=case["which"], seed=0, zeta=case["zeta"],
                       u1=u1, prec=case["prec"], keep=case["keep"], max_restarts=case["restarts"], device=True,
                       **_solve_opts(case))
        X = torch.zeros(case["k"] + 1, n, dtype=torch.float64, device=DEV)
        return dict(case=case, solver=s, X=X, u1=u1)
    if kind == "batch":
        probs = []
        for nx, ny, b, nu in _batch_problems(case, seed):
            rp, ci, v = _stencil((ny, nx), nu, b)
            probs.append(inputs.CSR(nx * ny, rp.cpu().numpy(), ci.cpu().numpy(), v.float().cpu().numpy()))
        B = rks.DevBatch(probs, case["k"], case["p"], case["d"], which="LR", tol=0.25e-8, seed=0, zeta=case["zeta"],
                         maxit=case["restarts"], conv="norm1", verify=1e-8, keep=case["keep"])
        return dict(case=case, batch=B)
    xs, qs = _network_inputs(case, seed)
    return dict(case=case, net=rks.WarmStart(case["H"], case["W"], seed=int(seed) % 1000), xs=xs, qs=qs)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _phased(lam, X, u1):
    """The eigenvectors (rows of X, a pair as Re and Im) with x^T u1 > 0, in place: their sign and phase are free."""
    c = X @ u1
    for j, im in enumerate(lam.imag):
        if im == 0:
            X[j] *= torch.sign(c[j])
        elif im > 0:
            z = torch.complex(c[j], c[j + 1])
            x = torch.complex(X[j], X[j + 1]) * (torch.conj(z) / z.abs())
            X[j], X[j + 1] = x.real, x.imag
    return X


def _pairs(size, lam, resid, rq, est):
    """Eigenvalues, residuals, Rayleigh quotients and estimates in arrays of ``size`` (k pairs, or k + 1 when a complex
    pair lies at the cut)."""
    cols = dict(lam_re=lam.real, lam_im=lam.imag, resid=resid, rq_re=rq.real, rq_im=rq.imag, est=est)
    return {q: np.concatenate([v, np.zeros(size - v.size)]) for q, v in cols.items()}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sketch":
        return rks.sketch_apply(state["x"], case["d"], case["zeta"], state["seed"])
    if kind == "product":
        f = rks.basis_product_f32 if case["prec"] == "f32" else rks.basis_product_df
        f(state["U"], state["ldu"], case["n"], case["nin"], state["Q"], state["out"])
        return state["out"]
    if kind == "qr":
        return rks.sketch_qr(state["K"], case["d"], case["zeta"], state["seed"], method=case["method"], Q=state["Q"])
    if kind == "solve":
        s = state["solver"]
        info = s.solve()
        lam, X, resid = s.eigpairs(X_out=state["X"])
        rq = s.rayleigh()
        X = _phased(lam, X, state["u1"])
        return dict(_pairs(case["k"] + 1, lam, resid, rq, s.estimates()), X=X, nmatvec=int(info["nmatvec"]))
    if kind == "batch":
        B = state["batch"]
        infos = B.solve()
        pairs = [B.eigpairs(i, want_vectors=False) for i in range(B.count)]
        pairs = [_pairs(B.k + 1, lam, resid, rq, est) for lam, _, resid, rq, est in pairs]
        out = {q: np.stack([p[q] for p in pairs]) for q in pairs[0]}
        return dict(out, nmatvec=np.array([i["nmatvec"] for i in infos]))
    net = state["net"]
    if case["mode"] == "forward":
        return [net.forward(x) for x in state["xs"]]
    net.zero_grad()
    loss = [net.accumulate(x, Q) for x, Q in zip(state["xs"], state["qs"])]
    return dict(loss=loss, grad=net.grad())


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

def _rows_nnz(case):
    op = case["op"]
    if op == "tridiag":
        return case["n"], 3 * case["n"]
    if op == "conv2d":
        return case["nx"] * case["ny"], 5 * case["nx"] * case["ny"]
    if op == "conv3d":
        n = case["nx"] * case["ny"] * case["nz"]
        return n, 7 * n
    return case["n"], int(case["n"] * (5.8 if op == "powerlaw" else 41))


def _restart_work(n, nnz, k, m, keep, restarts, P, PA, A_bytes):
    """Bytes and flops of the first expansion and ``restarts`` restarts: per
    step one read of A, the new vector and the basis (w read and written once),
    per restart one read of the basis and one write of what is kept."""
    kept = max(k, min(keep, m // 2))
    by = fl = 0.0
    for r in range(restarts):
        for c in range(1 if r == 0 else kept + 1, m + 1):
            by += nnz * PA + A_bytes + 2 * P * n + (c + 2) * P * n
            fl += 2.0 * nnz + 2.0 * n * c
        by += (m + kept) * P * n
        fl += 2.0 * n * m * kept
    by += (kept + k) * 8.0 * n + nnz * 8.0                # Ritz vectors and residuals
    fl += 2.0 * n * kept * k + 2.0 * nnz * k
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "sketch":
        return {"bytes": 8.0 * (case["n"] + case["d"]), "flops": 2.0 * case["n"] * case["zeta"]}
    if kind == "product":
        P = 4.0 if case["prec"] == "f32" else 8.0
        return {"bytes": P * case["n"] * (case["nin"] + case["nout"]),
                "flops": 2.0 * case["n"] * case["nin"] * case["nout"]}
    if kind == "qr":
        n, s = case["n"], case["s"]
        return {"bytes": 16.0 * n * s, "flops": 1.0 * n * s * s + 2.0 * n * s * case["zeta"]}
    if kind == "solve":
        n, nnz = _rows_nnz(case)
        stencil = case["op"] in ("tridiag", "conv2d", "conv3d")
        PA, m = (4.0 if case["op"] == "conv3d" else 8.0), case["k"] + case["p"]
        A_bytes = 0.0 if stencil else 4.0 * nnz + 4.0 * n
        P = 4.0 if case["prec"] == "mixed" else 8.0
        by, fl = _restart_work(n, nnz, case["k"], m, case["keep"], case["restarts"], P, PA, A_bytes)
        return {"bytes": by, "flops": fl}
    if kind == "batch":
        r = np.random.RandomState(case["sizes"])
        by = fl = 0.0
        for _ in range(case["count"]):
            nx, ny = (int(v) for v in r.randint(case["lo"], case["hi"] + 1, 2))
            r.rand(2)
            b, f = _restart_work(nx * ny, 5 * nx * ny, case["k"], case["k"] + case["p"], case["keep"], case["restarts"],
                                 8.0, 4.0, 0.0)
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    px = case["H"] * case["W"]
    macs = 9 * px * (3 * 32 + 32 * 32 + 2 * 32 * 32 + 32 + 4 * 32 * 32 / 4 + 4 * 32 * 32 / 16 + 2 * 32 * 32 / 64)
    by = 4.0 * px * (3 + 1)
    if case["mode"] == "forward":
        return {"bytes": by * case["batch"], "flops": 2.0 * macs * case["batch"]}
    return {"bytes": (by + 4.0 * px * case["q"]) * case["batch"] + 4.0 * 121_409, "flops": 6.0 * macs * case["batch"]}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------

_GAMMA = 0x9E3779B97F4A7C15


def _i64(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _mix64(z):
    """SplitMix64's output function (Steele, Lea & Flood 2014) on int64 tensors."""
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _omega(n, d, zeta, seed):
    """Rows (n x zeta) and signs of the sparse-sign embedding: distinct rows from the draws of (seed, column)."""
    base = _mix64(torch.arange(n, device=DEV) + _i64(seed * _GAMMA))
    rows = torch.full((n, zeta), -1, dtype=torch.int64, device=DEV)
    sign = torch.zeros(n, zeta, dtype=torch.float64, device=DEV)
    cnt = torch.zeros(n, dtype=torch.int64, device=DEV)
    act = torch.arange(n, device=DEV)
    r = 0
    while act.numel():
        h = _mix64(base[act] + _i64((r + 1) * _GAMMA))
        row = (_shr(h, 32) * d) >> 32
        new = ~(rows[act] == row[:, None]).any(dim=1)
        a = act[new]
        rows[a, cnt[a]] = row[new]
        sign[a, cnt[a]] = 1.0 - 2.0 * (h[new] & 1).double()
        cnt[a] += 1
        act = act[cnt[act] < zeta]
        r += 1
    return rows, sign


def _sketcher(n, d, zeta, seed):
    rows, sign = _omega(n, d, zeta, seed)
    flat = rows.reshape(-1)

    def apply(x):
        z = torch.zeros(d, dtype=torch.float64, device=DEV)
        return z.index_add_(0, flat, (sign * x[:, None]).reshape(-1)) / math.sqrt(zeta)
    return apply


def _normal_start(n, seed):
    i = torch.arange(n, device=DEV)
    u = [_shr(_mix64(_i64(seed) + (2 * i + t) * _i64(_GAMMA)), 11).double() * 2.0**-53 for t in (1, 2)]
    return torch.sqrt(-2.0 * torch.log1p(-u[0])) * torch.cos(2.0 * math.pi * u[1])


def _best(lam, which):
    """Indices of one member (Im >= 0) of every eigenvalue or pair, best first."""
    key = {"LM": -np.abs(lam), "SM": np.abs(lam), "LR": -lam.real, "SR": lam.real}[which]
    idx = [i for i in np.argsort(key, kind="stable") if lam[i].imag >= 0]
    return idx


def _krylov_schur(A, n, k, p, d, zeta, which, u1, keep, restarts, conv):
    """Ritz values, residuals, Rayleigh quotients and estimates after
    ``restarts`` restarts of randomized Krylov-Schur that locks nothing."""
    m = k + p
    om = _sketcher(n, d, zeta, 0)
    colsum = torch.zeros(n, dtype=torch.float64, device=DEV)
    norm1 = float(colsum.index_add_(0, A.col_indices().long(), A.values().abs()).max())
    U = torch.zeros(m + 1, n, dtype=torch.float64, device=DEV)
    S = torch.zeros(m + 1, d, dtype=torch.float64, device=DEV)
    B = np.zeros((m, m))
    s = om(u1)
    U[0], S[0] = u1 / s.norm(), s / s.norm()
    have = 0
    for _ in range(restarts):
        for j in range(have, m):
            w = A @ U[j]
            z = om(w)
            r = S[:j + 1] @ z
            r = r + S[:j + 1] @ (z - S[:j + 1].T @ r)
            w = w - U[:j + 1].T @ r
            s = om(w)
            beta = float(s.norm())
            U[j + 1], S[j + 1] = w / beta, s / beta
            B[:j + 1, j] = r.cpu().numpy()
            if j + 1 < m:
                B[j + 1, j] = beta
        lam, Y = np.linalg.eig(B)
        want, basis = max(k, min(keep, m // 2)), []
        for i in _best(lam, which):
            if len(basis) >= want:
                break
            basis += [Y[:, i].real] if lam[i].imag == 0 else [Y[:, i].real, Y[:, i].imag]
        Qk = np.linalg.qr(np.stack(basis, axis=1))[0]
        ka = Qk.shape[1]
        T, b = Qk.T @ B @ Qk, beta * Qk[m - 1]
        Qd = torch.from_numpy(Qk).to(DEV)
        U[:ka], S[:ka] = Qd.T @ U[:m], Qd.T @ S[:m]
        U[ka], S[ka] = U[m].clone(), S[m].clone()
        B[:] = 0.0
        B[:ka, :ka], B[ka, :ka] = T, b
        have = ka
    lam, Y = np.linalg.eig(T)
    out = dict(lam=[], resid=[], rq=[], est=[], x=[])
    for i in _best(lam, which):
        if len(out["lam"]) >= k:
            break
        y = Y[:, i] / np.linalg.norm(Y[:, i])
        Yd = torch.from_numpy(np.stack([y.real, y.imag])).to(DEV)
        x = Yd @ U[:ka]
        ax = torch.stack([A @ x[0], A @ x[1]])
        xx = float((x * x).sum())
        re = ax[0] - lam[i].real * x[0] + lam[i].imag * x[1]
        im = ax[1] - lam[i].real * x[1] - lam[i].imag * x[0]
        rq = complex(float((x * ax).sum()), float((x[0] * ax[1]).sum() - (x[1] * ax[0]).sum())) / xx
        res = math.sqrt(float((re * re).sum() + (im * im).sum())) / (norm1 * math.sqrt(xx))
        est = abs(b @ y) / (norm1 if conv == "norm1" else abs(lam[i]))
        for c in ([1] if lam[i].imag == 0 else [1, -1]):
            out["lam"].append(complex(lam[i].real, c * lam[i].imag))
            out["rq"].append(complex(rq.real, c * rq.imag if lam[i].imag else 0.0))
            out["resid"].append(res)
            out["est"].append(est)
        out["x"] += [x[0]] if lam[i].imag == 0 else [x[0], x[1]]
    lam, resid, rq, est = (np.array(out[q]) for q in ("lam", "resid", "rq", "est"))
    X = torch.stack(out["x"])
    if len(lam) == k:
        X = torch.cat([X, torch.zeros(1, n, dtype=torch.float64, device=DEV)])
    return _pairs(k + 1, lam, resid, rq, est), _phased(lam, X, u1)


def _csr64(rp, ci, v, n):
    return torch.sparse_csr_tensor(rp.long(), ci.long(), v.double(), size=(n, n))


def _exact_qr(case, seed):
    n, s, d, zeta = case["n"], case["s"], case["d"], case["zeta"]
    K = prepare(case, seed)["K"]
    rh = case["method"] == "rhqr"
    om = _sketcher(n - s if rh else n, d, zeta, int(seed) % 1000)
    sk = (lambda q: torch.stack([om(c[s:]) for c in q])) if rh else (lambda q: torch.stack([om(c) for c in q]))
    Sk = sk(K)
    if rh:
        Sk = torch.cat([K[:, :s], Sk], dim=1)

    def upper(M):                                         # R of the QR of the columns in M's rows, positive diagonal
        R = torch.linalg.qr(M.T)[1]
        return R * torch.sign(torch.diagonal(R))[:, None]
    R = upper(Sk)
    Q = torch.linalg.solve_triangular(R.T, K, upper=False)
    if case["method"] == "rcholqr":
        R2 = torch.linalg.cholesky(Q @ Q.T).T
        Q, R = torch.linalg.solve_triangular(R2.T, Q, upper=False), R2 @ R
    return Q, R.cpu().numpy(), sk(Q).T.cpu().numpy()


def _exact_network(case, seed):
    xs, qs = _network_inputs(case, seed)
    net = rks.WarmStart(case["H"], case["W"], seed=int(seed) % 1000)
    theta = net.params()                                  # the inputs: initial weights
    net.close()
    layers, o = [], 0
    for ci, co in [(3, 32)] + [(32, 32)] * 13 + [(32, 1)]:
        Wt = torch.from_numpy(theta[o:o + co * ci * 9]).to(DEV).half().double().reshape(co, ci, 3, 3)
        b = torch.from_numpy(theta[o + co * ci * 9:o + co * ci * 9 + co]).to(DEV).double()
        o += co * ci * 9 + co
        layers.append((Wt.requires_grad_(), b.requires_grad_()))

    def conv(z, j):                                       # 3 x 3, zero padding, as one product per layer
        Wt, b = layers[j]
        cols = torch.nn.functional.unfold(z[None], 3, padding=1)[0]
        return (Wt.reshape(Wt.shape[0], -1) @ cols + b[:, None]).reshape(-1, *z.shape[1:])

    def block(z, j):
        return torch.relu(conv(torch.relu(conv(z, j)), j + 1))

    def pool(z):
        return torch.nn.functional.avg_pool2d(z[None], 2)[0]

    def up(z):
        return z.repeat_interleave(2, dim=1).repeat_interleave(2, dim=2)
    us, losses = [], []
    for x, Q in zip(xs, qs):
        with torch.set_grad_enabled(case["mode"] == "grad"):
            e0 = block(x.double(), 0)
            e1 = block(pool(e0), 2)
            e2 = block(pool(e1), 4)
            d2 = block(up(block(pool(e2), 6)) + e2, 8)
            d1 = block(up(d2) + e1, 10)
            u = conv(block(up(d1) + e0, 12), 14)[0]
            if case["mode"] == "forward":
                us.append(u)
                continue
            v = u.reshape(-1)
            loss = 1.0 - ((Q.double() @ v) ** 2).sum() / (v * v).sum()
        loss.backward()
        losses.append(float(loss.detach()))
    if case["mode"] == "forward":
        return us
    grad = torch.cat([t.grad.reshape(-1) for pair in layers for t in pair])
    return dict(loss=losses, grad=grad)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sketch":
        st = prepare(case, seed)
        return _sketcher(case["n"], case["d"], case["zeta"], st["seed"])(st["x"])
    if kind == "product":
        st = prepare(case, seed)
        out = torch.zeros(case["nout"], st["ldu"], dtype=torch.float64, device=DEV)
        n, Qd = case["n"], torch.from_numpy(np.ascontiguousarray(st["Q"].T)).to(DEV)
        for a in range(0, n, 1 << 19):
            out[:, a:min(n, a + (1 << 19))] = Qd @ st["U"][:, a:min(n, a + (1 << 19))].double()
        return out
    if kind == "qr":
        return _exact_qr(case, seed)
    if kind == "solve":
        if case["prec"] == "mixed":                       # what the FP32 phase stores has no 64-bit value
            return None
        g = _gen(seed)
        rp, ci, v = _operator(case, g)
        n = rp.numel() - 1
        o, X = _krylov_schur(_csr64(rp, ci, v, n), n, case["k"], case["p"], case["d"], case["zeta"], case["which"],
                          _randn(g, n), case["keep"], case["restarts"], _solve_opts(case)["conv"])
        return dict(o, X=X, nmatvec=None)
    if kind == "batch":
        parts = []
        for nx, ny, b, nu in _batch_problems(case, seed):
            rp, ci, v = _stencil((ny, nx), nu, b)
            n = nx * ny
            parts.append(_krylov_schur(_csr64(rp, ci, v.float(), n), n, case["k"], case["p"], case["d"], case["zeta"],
                                       "LR", _normal_start(n, 1), case["keep"], case["restarts"], "norm1")[0])
        return dict({q: np.stack([o[q] for o in parts]) for q in parts[0]}, nmatvec=None)
    return _exact_network(case, seed)
