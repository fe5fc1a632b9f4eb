"""The calls that users of this library spend their time in, as measurable cases.

Every case goes through the public entry points of ``paper_2608_28952_gb300``
on inputs drawn on the GPU from a seed:

* ``evd``          ``syev``: one dense symmetric matrix, plain FP64, FP64 with
                   emulated products or the mixed form;
* ``svd``          ``gesvd``: one tall matrix, direct or QR-preconditioned;
* ``step``         ``jacobi_syev_step`` / ``jacobi_syev_step_lowp``: a single
                   parallel step, the block that the large solves repeat;
* ``batched_evd``  an EVD ``Plan`` over many matrices of uneven order;
* ``batched_svd``  a one-sided SVD ``Plan`` over tall matrices.

A whole solve's eigenvectors and singular vectors are defined up to their
sign; ``run`` fixes it the usual way (the entry of largest magnitude is
positive), as a program does that stores or compares vectors.
"""
from __future__ import annotations

import math

import torch

import paper_2608_28952_gb300 as jg

DEV = "cuda"


def listed():
    return [
        # the smallest calls: a Hessian or covariance block, latency only
        dict(name="evd64", kind="evd", n=64, b=16, precision="fp64"),
        # the repository's small benchmark (n = 256, b = 16): 150 dependent steps
        dict(name="evd256", kind="evd", n=256, b=16, precision="fp64"),
        # an ordinary FP64 solve, default block size, an order that is no multiple of it
        dict(name="evd1000", kind="evd", n=1000, b=32, precision="fp64"),
        # FP64-accurate products on the tensor cores, half the benchmark's order
        dict(name="evd2048emu", kind="evd", n=2048, b=64, precision="emu"),
        # the mixed form with FP64-accurate closing products (benchmark mixed4096emu): the largest whole call
        dict(name="mixed4096emu", kind="evd", n=4096, b=64, precision="mixed"),
        # one low-precision step of the largest benchmark (n = 8192, b = 128), FP32 matrices
        dict(name="step8192lowp", kind="step", n=8192, b=128, precision="lowp"),
        # one emulated FP64 step of the same order: the closing sweeps' block
        dict(name="step8192emu", kind="step", n=8192, b=128, precision="emu"),
        # a least-squares or PCA sized one-sided SVD, direct FP64, ragged
        dict(name="svd1000x200", kind="svd", m=1000, n=200, b=16, precision="fp64", qr=False),
        # the QR-preconditioned SVD with emulated products, an eighth of the benchmark's matrix
        dict(name="svd8192x1024qremu", kind="svd", m=8192, n=1024, b=64, precision="emu", qr=True),
        # the benchmark's batches (orders 8..512, FP32 and FP64; tall 1024 x 64), fewer matrices of each
        dict(name="batched_f32", kind="batched_evd", count=1000, lo=8, hi=512, dtype="f32"),
        dict(name="batched_f64", kind="batched_evd", count=200, lo=8, hi=512, dtype="f64"),
        dict(name="batched_svd_f32", kind="batched_svd", count=2048, m=1024, n=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges; sizes log-uniform, mostly odd ones."""
    kind = rng.choice(["evd", "evd", "evd", "svd", "svd", "step", "batched_evd", "batched_svd"])
    if kind == "evd":
        precision = rng.choice(["fp64", "fp64", "emu", "mixed"])
        if precision == "fp64":
            n = _log_int(rng, 40, 1200)
            b = rng.choice([8, 16] if n < 100 else [16, 32] if n < 400 else [16, 32, 64])
        else:
            n = _log_int(rng, 500, 2600)
            b = rng.choice([32, 64] if n < 1000 else [64, 128])
        return dict(kind="evd", n=n, b=b, precision=precision)
    if kind == "svd":
        qr = rng.random() < 0.5
        precision = rng.choice(["fp64", "emu"]) if qr else "fp64"
        n = _log_int(rng, 40, 700 if qr else 300)
        m = min(6000, _log_int(rng, n, 10 * n))
        b = rng.choice([8, 16] if n < 100 else [16, 32] if n < 400 else [32, 64])
        return dict(kind="svd", m=m, n=n, b=b, precision=precision, qr=qr)
    if kind == "step":
        b = rng.choice([32, 64, 128])
        N = 2 * _log_int(rng, 4, 4096 // b)
        return dict(kind="step", n=N * b, b=b, precision=rng.choice(["lowp", "emu", "fp64"]) if N * b <= 4096 else
                    rng.choice(["lowp", "emu"]))
    if kind == "batched_evd":
        dtype = rng.choice(["f32", "f64"])
        lo = _log_int(rng, 2, 64)
        hi = _log_int(rng, max(lo, 32), 512)
        most = 1000 if dtype == "f32" else 200
        return dict(kind="batched_evd", count=_log_int(rng, 20, most), lo=lo, hi=hi, dtype=dtype)
    n = _log_int(rng, 8, 96)
    m = min(1024, _log_int(rng, n, 32 * n))
    return dict(kind="batched_svd", count=_log_int(rng, 50, 2048), m=m, n=n)


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 17)


def _sym(n, g):
    M = torch.randn((n, n), generator=g, device=DEV, dtype=torch.float64)
    return 0.5 * (M + M.t())


def _tall(m, n, g):
    """U diag(sigma) V^T with sigma falling over two decades (a condition
    number of 100, as data matrices have), U and V orthonormal."""
    U, _ = torch.linalg.qr(torch.randn((m, n), generator=g, device=DEV, dtype=torch.float64))
    V, _ = torch.linalg.qr(torch.randn((n, n), generator=g, device=DEV, dtype=torch.float64))
    s = 10.0 ** (-2.0 * torch.arange(n, device=DEV, dtype=torch.float64) / max(n - 1, 1))
    return (U * s) @ V.t()


def _sizes(case):
    """The batch's orders, uniform in lo..hi: the same for every seed."""
    g = torch.Generator().manual_seed(7)
    return torch.randint(case["lo"], case["hi"] + 1, (case["count"],), generator=g).tolist()


def _views(flat, shapes):
    """Column-major (m, n) views into a flat buffer, one after the other."""
    out, at = [], 0
    for m, n in shapes:
        out.append(flat[at:at + m * n].view(n, m).t())
        at += m * n
    return out


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "evd":
        return _sym(case["n"], g)
    if kind == "svd":
        return _tall(case["m"], case["n"], g)
    if kind == "step":
        n, dt = case["n"], torch.float32 if case["precision"] == "lowp" else torch.float64
        # a few sweeps into a solve: the eigenvalues spread over the diagonal, the rest small but far from done
        A = (1e-3 * _sym(n, g) + torch.diag(torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * 2 - 1)).to(dt)
        Q = (torch.randn((n, n), generator=g, device=DEV, dtype=torch.float32) / math.sqrt(n)).to(dt)
        return A, Q
    if kind == "batched_evd":
        ns = _sizes(case)
        dt = torch.float32 if case["dtype"] == "f32" else torch.float64
        flat = torch.randn(sum(n * n for n in ns), generator=g, device=DEV, dtype=dt)
        for v in _views(flat, [(n, n) for n in ns]):
            v.copy_(0.5 * (v + v.t()))
        return ns, flat
    return torch.randn((case["count"], case["n"], case["m"]), generator=g, device=DEV, dtype=torch.float32)


def prepare(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "evd":
        kw = dict(b=case["b"])
        if case["precision"] == "emu":
            kw["precision"] = jg.PREC_FP64_EMU
        elif case["precision"] == "mixed":
            kw.update(precision=jg.PREC_MIXED_BF16X3, fp64_products=1, refine_steps=2)
        return dict(kind=kind, A=x, kw=kw)
    if kind == "svd":
        kw = dict(b=case["b"], svd_qr=int(case["qr"]))
        if case["precision"] == "emu":
            kw["precision"] = jg.PREC_FP64_EMU
        return dict(kind=kind, G=x, kw=kw)
    if kind == "step":
        prec = {"lowp": jg.PREC_MIXED_BF16X3, "emu": jg.PREC_FP64_EMU, "fp64": jg.PREC_FP64}[case["precision"]]
        A, Q = (jg.colmajor(y) for y in x)
        return dict(kind=kind, lowp=case["precision"] == "lowp", A=A, Q=Q, p=jg.params(b=case["b"], precision=prec))
    if kind == "batched_evd":
        ns, flat = x
        w = torch.empty(sum(ns), dtype=flat.dtype, device=DEV)
        Z = torch.empty_like(flat)
        ws, at = [], 0
        for n in ns:
            ws.append(w[at:at + n])
            at += n
        shapes = [(n, n) for n in ns]
        plan = jg.Plan(0, jg.PREC_FP32 if case["dtype"] == "f32" else jg.PREC_FP64, ns, p=jg.params())
        return dict(kind=kind, plan=plan, flat=flat, w=w, Z=Z, X=_views(flat, shapes), ws=ws, Zs=_views(Z, shapes),
                    info=torch.zeros(len(ns), dtype=torch.int32, device=DEV))
    count, n, m = x.shape
    U = torch.empty_like(x)
    s = torch.empty((count, n), dtype=x.dtype, device=DEV)
    V = torch.empty((count, n, n), dtype=x.dtype, device=DEV)
    plan = jg.Plan(1, jg.PREC_FP32, [n] * count, m=[m] * count, p=jg.params())
    return dict(kind=kind, plan=plan, G=x, U=U, s=s, V=V, Us=[u.t() for u in U], ss=list(s), Vs=[v.t() for v in V],
                info=torch.zeros(count, dtype=torch.int32, device=DEV))


# ------------------------------------------------------------------ one pass
def _signs(Q):
    """+-1 per column: the sign of its entry of largest magnitude."""
    top = Q.gather(0, Q.abs().argmax(0, keepdim=True))
    return torch.where(top < 0, -1.0, 1.0).to(Q.dtype)


def run(state):
    kind = state["kind"]
    if kind == "evd":
        w, Q, D, _ = jg.syev(state["A"], **state["kw"])
        return dict(w=w, Q=Q * _signs(Q), D=D)
    if kind == "svd":
        U, s, V, _ = jg.gesvd(state["G"], **state["kw"])
        sg = _signs(V)
        return dict(U=U * sg, s=s, V=V * sg)
    if kind == "step":
        # the step works in place; the program keeps the matrix it steps from
        A, Q = state["A"].clone(), state["Q"].clone()
        f = jg.jacobi_syev_step_lowp if state["lowp"] else jg.jacobi_syev_step
        rc = f(A, Q, 0, state["p"])
        if rc != 0:
            raise RuntimeError(f"step: {rc}")
        return dict(A=A, Q=Q)
    if kind == "batched_evd":
        rc, _ = state["plan"].execute(state["X"], state["ws"], state["Zs"], state["info"])
        if rc != 0:
            raise RuntimeError(f"execute: {rc}")
        return dict(w=state["w"], Q=state["Z"], info=state["info"])
    state["U"].copy_(state["G"])     # the one-sided solve overwrites its input
    rc, _ = state["plan"].execute(state["Us"], state["ss"], state["Vs"], state["info"])
    if rc != 0:
        raise RuntimeError(f"execute: {rc}")
    return dict(U=state["U"], s=state["s"], V=state["V"], info=state["info"])


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: a dense
    symmetric EVD with vectors cannot do without about 9 n^3, a tall SVD with
    both sets of vectors without about 6 m n^2 + 11 n^3; a step without its
    symmetric two-sided update (4 n^2 b), its column update of Q (4 n^2 b)
    and one sweep of rotations of every pivot and its transform."""
    kind = case["kind"]
    if kind == "evd":
        n = case["n"]
        return dict(bytes=8.0 * (2 * n * n + 2 * n), flops=9.0 * n ** 3)
    if kind == "svd":
        m, n = case["m"], case["n"]
        return dict(bytes=8.0 * (2 * m * n + n * n + n), flops=6.0 * m * n * n + 11.0 * n ** 3)
    if kind == "step":
        n, b = case["n"], case["b"]
        size = 4 if case["precision"] == "lowp" else 8
        k = 2 * b
        return dict(bytes=4.0 * size * n * n, flops=8.0 * n * n * b + (n // k) * 6.0 * k ** 3)
    if kind == "batched_evd":
        # orders uniform in lo..hi
        lo, hi, size = case["lo"], case["hi"], 4 if case["dtype"] == "f32" else 8
        ns = range(lo, hi + 1)
        n2 = sum(n * n for n in ns) / len(ns)
        n3 = sum(n ** 3 for n in ns) / len(ns)
        return dict(bytes=case["count"] * size * (2 * n2 + (lo + hi) / 2), flops=case["count"] * 9.0 * n3)
    m, n, c = case["m"], case["n"], case["count"]
    return dict(bytes=4.0 * c * (2 * m * n + n * n + n), flops=c * (6.0 * m * n * n + 11.0 * n ** 3))


# ------------------------------------------------------------------ the same in 64 bits
def _round_robin(k, r):
    """Pairs (p, q), p < q, of round r of the round-robin order of k indices."""
    at = lambda pos: 0 if pos == 0 else 1 + (pos - 1 + r) % (k - 1)  # noqa: E731
    pairs = [sorted((at(e), at(k - 1 - e))) for e in range(k // 2)]
    return [p for p, _ in pairs], [q for _, q in pairs]


def _exact_step(case, seed):
    """One parallel step with one sweep of each pivot, in FP64."""
    n, b, k = case["n"], case["b"], 2 * case["b"]
    A, Q = (x.double() for x in _inputs(case, seed))
    I, J = _round_robin(n // b, 0)
    ar = torch.arange(b, device=DEV)
    cols = torch.stack([torch.cat([i * b + ar, j * b + ar]) for i, j in zip(I, J)])    # pairs x k
    P = A[cols[:, :, None], cols[:, None, :]]
    V = torch.eye(k, device=DEV, dtype=torch.float64).repeat(len(I), 1, 1)
    tol = 4.0 * 2.0 ** -53
    for r in range(k - 1):
        p, q = (torch.tensor(x, device=DEV) for x in _round_robin(k, r))
        app, aqq, apq = P[:, p, p], P[:, q, q], P[:, p, q]
        on = apq.abs() > tol * (app.abs().sqrt() * aqq.abs().sqrt())
        zeta = (aqq - app) / torch.where(on, 2 * apq, 1.0)
        t = torch.where(zeta >= 0, 1.0, -1.0) / (zeta.abs() + (1 + zeta * zeta).sqrt())
        t = torch.where(on, t, 0.0)
        c = 1 / (1 + t * t).sqrt()
        s = t * c
        x, y = P[:, p, :], P[:, q, :]
        P[:, p, :], P[:, q, :] = c[:, :, None] * x - s[:, :, None] * y, s[:, :, None] * x + c[:, :, None] * y
        for M in (P, V):
            x, y = M[:, :, p], M[:, :, q]
            M[:, :, p], M[:, :, q] = c[:, None, :] * x - s[:, None, :] * y, s[:, None, :] * x + c[:, None, :] * y
        P[:, p, q] = torch.where(on, 0.0, P[:, p, q])
        P[:, q, p] = torch.where(on, 0.0, P[:, q, p])
    order = P.diagonal(dim1=1, dim2=2).argsort(dim=1, descending=True, stable=True)
    V = V.gather(2, order[:, None, :].expand(-1, k, -1))
    P = P.gather(1, order[:, :, None].expand(-1, -1, k)).gather(2, order[:, None, :].expand(-1, k, -1))
    A1, Q1 = A.clone(), Q.clone()
    for c, v in zip(cols, V):
        A1[:, c] = A[:, c] @ v
        Q1[:, c] = Q[:, c] @ v
    A2 = A1.clone()
    for c, v in zip(cols, V):
        A2[c, :] = v.t() @ A1[c, :]
    A2[cols[:, :, None], cols[:, None, :]] = P
    return dict(A=A2, Q=Q1)


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "evd":
        w, Q = torch.linalg.eigh(x)
        return dict(w=w, Q=Q * _signs(Q), D=torch.diag(w))
    if kind == "svd":
        Qr, R = torch.linalg.qr(x)
        U, s, Vh = torch.linalg.svd(R)
        U, V = Qr @ U, Vh.t()
        sg = _signs(V)
        return dict(U=U * sg, s=s, V=V * sg)
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "batched_evd":
        ns, flat = x
        w = torch.cat([torch.linalg.eigvalsh(v.double()) for v in _views(flat, [(n, n) for n in ns])])
        return dict(w=w, Q=None, info=None)      # a vector's sign is the solver's own
    s = torch.linalg.eigvalsh(x.double() @ x.double().transpose(1, 2)).flip(1).clamp(min=0).sqrt()
    return dict(U=None, s=s, V=None, info=None)
