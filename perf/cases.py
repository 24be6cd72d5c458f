"""The calls whose speed is measured: what a program asks of this library, over the sizes
it is made for.

Every case goes through the public entry points of the Python binding, on inputs made on
the device from the case's seed. Kinds:

  qr        factor + thin Q of one matrix
  qr_solve  factor, thin Q, Q^T b and the triangular solve (the headline step)
  orth      Q-only TSQR of a tall block (orthonormalize)
  project   residual of B against range(A) with a kept factor set: Q^T B, the first n rows
            cleared, Q times the rest (both directions of the implicit Q)
  lstsq     one least-squares problem, FP64 or mixed precision
  batch_r   R of many uneven matrices, half FP64 and half mixed, in one call
  batch_x   a batch of least-squares requests, as a server forms them
  caqr      factor + thin Q of a wider matrix
  host      the FP64 path on pinned host buffers, copies in and out

Rows of Q^T B below the first n depend on the choice of reflectors, so no case returns
them; everything returned (R with diag(R) >= 0, thin Q, X, residuals) is unique.
"""
import math

import numpy as np
import torch

import paper_0912_2572_gb300 as ts

KINDS = ("qr", "qr_solve", "orth", "project", "lstsq", "batch_r", "batch_x", "caqr", "host")
BATCH_WIDTHS = (8, 16, 32, 64)
SERVED_WIDTHS = (16, 32, 64, 128)


def listed():
    return [
        # the smallest documented factorization (256-row leaves, a pure binary tree): launches and latency
        {"name": "qr_4096x16", "kind": "qr", "m": 4096, "n": 16, "leaf_h": 256, "two_level": False, "decades": 0.0},
        # one small request solved at once by a program that waits for its answer
        {"name": "lstsq_1000x16", "kind": "lstsq", "m": 1000, "n": 16, "k": 1, "mixed": False, "decades": 2.0},
        # a matrix of no round size, with the binding's defaults
        {"name": "qr_300007x37", "kind": "qr", "m": 300007, "n": 37, "leaf_h": 256, "two_level": True, "decades": 3.0},
        # the headline matrix and step
        {"name": "step_4194304x64", "kind": "qr_solve", "m": 4194304, "n": 64, "k": 1, "decades": 6.0},
        # orthonormalization of a tall block of a block eigensolver's basis
        {"name": "orth_16777216x16", "kind": "orth", "m": 16777216, "n": 16, "decades": 0.0},
        # many columns against a kept factor set, both directions of Q
        {"name": "project_1048576x64_k32", "kind": "project", "m": 1048576, "n": 64, "k": 32, "decades": 3.0},
        # the largest request of the served range, solved alone in FP64
        {"name": "lstsq_1000000x64_k4", "kind": "lstsq", "m": 1000000, "n": 64, "k": 4, "mixed": False, "decades": 4.0},
        # the large mixed-precision least-squares problem
        {"name": "mixed_16777216x32_k4", "kind": "lstsq", "m": 16777216, "n": 32, "k": 4, "mixed": True, "decades": 4.0},
        # uneven instances in one call, half FP64 and half mixed, R only
        {"name": "batch_r_2000", "kind": "batch_r", "count": 2000, "m_max": 65536},
        # one batch of served least-squares requests in FP64 and one in mixed precision
        {"name": "served_fp64_32", "kind": "batch_x", "count": 32, "m_max": 1000000, "mixed": False},
        {"name": "served_mixed_64", "kind": "batch_x", "count": 64, "m_max": 1000000, "mixed": True},
        # a matrix wide enough for CAQR: panels of 64 columns and their trailing updates
        {"name": "caqr_262144x256", "kind": "caqr", "m": 262144, "n": 256},
    ]


def _between(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(KINDS)
    if kind == "qr":
        n = _between(rng, 2, 128)
        m = _between(rng, max(1000, 2 * n), min(4000000, (1 << 28) // n))
        return {"kind": kind, "m": m, "n": n, "leaf_h": rng.choice([max(n, 128), 256, 512, 1000]),
                "two_level": rng.random() < 0.75, "decades": rng.choice([0.0, 2.0, 4.0])}
    if kind in ("qr_solve", "host"):
        n = _between(rng, 8, 64)
        m = _between(rng, 20000, (1 << 28) // n if kind == "qr_solve" else 500000)
        return {"kind": kind, "m": m, "n": n, "k": rng.choice([1, 1, 2, 4]), "decades": rng.choice([0.0, 2.0, 4.0, 6.0])}
    if kind == "orth":
        n = rng.choice([8, 16, 32, 64, _between(rng, 4, 64)])
        return {"kind": kind, "m": _between(rng, 20000, (1 << 28) // n), "n": n, "decades": rng.choice([0.0, 2.0])}
    if kind == "project":
        n = _between(rng, 8, 128)
        k = _between(rng, 1, 64)
        return {"kind": kind, "m": _between(rng, 5000, (1 << 26) // max(n, k)), "n": n, "k": k,
                "decades": rng.choice([0.0, 2.0, 3.0])}
    if kind == "lstsq":
        n = _between(rng, 4, 128)
        mixed = rng.random() < 0.5
        return {"kind": kind, "m": _between(rng, max(1000, 4 * n), (1 << (28 if mixed else 27)) // n), "n": n,
                "k": rng.randint(1, 8), "mixed": mixed, "decades": rng.choice([0.0, 2.0, 4.0])}
    if kind == "batch_r":
        return {"kind": kind, "count": _between(rng, 8, 2000), "m_max": _between(rng, 4000, 65536)}
    if kind == "batch_x":
        mixed = rng.random() < 0.5
        return {"kind": kind, "count": _between(rng, 2, 64 if mixed else 32), "m_max": _between(rng, 20000, 1000000),
                "mixed": mixed}
    n = _between(rng, 130, 512)
    return {"kind": kind, "m": _between(rng, max(3000, 3 * n), (1 << 26) // n), "n": n}


# ------------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randn(rows, cols, g):
    """Column-major rows x cols, iid N(0, 1)."""
    return torch.randn((cols, rows), generator=g, dtype=torch.float64, device="cuda").t()


def _matrix(m, n, decades, g):
    """G diag(sigma) V^T with sigma log-spaced over `decades` and V orthogonal; G itself for 0 decades."""
    G = _randn(m, n, g)
    if decades == 0.0 or n == 1:
        return G
    V, _ = torch.linalg.qr(_randn(n, n, g).contiguous())
    sigma = 10.0 ** (-decades * torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1))
    return torch.matmul(V * sigma, G.t()).t()


def _rhs(A, k, g, noise=1e-6):
    """A x + noise, x and the noise iid N(0, 1), column-major."""
    x = _randn(A.shape[1], k, g)
    return (torch.matmul(x.t(), A.t()) + noise * _randn(A.shape[0], k, g).t()).t()


def _sizes(case):
    """The (m, n, k, decades) of a batch's problems. They belong to the case; the seed makes the values."""
    r = np.random.default_rng([case["count"], case["m_max"]])
    out = []
    for _ in range(case["count"]):
        if case["kind"] == "batch_r":  # widths 8..64, m log-uniform from 256
            n = int(r.choice(BATCH_WIDTHS))
            out.append((max(n, int(math.exp(r.uniform(math.log(256), math.log(case["m_max"]))))), n, 0, 0.0))
        else:  # widths 16..128, 1..8 right-hand sides, condition numbers up to 1e4
            n, k = int(r.choice(SERVED_WIDTHS)), int(r.integers(1, 9))
            m = int(math.exp(r.uniform(math.log(1000), math.log(case["m_max"]))))
            out.append((m, n, k, float(r.uniform(0.1, 4.0))))
    return out


def _problems(case, seed):
    """The requests of a batch: R alone, alternately FP64 and mixed, or least squares in one precision."""
    g = _generator(seed)
    out = []
    for q, (m, n, k, decades) in enumerate(_sizes(case)):
        A = _matrix(m, n, decades, g)
        if case["kind"] == "batch_r":
            out.append({"A": A, "prec": ts.MIXED if q & 1 else ts.FP64})
        else:
            out.append({"A": A, "B": _rhs(A, k, g), "prec": ts.MIXED if case["mixed"] else ts.FP64, "want_r": False})
    return out


def _inputs(case, seed):
    g = _generator(seed)
    A = _matrix(case["m"], case["n"], case.get("decades", 0.0), g)
    if case["kind"] in ("qr_solve", "lstsq", "host"):
        return A, _rhs(A, case["k"], g)
    if case["kind"] == "project":
        return A, _randn(case["m"], case["k"], g)
    return A, None


def _tile_rows(m, n):
    """Leaves of one on-chip tile, as the benchmark plans its matrices."""
    return ts.plan_describe(m, n, 4096, 2, True)["tile_rows"]


def _views(sizes):
    """One buffer and column-major views (rows, cols) of it, so that a batch's results are one tensor."""
    buf = torch.empty(sum(r * c for r, c in sizes), dtype=torch.float64, device="cuda")
    out, at = [], 0
    for r, c in sizes:
        out.append(buf[at:at + r * c].view(c, r).t())
        at += r * c
    return buf, out


# -------------------------------------------------------------------- the passes
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch_r", "batch_x"):
        items = _problems(case, seed)
        name = "R" if kind == "batch_r" else "X"
        buf, views = _views([(it["A"].shape[1], it["A"].shape[1] if name == "R" else it["B"].shape[1]) for it in items])
        for it, v in zip(items, views):
            it[name] = v
        return {"kind": kind, "items": items, "out": buf}
    A, B = _inputs(case, seed)
    s = {"kind": kind, "A": A, "B": B, "case": case}
    m, n = A.shape
    if kind == "qr_solve":
        s["W"] = ts.colmajor(torch.empty_like(B))
        s["leaf_h"] = _tile_rows(m, n)
    elif kind == "orth":
        s["leaf_h"] = _tile_rows(m, n)
    elif kind == "project":
        s["F"] = ts.factor(A)
        s["W"] = torch.empty((case["k"], m), dtype=torch.float64, device="cuda").t()
    elif kind == "caqr":
        s["leaf_h"] = _tile_rows(m, 64)
    elif kind == "host":
        k = case["k"]
        for name, rows, cols in (("A", m, n), ("B", m, k), ("Q", m, n), ("R", n, n), ("X", n, k)):
            h = torch.empty((cols, rows), dtype=torch.float64, pin_memory=True).t()
            if name in ("A", "B"):
                h.copy_(s[name])
            s[name] = h
        s["leaf_h"] = _tile_rows(m, n)
        s["done"] = torch.cuda.Event()
    return s


def run(s):
    kind = s["kind"]
    if kind in ("batch_r", "batch_x"):
        ts.batch_solve(s["items"])
        return s["out"]
    A, case = s["A"], s["case"]
    if kind == "qr":
        F = ts.factor(A, leaf_h=case["leaf_h"], two_level=case["two_level"])
        Q = F.form_q()
        F.free()
        return {"Q": Q, "R": F.R}
    if kind == "qr_solve":
        F = ts.factor(A, leaf_h=s["leaf_h"], cluster=True)
        Q = F.form_q()
        s["W"].copy_(s["B"])
        X = F.solve_r(F.apply_qt(s["W"]))
        F.free()
        return {"Q": Q, "R": F.R, "X": X}
    if kind == "orth":
        Q, R = ts.orthonormalize(A, leaf_h=s["leaf_h"])
        return {"Q": Q, "R": R}
    if kind == "project":
        W = s["W"]
        W.copy_(s["B"])
        s["F"].apply_qt(W)
        W[: case["n"]].zero_()
        s["F"].apply_q(W)
        return W
    if kind == "lstsq":
        return ts.lstsq(A, s["B"], leaf_h=512 if case["mixed"] else 256, prec=ts.MIXED if case["mixed"] else ts.FP64)
    if kind == "caqr":
        F = ts.caqr(A, panel=64, leaf_h=s["leaf_h"])
        Q = F.form_q()
        F.free()
        return {"Q": Q, "R": F.R}
    ts.qr_solve_host(A, s["B"], Q=s["Q"], R=s["R"], X=s["X"], leaf_h=s["leaf_h"])
    s["done"].record()  # the program reads its results here
    s["done"].synchronize()
    return {"Q": s["Q"], "R": s["R"], "X": s["X"]}


# --------------------------------------------------------------- what it takes
def _qr_flops(m, n):
    return 2.0 * m * n * n - 2.0 * n ** 3 / 3.0


def work(case):
    kind = case["kind"]
    if kind in ("batch_r", "batch_x"):
        sizes = _sizes(case)
        return {"bytes": sum(8.0 * (m * (n + k) + (n * k if k else n * n)) for m, n, k, _ in sizes),
                "flops": sum(_qr_flops(m, n) + 4.0 * m * n * k for m, n, k, _ in sizes)}
    m, n, k = case["m"], case["n"], case.get("k", 0)
    if kind in ("qr", "orth", "caqr"):
        return {"bytes": 8.0 * (2 * m * n + n * n), "flops": 2 * _qr_flops(m, n)}
    if kind in ("qr_solve", "host"):
        return {"bytes": 8.0 * (2 * m * n + m * k + n * n + n * k),
                "flops": 2 * _qr_flops(m, n) + 4.0 * m * n * k - 2.0 * n * n * k + n * n * k}
    if kind == "project":
        return {"bytes": 8.0 * (m * n + 2 * m * k), "flops": 2 * (4.0 * m * n * k - 2.0 * n * n * k)}
    return {"bytes": 8.0 * (m * n + m * k + n * k), "flops": _qr_flops(m, n) + 4.0 * m * n * k}


# -------------------------------------------------------------- in plain 64 bits
def _exact_qr(A):
    Q, R = torch.linalg.qr(A)
    d = torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(R.dtype)
    return Q * d, R * d[:, None]


def _exact_solve(Q, R, A, B):
    """Least squares by the thin Q, with one step of refinement."""
    X = torch.linalg.solve_triangular(R, torch.matmul(Q.t(), B), upper=True)
    return X + torch.linalg.solve_triangular(R, torch.matmul(Q.t(), B - torch.matmul(A, X)), upper=True)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch_r", "batch_x"):
        parts = []
        for it in _problems(case, seed):
            if kind == "batch_r":
                R = torch.linalg.qr(it["A"], mode="r").R
                Z = R * torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(R.dtype)[:, None]
            else:
                Z = _exact_solve(*_exact_qr(it["A"]), it["A"], it["B"])
            parts.append(Z.t().reshape(-1))
        return torch.cat(parts)
    A, B = _inputs(case, seed)
    Q, R = _exact_qr(A)
    if kind == "project":
        W = B - torch.matmul(Q, torch.matmul(Q.t(), B))
        return W - torch.matmul(Q, torch.matmul(Q.t(), W))
    if kind == "lstsq":
        return _exact_solve(Q, R, A, B)
    if kind in ("qr_solve", "host"):
        return {"Q": Q, "R": R, "X": _exact_solve(Q, R, A, B)}
    return {"Q": Q, "R": R}
