"""Matrices whose rows differ in scale, the heavy rows first: the order in which Householder
QR in FP64 keeps the bits of every row (weighted least squares, soft equality constraints).
Solutions are compared with the exact ones (rational normal equations). A route's error may
be ten times that of Householder QR in FP64 (the oracle) or of sqrt(n) roundings, whichever
is larger; work rounded to a fixed fraction of the column's norm is off by the weight times
2^-61, 1e-11 at a weight of 1e8."""
import decimal
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_0912_2572_gb300 import inputs
from conftest import to_dev, to_host

pytestmark = pytest.mark.gpu


def _exact(A, B):
    """argmin ||B - A X|| in 150 digits from the exact normal equations."""
    def whole(M):
        out = np.empty(M.shape, dtype=object)
        out.flat = [int(Fraction(float(x)) * 2 ** 160) for x in M.flat]
        return out

    a, b = whole(A), whole(B)
    n, k = A.shape[1], B.shape[1]
    with decimal.localcontext() as ctx:
        ctx.prec = 150
        N = np.concatenate([a.T.dot(a), a.T.dot(b)], axis=1)
        M = np.empty(N.shape, dtype=object)
        M.flat = [decimal.Decimal(x) for x in N.flat]
        for j in range(n):  # Gaussian elimination of a positive definite matrix
            for i in range(j + 1, n):
                M[i, j:] -= M[j, j:] * (M[i, j] / M[j, j])
        X = np.empty((n, k), dtype=object)
        for i in range(n - 1, -1, -1):
            for c in range(k):
                X[i, c] = (M[i, n + c] - sum((M[i, l] * X[l, c] for l in range(i + 1, n)), decimal.Decimal(0))) / M[i, i]
        return X.astype(np.float64)


def _problem(m, n, k, kind, w, seed):
    """A, B with rows weighted by w: `dense` three heavy rows first; `few` twenty that involve
    three unknowns only; `falling` all rows, from w down to 1. (A heavy row that is not among
    the first of its leaf mixes into a light pivot row in FP64 too.)"""
    A = inputs.gaussian(m, n, seed)
    B = A @ inputs.gaussian(n, k, seed + 1) + 1e-3 * inputs.gaussian(m, k, seed + 2)
    s = np.ones(m)
    if kind == "dense":
        s[:3] = w
    elif kind == "falling":
        s = w ** np.linspace(1, 0, m)
    else:
        A[:20, 3:] = 0.0
        s[:20] = w
        B[:20] = A[:20] @ inputs.gaussian(n, k, seed + 1)
    return A * s[:, None], B * s[:, None]


def _tolerance(A, B, X):
    err = np.linalg.norm(oracle.lstsq(A, B) - X) / np.linalg.norm(X)
    return 10.0 * max(err, 2.0 ** -52 * np.sqrt(A.shape[1]))


CASES = [("dense", 1e4), ("dense", 1e8), ("dense", 1e12), ("dense", 1e15), ("few", 1e8), ("few", 1e12),
         ("falling", 1e10)]


@pytest.mark.parametrize("kind,w", CASES)
@pytest.mark.parametrize("m,n,k", [(900, 6, 2), (900, 24, 1), (1300, 40, 24), (700, 60, 2), (700, 100, 2)])
def test_weighted_lstsq(cuda_lib, kind, w, m, n, k):
    """One problem: a flat chain, the two-level tree and the binary tree, right-hand sides
    factored along."""
    import paper_0912_2572_gb300 as ts
    A, B = _problem(m, n, k, kind, w, 10 * n + k)
    X = _exact(A, B)
    tol = _tolerance(A, B, X)
    for kw in ({"arity": 0}, {}, {"leaf_h": max(n, 64), "two_level": False}):
        Z = to_host(ts.lstsq(to_dev(A), to_dev(B), **kw))
        err = np.linalg.norm(Z - X) / np.linalg.norm(X)
        assert err <= tol, (kw, err, tol)


# leaves of one and of several tiles (512, 288, 144, 96, 72 and 56 rows by width), tiles
# shorter than n, one chain and several with tree nodes
@pytest.mark.parametrize("kind,w", [c for c in CASES if c[1] != 1e12])
@pytest.mark.parametrize("m,n,k", [(2500, 6, 2), (1600, 24, 1), (1300, 40, 24), (900, 60, 33), (800, 100, 2),
                                   (700, 120, 16)])
def test_weighted_lstsq_batched(cuda_lib, kind, w, m, n, k):
    """FP64 items of a batch, beside an ordinary one, and the same requests served by the
    resident kernel (bitwise the same)."""
    import paper_0912_2572_gb300 as ts
    A, B = _problem(m, n, k, kind, w, 10 * n + k)
    X = _exact(A, B)
    tol = _tolerance(A, B, X)
    other = {"A": to_dev(inputs.gaussian(500, 9, 1)), "prec": ts.FP64}
    for chain_tiles in (2, 16):
        it = {"A": to_dev(A), "B": to_dev(B), "prec": ts.FP64}
        (R, Z), _ = ts.batch_solve([it, other], chain_tiles=chain_tiles)
        R, Z = to_host(R), to_host(Z)
        err = np.linalg.norm(Z - X) / np.linalg.norm(X)
        assert err <= tol, (chain_tiles, err, tol)
        with ts.Server(resident=True, chain_tiles=chain_tiles, ctas_per_sm=1) as srv:
            _, (Rs, Zs) = srv.submit(it)
            srv.drain()
            srv.poll()
        assert np.array_equal(to_host(Rs), R) and np.array_equal(to_host(Zs), Z)


def test_weighted_mixed_items(cuda_lib):
    """Tree nodes of mixed items: one chain's triangle far above the others'. R carries FP32
    leaf accuracy by rows of like scale, and X the refinement's."""
    import paper_0912_2572_gb300 as ts
    for n in (16, 60, 100):
        A = inputs.gaussian(6000, n, n)
        A[:1500] *= 1e6
        B = inputs.gaussian(6000, 2, n + 1)
        outs = ts.batch_solve([{"A": to_dev(A), "B": to_dev(B), "prec": ts.MIXED},
                               {"A": to_dev(A), "prec": ts.MIXED}], chain_tiles=1)
        X, R = to_host(outs[0][1]), to_host(outs[1][0])
        assert np.linalg.norm(R - oracle.r_factor(A)) <= 1e-5 * np.linalg.norm(R)
        Xo = oracle.lstsq(A, B)
        assert np.linalg.norm(X - Xo) <= 1e-9 * np.linalg.norm(Xo)


@pytest.mark.parametrize("kind,w", [c for c in CASES if c[1] != 1e12])
@pytest.mark.parametrize("m,n,k", [(900, 24, 12), (1300, 40, 24), (1500, 8, 40)])
def test_weighted_qt_b_then_solve(cuda_lib, kind, w, m, n, k):
    """Q^T B of more than 8 columns and the triangular solve, and the same through CAQR
    (whose trailing update is a Q^T B)."""
    import paper_0912_2572_gb300 as ts
    A, B = _problem(m, n, k, kind, w, 10 * n + k)
    X = _exact(A, B)
    tol = _tolerance(A, B, X)
    for how in ("chain", "tree", "caqr"):
        Ad = to_dev(A)
        if how == "caqr":
            F = ts.caqr(Ad, panel=(n + 1) // 2)
        else:
            F = ts.factor(Ad, arity=0 if how == "chain" else 2, two_level=how == "chain")
        Z = to_host(F.solve_r(F.apply_qt(to_dev(B))))
        F.free()
        err = np.linalg.norm(Z - X) / np.linalg.norm(X)
        assert err <= tol, (how, err, tol)


@pytest.mark.parametrize("m,n,two", [(900, 24, True), (1300, 40, False), (700, 100, True)])
def test_light_rows_of_q(cuda_lib, m, n, two):
    """Rows of Q far below their column keep their digits as rows: three rows weighted by
    1e12, the other rows of Q's first three columns are 1e-12 of them; and Q Q^T B = B for a
    B of such rows, by rows."""
    import paper_0912_2572_gb300 as ts
    A, B = _problem(m, n, 24, "dense", 1e12, n)
    F = ts.factor(to_dev(A), two_level=two)
    Q = to_host(F.form_q())
    Z = to_host(F.apply_q(F.apply_qt(to_dev(B))))
    F.free()
    Qo = oracle.qr(A)[0]
    assert np.linalg.norm((Q - Qo)[3:, :3]) <= 1e-12 * np.linalg.norm(Qo[3:, :3])
    assert np.linalg.norm((Q - Qo)[:, 3:]) <= 1e-12 * np.sqrt(n)
    assert oracle.orth_error(Q) <= 1e-13
    assert np.linalg.norm((Z - B)[3:]) <= 1e-12 * np.linalg.norm(B[3:])


@pytest.mark.parametrize("m,n,k,decades", [(1_000_000, 64, 32, 4.0), (4_000_000, 32, 16, 6.0)])
def test_small_components_of_tall_qt_b(cuda_lib, m, n, k, decades):
    """The same on tall matrices, where a tile is a small part of its column: consistent
    systems with exactly representable right-hand sides (A rounded to 2^-30, X small whole
    numbers), within 2.5 times the FP64 kernel's error."""
    import torch
    import paper_0912_2572_gb300 as ts
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    V = torch.linalg.qr(torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda"))[0]
    s = 10.0 ** (-decades * torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1))
    A = torch.randn((m, n), generator=g, dtype=torch.float64, device="cuda") @ (V * s).T
    A = ts.colmajor((A * 2.0 ** 30).round() / 2.0 ** 30)
    X = torch.randint(-8, 9, (n, k), generator=g, device="cuda").double()
    B = A @ X
    F = ts.factor(A, leaf_h=512)
    at_once = F.solve_r(F.apply_qt(ts.colmajor(B.clone())))
    eights = torch.cat([F.solve_r(F.apply_qt(ts.colmajor(B[:, c:c + 8].clone()))) for c in range(0, k, 8)], 1)
    F.free()
    assert float((at_once - X).norm()) <= 2.5 * float((eights - X).norm())


@pytest.mark.parametrize("k", [9, 16, 32])
@pytest.mark.parametrize("decades", [4.0, 6.0])
def test_small_components_of_qt_b(cuda_lib, decades, k):
    """B in the range of an ill-conditioned A: the components of Q^T B fall off like R's rows and
    R^-1 magnifies their errors. X through Q^T B of all columns at once is as near the exact
    solution (FP64 refined with residuals in extended precision) as eight columns at a time
    on the FP64 kernel, within a factor of two; so is X through CAQR."""
    import paper_0912_2572_gb300 as ts
    m, n = 20000, 32
    A = inputs.graded(m, n, decades, seed_g=int(decades) + k, seed_v=2)
    B = A @ inputs.gaussian(n, k, 3) + 1e-6 * inputs.gaussian(m, k, 4)
    Q, R = oracle.qr(A)[:2]
    X = np.zeros((n, k), np.longdouble)
    for _ in range(6):
        r = (B - A.astype(np.longdouble) @ X).astype(np.float64)
        X = X + np.linalg.solve(R, Q.T @ r)

    def err(Z):
        return float(np.linalg.norm(to_host(Z) - X) / np.linalg.norm(X))

    Ad, Bd = to_dev(A), to_dev(B)
    F = ts.factor(Ad, leaf_h=144)
    at_once = err(F.solve_r(F.apply_qt(to_dev(B))))
    by_eights = []
    for c in range(0, k, 8):
        by_eights.append(to_host(F.solve_r(F.apply_qt(to_dev(B[:, c:c + 8])))))
    F.free()
    e8 = err(to_dev(np.concatenate(by_eights, axis=1)))
    Fc = ts.caqr(Ad, panel=16)
    ec = err(Fc.solve_r(Fc.apply_qt(Bd)))
    Fc.free()
    print(f"at once {at_once:.2e}, by eights {e8:.2e}, caqr {ec:.2e}")
    assert at_once <= 2 * e8 and ec <= 2 * e8, (at_once, e8, ec)
