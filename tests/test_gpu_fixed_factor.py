"""The fixed-point factorization job: R, thin Q and the factorization
itself at the edges of its tiles, of its number range and of its input checks, against the
oracle. Tolerances are the library's stated ones (R 1e-12, backward error and orthogonality
1e-13): the job carries 60 bits per column, more than FP64 arithmetic does."""
import numpy as np
import pytest

import oracle
from paper_0912_2572_gb300 import inputs
from conftest import to_dev, to_host

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _check(ts, A, Ad=None, **kw):
    F = ts.factor(to_dev(A) if Ad is None else Ad, **kw)
    Q, R = to_host(F.form_q()), to_host(F.R)
    F.free()
    assert _rel(R, oracle.r_factor(A)) <= 1e-12
    assert oracle.backward_error(A, Q, R) <= 1e-13
    assert oracle.orth_error(Q) <= 1e-13
    return R, Q


# widths at the edges of the column groups (2, 4 and 8 columns a warp), heights at the edges
# of a lane's rows and of the tile, chains whose last tile holds one row, tree nodes
@pytest.mark.parametrize("m,n,h,arity,two", [
    (1, 1, 1, 2, True), (513, 1, 512, 2, True), (1025, 8, 512, 2, True), (1537, 9, 512, 0, True),
    (64, 16, 64, 2, False), (65, 16, 64, 2, True), (2049, 16, 256, 4, False), (577, 17, 288, 0, True),
    (33, 32, 32, 2, False), (865, 32, 288, 0, True), (161, 33, 160, 2, True), (145, 64, 144, 0, True),
    (433, 64, 144, 0, True), (64, 64, 64, 2, False), (4097, 63, 64, 3, False), (3000, 41, 41, 16, False),
    (66, 65, 65, 2, True), (289, 127, 144, 0, True), (1153, 128, 144, 2, False), (900, 96, 100, 3, False),
])
def test_fixed_point_edges(cuda_lib, m, n, h, arity, two):
    import paper_0912_2572_gb300 as ts
    _check(ts, inputs.gaussian(m, n, m + n), leaf_h=h, arity=arity, two_level=two)


@pytest.mark.parametrize("off", [0, 1])
def test_fixed_point_misaligned_columns(cuda_lib, off):
    """Odd leading dimensions and an 8-byte base: row pairs without 16-byte alignment."""
    import torch
    import paper_0912_2572_gb300 as ts
    m, n, ld = 2000, 24, 2003
    buf = torch.zeros(ld * n + 1, dtype=torch.float64, device="cuda")
    Ad = buf[off:off + ld * n].view(n, ld).t()[:m]
    A = inputs.gaussian(m, n, 5)
    Ad.copy_(to_dev(A))
    R0, Q0 = _check(ts, A)
    R1, Q1 = _check(ts, A, Ad)
    assert np.array_equal(R0, R1) and np.array_equal(Q0, Q1)


def test_fixed_point_column_scales(cuda_lib):
    """Columns scaled over 400 decades (each has its own exponent), and a chain whose tiles
    grow by decades (the exponent grows along the chain)."""
    import paper_0912_2572_gb300 as ts
    m, n = 3000, 40
    A = inputs.gaussian(m, n, 6)
    s = 10.0 ** np.linspace(-100, 100, n)
    F = ts.factor(to_dev(A * s), leaf_h=144, arity=0)
    R, Q = to_host(F.R), to_host(F.form_q())
    F.free()
    assert _rel(R / s, oracle.r_factor(A)) <= 1e-12
    assert oracle.orth_error(Q) <= 1e-13
    g = 10.0 ** np.linspace(-8, 8, m)[:, None]
    for B in (A * g, A * g[::-1]):
        _check(ts, B, leaf_h=144, arity=0)


def test_fixed_point_degenerate_columns(cuda_lib):
    """Zero columns, a zero leading tile, repeated columns and a triangular matrix: H = I
    where a tail is empty, R within the oracle's normwise error, Q orthonormal."""
    import paper_0912_2572_gb300 as ts
    m, n = 1200, 20
    A = inputs.gaussian(m, n, 7)
    A[:, 3] = 0.0
    A[:, 9] = A[:, 2]
    A[:300, 5] = 0.0
    F = ts.factor(to_dev(A), leaf_h=100, arity=0)
    R, Q = to_host(F.R), to_host(F.form_q())
    F.free()
    assert oracle.backward_error(A, Q, R) <= 1e-13 and oracle.orth_error(Q) <= 1e-13
    assert np.all(R[:, 3] == 0.0) and abs(R[9, 9]) <= 1e-13 * np.linalg.norm(A[:, 9])
    T = np.triu(inputs.gaussian(64, 64, 8))
    F = ts.factor(to_dev(T), leaf_h=64)
    # one rounding of each entry to 2^-61 of 2^E, where the column's norm is above 0.47 2^E
    D = T * np.where(np.diag(T) < 0, -1.0, 1.0)[:, None]
    assert np.all(np.abs(to_host(F.R) - D) <= 2.0 ** -59 * np.linalg.norm(T, axis=0))
    F.free()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e-290, 1e290])
@pytest.mark.parametrize("row,n", [(10, 24), (500, 24), (1990, 24), (700, 90)])
def test_entries_outside_the_fixed_point_range(cuda_lib, bad, row, n):
    """A tile with an entry the fixed-point form cannot take goes through the FP64 job, and
    with it the rest of its chain: columns left of a non-finite entry are those of the clean
    matrix, columns from it on are not finite; tiny entries behave as zeros to FP64 rounding
    and huge ones (inside FP64, outside its squares) are not refused."""
    import paper_0912_2572_gb300 as ts
    m, c = 2000, 7
    A = inputs.gaussian(m, n, 9)
    Rc = oracle.r_factor(A)
    B = A.copy()
    if bad == 1e-290:
        B[row, :] = bad
        F = ts.factor(to_dev(B), leaf_h=144, arity=0)
        R, Q = to_host(F.R), to_host(F.form_q())
        assert _rel(R, oracle.r_factor(B)) <= 1e-12 and oracle.orth_error(Q) <= 1e-13
    else:
        B[row, c] = bad
        F = ts.factor(to_dev(B), leaf_h=144, arity=0)
        R = to_host(F.R)
        assert _rel(R[:, :c], Rc[:, :c]) <= 1e-12
        assert not np.all(np.isfinite(R[:, c]))
    F.free()


def test_non_finite_entry_in_a_wide_cluster_tree(cuda_lib):
    """A combine of more than 64 columns in the cluster tier that meets a non-finite triangle
    hands it to the FP64 job on half of its warps; the per-level tree gives the same R."""
    import paper_0912_2572_gb300 as ts
    m, n, c = 4000, 72, 30
    A = inputs.gaussian(m, n, 10)
    A[2500, c] = np.nan
    R = {}
    for cl in (False, True):
        F = ts.factor(to_dev(A), leaf_h=144, two_level=False, cluster=cl)
        R[cl] = to_host(F.R)
        F.free()
    assert np.array_equal(R[True], R[False], equal_nan=True)
    A[2500, c] = 0.0
    assert _rel(R[True][:, :c], oracle.r_factor(A)[:, :c]) <= 1e-12
    # row i of R takes column c only at reflector i; reflector c spoils every row from c on
    assert not np.any(np.isfinite(R[True][c, c:])) and not np.any(np.isfinite(R[True][:c, c]))


# right-hand sides factored along, or a pass of their own (64 < n + k, m above 24,000 k); chains
# and tree nodes of 9 to 16 columns on the FP64 job and beside it. Well-conditioned: both
# solutions are within 1e-12 of the normal one.
@pytest.mark.parametrize("m,n,k", [(24000, 64, 1), (24001, 64, 1), (48001, 60, 8), (300, 64, 64), (1000, 4, 8),
                                   (1025, 8, 1), (5000, 8, 8), (3000, 9, 3), (3000, 12, 1), (700, 2, 2)])
def test_lstsq_routes(cuda_lib, m, n, k):
    import paper_0912_2572_gb300 as ts
    A, B = inputs.gaussian(m, n, m + n), inputs.gaussian(m, k, m + k)
    X = to_host(ts.lstsq(to_dev(A), to_dev(B)))
    ref = np.linalg.lstsq(A, B, rcond=None)[0]
    assert np.linalg.norm(X - ref) <= 1e-12 * np.linalg.norm(ref) + 1e-12 * np.linalg.norm(B) / np.linalg.norm(A)


# a pass of Q^T B of its own: on both sides of the number of rows where it begins (20,000 from
# five columns on, 24,000 k below), 9 to 64 right-hand sides, more than 128 columns in all
@pytest.mark.parametrize("m,n,k", [(20000, 60, 5), (20001, 60, 5), (20001, 57, 8), (96001, 62, 4), (24001, 60, 9), (21000, 64, 64),
                                   (500, 128, 9), (2000, 128, 64), (300, 100, 33), (48001, 63, 2), (400, 126, 3)])
def test_lstsq_passes(cuda_lib, m, n, k):
    import paper_0912_2572_gb300 as ts
    A, B = inputs.gaussian(m, n, m + n), inputs.gaussian(m, k, m + k)
    X = to_host(ts.lstsq(to_dev(A), to_dev(B)))
    ref = np.linalg.lstsq(A, B, rcond=None)[0]
    assert np.linalg.norm(X - ref) <= 1e-12 * np.linalg.norm(ref) + 1e-12 * np.linalg.norm(B) / np.linalg.norm(A)


@pytest.mark.parametrize("m,n,k", [(40000, 128, 64)])
def test_more_right_hand_sides_do_not_repeat_the_pass(cuda_lib, m, n, k):
    """Least squares with k > 8 right-hand sides takes less than 2.5 times as long as with 8 (V
    is read once for up to 64 columns, not once for every 8)."""
    import torch
    import paper_0912_2572_gb300 as ts
    A = to_dev(inputs.gaussian(m, n, 1))
    t = {}
    for c in (8, k):
        B = to_dev(inputs.gaussian(m, c, 2))
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ts.lstsq(A, B)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        t[c] = best
    assert t[k] <= 2.5 * t[8], t
