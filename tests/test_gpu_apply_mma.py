"""The tensor-core apply (more than 8 columns of B, thin Q of more than 8 columns) at the
edges of its tiles, column groups, row groups and reflector panels, against the FP64 warp
kernel (the same factor set applied 8 columns at a time) and the oracle. Q^T B of a column is
unique given the factor set, so the two kernels agree to FP64 rounding of the products, below
1e-13 of the column's norm (the round-trip tolerance of the library's tests)."""
import numpy as np
import pytest

import oracle
from paper_0912_2572_gb300 import inputs
from conftest import to_dev, to_host

pytestmark = pytest.mark.gpu


def _by_eights(fn, B):
    """fn applied to 8 columns at a time: the warp kernel."""
    return np.hstack([to_host(fn(to_dev(np.asfortranarray(B[:, c:c + 8])))) for c in range(0, B.shape[1], 8)])


# leaf heights at the edges of 4-, 9- and 8-block tiles and of one, two and four row groups;
# widths at the edges of a panel (8 reflectors) and a column group; ragged last tiles of a row
@pytest.mark.parametrize("m,n,k,h,arity,two", [
    (9, 9, 9, 9, 2, False), (64, 64, 64, 64, 2, False), (65, 8, 10, 64, 2, True), (129, 1, 16, 64, 0, True),
    (1000, 17, 17, 144, 0, True), (289, 63, 63, 144, 0, True), (146, 64, 65, 145, 2, True), (577, 24, 33, 288, 0, True),
    (1025, 16, 9, 512, 0, True), (2500, 100, 130, 144, 2, False), (3000, 128, 24, 256, 4, False),
    (1500, 65, 72, 200, 0, True), (5000, 33, 12, 64, 16, False),
])
def test_matches_the_warp_kernel(cuda_lib, m, n, k, h, arity, two):
    import paper_0912_2572_gb300 as ts
    A, B = inputs.gaussian(m, n, m + n), inputs.gaussian(m, k, m + k)
    F = ts.factor(to_dev(A), leaf_h=h, arity=arity, two_level=two)
    for fn in (F.apply_qt, F.apply_q):
        got, ref = to_host(fn(to_dev(B))), _by_eights(fn, B)
        assert np.max(np.linalg.norm(got - ref, axis=0) / np.linalg.norm(ref, axis=0)) <= 1e-13
    Q = to_host(F.form_q())
    E = np.zeros((m, n))
    E[:n] = np.diag(np.where(np.diag(to_host(F.R)) < 0, -1.0, 1.0))
    F.free()
    assert oracle.orth_error(Q) <= 1e-13
    assert oracle.backward_error(A, Q, to_host(ts.factor(to_dev(A), leaf_h=h, arity=arity, two_level=two).R)) <= 1e-13


def test_odd_strides_scales_and_zero_columns(cuda_lib):
    """Columns of B 8-byte aligned only, scaled over 600 decades, and zero: each column has its
    own exponent, so a scaled column gives the scaled result to rounding."""
    import torch
    import paper_0912_2572_gb300 as ts
    m, n, k, ld = 3000, 40, 20, 3001
    A, B = inputs.gaussian(m, n, 1), inputs.gaussian(m, k, 2)
    B[:, 7] = 0.0
    s = 10.0 ** np.linspace(-300, 300, k)
    F = ts.factor(to_dev(A))
    ref = to_host(F.apply_qt(to_dev(B)))
    buf = torch.zeros(ld * k + 1, dtype=torch.float64, device="cuda")
    W = buf[1:1 + ld * k].view(k, ld).t()[:m]
    W.copy_(to_dev(B * s))
    got = to_host(F.apply_qt(W)) / s
    assert np.all(got[:, 7] == 0.0)
    nz = [c for c in range(k) if c != 7]
    assert np.max(np.linalg.norm((got - ref)[:, nz], axis=0) / np.linalg.norm(ref[:, nz], axis=0)) <= 1e-13
    F.free()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_columns_stay_alone(cuda_lib, bad):
    """A column of B with a non-finite entry gives a non-finite column, the others are bitwise
    those of the clean B; a non-finite column of A leaves the columns of the thin Q before it."""
    import paper_0912_2572_gb300 as ts
    m, n, k, c = 2000, 24, 16, 5
    A, B = inputs.gaussian(m, n, 3), inputs.gaussian(m, k, 4)
    F = ts.factor(to_dev(A), leaf_h=144, arity=0)
    clean = to_host(F.apply_qt(to_dev(B)))
    B2 = B.copy()
    B2[100, c] = bad
    got = to_host(F.apply_qt(to_dev(B2)))
    rest = [q for q in range(k) if q != c]
    assert np.array_equal(got[:, rest], clean[:, rest])
    assert not np.any(np.isfinite(got[:n, c]))
    Q0 = to_host(F.form_q())
    F.free()
    A2 = A.copy()
    A2[1200, 11] = bad
    F = ts.factor(to_dev(A2), leaf_h=144, arity=0)
    Q1 = to_host(F.form_q())
    F.free()
    assert np.all(np.isfinite(Q1[:, :11])) and np.linalg.norm(Q1[:, :11] - Q0[:, :11]) <= 1e-12
    assert not np.any(np.isfinite(Q1[:, 11]))


# 9 to 16 columns against few reflectors (n k <= 216: a CTA per job in FP64) and the first
# widths above it; tiles at the edges of its three heights (128, 256, 512 rows), ragged tails,
# a last group of 9 columns after 64
@pytest.mark.parametrize("m,n,k,h,arity,two", [
    (9, 1, 9, 9, 2, False), (129, 8, 16, 128, 0, True), (513, 13, 16, 256, 0, True), (2049, 24, 9, 512, 0, True),
    (1537, 12, 15, 512, 4, False), (700, 8, 73, 100, 16, False), (600, 14, 16, 257, 0, True),
])
def test_few_reflectors(cuda_lib, m, n, k, h, arity, two):
    test_matches_the_warp_kernel(cuda_lib, m, n, k, h, arity, two)


# 17 to 32 columns against fewer reflectors (n k <= 128), and the first widths above
@pytest.mark.parametrize("m,n,k,h,arity,two", [
    (129, 4, 32, 128, 0, True), (513, 7, 18, 256, 0, True), (2049, 5, 25, 512, 0, True), (1537, 4, 17, 512, 4, False),
    (700, 3, 31, 100, 16, False), (600, 5, 26, 257, 0, True), (600, 2, 33, 257, 0, True), (600, 1, 97, 64, 0, True),
])
def test_few_reflectors_and_more_columns(cuda_lib, m, n, k, h, arity, two):
    test_matches_the_warp_kernel(cuda_lib, m, n, k, h, arity, two)
