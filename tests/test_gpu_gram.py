"""The tensor-core Gram matrix (csrc/gram_tc.cu) at the edges of its tiles, chunks and row splits.

The first row of the pivoted Cholesky factor is the pivot's row of G over sqrt(G_pp), so R_00 R_0j gives
that row of G back with three roundings of the double-float arithmetic (at most 2^-46 each) on top of the
Gram's own error (FP64 grade, 2^-46 allowed): 8 x 2^-46 of sqrt(G_pp G_jj) bounds both. Every later row
adds one rounding a step: (d + 8) 2^-46 for the whole R^T R.
"""
import numpy as np
import pytest

from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return lev_module()


@pytest.fixture()
def h(L):
    handle = L.Handle(0)
    yield handle
    handle.close()


def _matrix(m, d, rows):
    rng = np.random.default_rng(m + d)
    A = rng.standard_normal((m, d))
    if rows == "lognormal":
        A *= np.exp(2.0 * rng.standard_normal((m, 1)))
    elif rows == "sparse":
        A *= rng.random((m, d)) < 0.1
    elif rows == "outlier":
        A[m // 2] *= 1e4
    A[:, 1] *= 2.0 ** -40                                  # a column of another scale
    return A.astype(np.float32)


# 1.5e8 products m d (d + 32) / 2 and 33 columns are the kernel's smallest; 128-column tiles, 192-row chunks
@pytest.mark.parametrize("m,d,rows", [(140000, 33, "normal"), (14500, 129, "lognormal"), (4100, 256, "outlier"),
                                      (4099, 257, "sparse"), (301, 1000, "normal"), (293, 1024, "lognormal"),
                                      (20011, 383, "normal")])
def test_gram_row_and_product_match_fp64(L, h, m, d, rows):
    import torch
    A = _matrix(m, d, rows)
    perm = torch.empty(d, dtype=torch.int32, device="cuda")
    R = torch.empty((d, d), dtype=torch.float64, device="cuda")
    r = L.lev_rrqr(h, to_dev(A), 1e-6, perm, R)
    assert L.lev_device_status(h) == 0
    P, R = to_np(perm).astype(np.int64), to_np(R)
    X = A[:, P].astype(np.longdouble)
    scale = np.sqrt((X * X).sum(axis=0).astype(np.float64))
    row = (X[:, :1] * X).sum(axis=0).astype(np.float64)
    assert np.max(np.abs(R[0, 0] * R[0] - row) / (scale[0] * scale)) <= 8 * 2.0 ** -46
    G = A[:, P].astype(np.float64).T @ A[:, P].astype(np.float64)
    E = np.abs(R.T @ R - G) / (scale[:, None] * scale[None, :])
    assert np.max(E[:r, :r]) <= (d + 8) * 2.0 ** -46 + m * 2.0 ** -53
    again = torch.empty_like(torch.from_numpy(R)).cuda()
    L.lev_rrqr(h, to_dev(A), 1e-6, perm, again)
    assert np.array_equal(to_np(again), R)                 # splits and chunks add in a fixed order


@pytest.mark.parametrize("lda", [129, 131, 132])
def test_gram_of_strided_rows(L, h, lda):
    import torch
    n, d = 14501, 129
    A = _matrix(n, d, "normal")
    buf = torch.full((n, lda), float("nan"), device="cuda")
    buf[:, :d] = to_dev(A)
    theta = torch.empty(n, dtype=torch.float32, device="cuda")
    want = torch.empty_like(theta)
    assert L.lev_exact_reference_dense(h, buf[:, :d], 1e-5, theta) == L.lev_exact_reference_dense(h, to_dev(A), 1e-5, want)
    np.testing.assert_allclose(to_np(theta), to_np(want), rtol=1e-5)


@pytest.mark.parametrize("m,d", [(2055, 1023), (4100, 258), (40000, 100)])
def test_equal_columns_tie(L, h, m, d):
    """Twin columns lie in tiles on and above the diagonal; their entries of G are the same numbers, so the
    lower index of each pair is the pivot and the rank is the number of pairs (and the odd column)."""
    import torch
    A = np.random.default_rng(d).standard_normal((m, d)).astype(np.float32)
    A[:, d - d // 2:] = A[:, :d // 2]
    perm = torch.empty(d, dtype=torch.int32, device="cuda")
    R = torch.empty((d, d), dtype=torch.float64, device="cuda")
    r = L.lev_rrqr(h, to_dev(A), 1e-4, perm, R)
    assert L.lev_device_status(h) == 0
    assert r == d - d // 2
    assert to_np(perm)[:r].max() < r
