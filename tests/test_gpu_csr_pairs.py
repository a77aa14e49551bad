"""The CSR final pass by entry pairs (rows of at most 32 entries) at the edges of its row classes: every length
on its own, mixed lengths, columns that repeat or lie outside [0, d), and row counts off the groups of 32."""
import numpy as np
import pytest

from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


def _rows(lens, d, rng, outside):
    row_ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    nnz = int(row_ptr[-1])
    col = rng.integers(0, d, nnz).astype(np.int32)               # unsorted, with repeats
    if outside:
        at = rng.random(nnz) < 0.1
        col[at] = rng.choice(np.array([-1, d, d + 7], dtype=np.int32), int(at.sum()))
    return row_ptr, col, rng.standard_normal(nnz).astype(np.float32)


@pytest.mark.parametrize("d", [40, 257, 1024])
@pytest.mark.parametrize("length", [1, 2, 3, 7, 8, 9, 12, 15, 16, 17, 31, 32, None])
def test_pairs_at_the_edges_of_the_row_classes(length, d):
    import torch
    L = lev_module()
    h = L.Handle(0)
    n, k = 1003, 264                                             # nnz < n k / 8: the form by pairs
    rng = np.random.default_rng(d * 64 + (length or 0))
    lens = rng.integers(0, 33, n) if length is None else np.full(n, length)
    row_ptr, col, val = _rows(lens, d, rng, outside=length is None)
    M = rng.standard_normal((d, k)).astype(np.float32)
    theta = torch.full((n,), -1.0, dtype=torch.float32, device="cuda")
    L.lev_final_csr(h, to_dev(row_ptr), to_dev(col), to_dev(val), n, d, to_dev(M), "fp32", theta)
    got = to_np(theta).astype(np.float64)
    P = M.astype(np.float64) @ M.astype(np.float64).T
    want, scale = np.zeros(n), np.zeros(n)
    for i in range(n):
        e = slice(row_ptr[i], row_ptr[i + 1])
        ok = (col[e] >= 0) & (col[e] < d)
        c, v = col[e][ok], val[e][ok].astype(np.float64)
        T = np.outer(v, v) * P[np.ix_(c, c)]
        want[i], scale[i] = T.sum(), np.abs(T).sum()
    # P as an FP32 pair (2^-48) of a compensated Gram matrix, double-float sums of up to 528 terms (a few
    # 2^-48 a term at most), and the rounding to FP32
    assert np.all(np.abs(got - want) <= 2.0 ** -24 * np.abs(want) + 2.0 ** -38 * scale)
    assert L.lev_device_status(h) == 0
    h.close()


@pytest.mark.parametrize("n", [31, 33, 1100, 40000])
def test_long_rows_among_short_ones(n):
    """Rows of more than 32 entries, whose pass runs only when the short rows' pass met one: every row gets its score
    whichever group it is in, with one matrix after the other on the same handle."""
    import torch
    L = lev_module()
    h = L.Handle(0)
    d, k = 200, 512
    rng = np.random.default_rng(n)
    M = rng.standard_normal((d, k)).astype(np.float32)
    M64 = M.astype(np.float64)
    for frac in (0.2, 0.0, 0.2):
        lens = np.where(rng.random(n) < frac, rng.integers(33, 80, n), rng.integers(0, 12, n))
        if frac:
            lens[-1] = 33
        row_ptr, col, val = _rows(lens, d, rng, outside=False)
        theta = torch.full((n,), -1.0, dtype=torch.float32, device="cuda")
        L.lev_final_csr(h, to_dev(row_ptr), to_dev(col), to_dev(val), n, d, to_dev(M), "fp32", theta)
        got = to_np(theta).astype(np.float64)
        for i in list(range(min(n, 200))) + list(range(max(0, n - 200), n)):
            e = slice(row_ptr[i], row_ptr[i + 1])
            v = val[e].astype(np.float64)
            want = float(((v @ M64[col[e]]) ** 2).sum())
            # FP32 sums of at most 80 products a column, squared and summed over k: first-order bound
            bound = float(((np.abs(v) @ np.abs(M64[col[e]])) ** 2).sum())
            assert abs(got[i] - want) <= 2.0 ** -24 * (2 * 82 * bound + (k // 32 + 40) * want)
        assert np.all(got >= 0)
    h.close()
