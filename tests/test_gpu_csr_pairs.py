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
