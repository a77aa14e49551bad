"""The CSR CountSketch on rows whose columns ascend (plain adds) and on rows that do not (atomics), rows around
and past 32 entries, column counts that do and do not allow 16-byte stores."""
import numpy as np
import pytest

from oracle import estimator as E
from tests._gpu import lev_module, sketch_abs_scale, to_dev, to_np

pytestmark = pytest.mark.gpu


def _sketch(L, h, row_ptr, col, val, n, d, p, m):
    import torch
    out = torch.empty((m, d), dtype=torch.float32, device="cuda")
    L.lev_sketch_csr(h, to_dev(row_ptr), to_dev(col), to_dev(val), n, d, p, out)
    return to_np(out)


@pytest.mark.parametrize("d", [100, 101, 1024])
def test_csr_sketch_of_sorted_shuffled_and_repeated_columns(d):
    L = lev_module()
    h = L.Handle(0)
    n, s, m, seed = 3001, 97, 64, 9                              # about 31 rows a bucket
    rng = np.random.default_rng(d)
    lens = rng.choice([0, 1, 8, 31, 32, 33, 70], n)
    row_ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    cols = [np.sort(rng.choice(d, l, replace=False)) for l in lens]
    mix = [rng.permutation(l) for l in lens]
    col = np.concatenate(cols).astype(np.int32)
    val = rng.standard_normal(col.size).astype(np.float32)
    p = L.make_params(s=s, m=m, k=8, seed=seed, sketch_prec="fp32")
    got = _sketch(L, h, row_ptr, col, val, n, d, p, m)
    order = np.concatenate([row_ptr[i] + mix[i] for i in range(n)]).astype(np.int64)
    # distinct columns: a column takes one sum a row, whatever the order within it
    assert np.array_equal(got, _sketch(L, h, row_ptr, col[order], val[order], n, d, p, m))

    def dense(c):
        A = np.zeros((n, d))
        np.add.at(A, (np.repeat(np.arange(n), lens), c), val.astype(np.float64))
        return A
    # (97 + 45) roundings a sum at most, each 2^-24 of the scale
    A = dense(col)
    assert np.all(np.abs(got - E.sketch(A, s, m, seed)) <= 1e-5 * sketch_abs_scale(A, s, m, seed) + 1e-30)
    twice = (col // 2).astype(np.int32)                          # neighbours meet in one column
    A = dense(twice)
    scale = np.zeros((n, d))
    np.add.at(scale, (np.repeat(np.arange(n), lens), twice), np.abs(val).astype(np.float64))
    got2 = _sketch(L, h, row_ptr, twice, val, n, d, p, m)
    assert np.all(np.abs(got2 - E.sketch(A, s, m, seed)) <= 1e-5 * sketch_abs_scale(scale, s, m, seed) + 1e-30)
    h.close()
