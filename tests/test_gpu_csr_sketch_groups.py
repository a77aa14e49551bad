"""The CSR CountSketch takes a bucket's rows 32 at a time: a group without a row of more than 32 entries by plain
adds past L1, a group with one by atomics with the long rows' entries loaded ahead. Columns are distinct, so each
entry of B is one sum in row order, and the sketch is the dense sketch of the same matrix bit for bit."""
import numpy as np
import pytest

from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


# (lengths, one row in `every` is the last length); about 80 rows a bucket: two whole groups and a part of one
@pytest.mark.parametrize("lens,every", [([0, 1, 7, 31, 32], 0), ([0, 5, 32, 33], 90), ([3, 32, 64], 40), ([9, 65], 60),
                                        ([2, 96, 97], 2), ([33], 1), ([200], 1)])
@pytest.mark.parametrize("d", [256, 257])
@pytest.mark.parametrize("shuffled", [False, True])
def test_equals_the_dense_sketch(lens, every, d, shuffled):
    import torch
    L = lev_module()
    h = L.Handle(0)
    n, s, m = 4003, 50, 64
    rng = np.random.default_rng(d + every)
    ln = rng.choice(lens[:-1] if every > 1 else lens, n)
    if every > 1:
        ln[rng.random(n) < 1.0 / every] = lens[-1]
    rp = np.concatenate([[0], np.cumsum(ln)]).astype(np.int64)
    A = np.zeros((n, d), dtype=np.float32)
    col = np.zeros(rp[-1], dtype=np.int32)
    for i in range(n):
        c = rng.choice(d, ln[i], replace=False)
        col[rp[i]:rp[i + 1]] = c if shuffled else np.sort(c)
    val = rng.standard_normal(rp[-1]).astype(np.float32)
    A[np.repeat(np.arange(n), ln), col] = val
    p = L.make_params(s=s, m=m, k=8, seed=4, sketch_prec="fp32")
    got, want = (torch.empty((m, d), device="cuda") for _ in range(2))
    L.lev_sketch_csr(h, to_dev(rp), to_dev(col), to_dev(val), n, d, p, got)
    L.lev_sketch_dense(h, to_dev(A), p, want)
    h.close()
    assert np.array_equal(to_np(got), to_np(want))
