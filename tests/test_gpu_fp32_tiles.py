"""The FP32 final pass and Gaussian stage at the edges of their tiles: both row counts a thread takes, ragged
rows and columns, 16-byte and scalar loads, and K slices that end inside a 16-wide step."""
import numpy as np
import pytest

from oracle import estimator as E
from tests._gpu import lev_module, sketch_abs_scale, to_dev, to_np
from workloads import dense_gaussian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,k,lda", [(38911, 64, 256, 64), (38912, 64, 260, 68), (39041, 37, 300, 37),
                                       (40001, 256, 257, 256), (1, 5, 1, 5), (65, 17, 8, 20)])
def test_final_pass_row_tiles(n, d, k, lda):
    import torch
    L = lev_module()
    h = L.Handle(0)
    A = dense_gaussian(n, d, seed=n).astype(np.float32)
    M = dense_gaussian(d, k, seed=k).astype(np.float32)
    buf = torch.zeros((n, lda), device="cuda")
    buf[:, :d] = to_dev(A)
    theta = torch.empty(n, dtype=torch.float32, device="cuda")
    L.lev_final_dense(h, buf[:, :d], to_dev(M), "fp32", theta)
    Y = A.astype(np.float64) @ M.astype(np.float64)
    # the parity tolerance of the FP32 form, against sum_q (|a| |M|)_q^2 so that cancelling rows count as they round
    bound = np.sum((np.abs(A).astype(np.float64) @ np.abs(M).astype(np.float64)) * np.abs(Y), axis=1)
    assert np.all(np.abs(to_np(theta) - np.sum(Y * Y, axis=1)) <= 1e-5 * bound)
    h.close()


@pytest.mark.parametrize("n,d,s,m", [(3000, 132, 1604, 129), (3000, 256, 1000, 257), (2000, 260, 700, 128),
                                     (3000, 133, 1604, 129), (2000, 20, 1600, 80), (500, 7, 65, 28)])
def test_sketch_split_k(n, d, s, m):
    import torch
    L = lev_module()
    h = L.Handle(0)
    A = dense_gaussian(n, d, seed=d).astype(np.float32)
    p = L.make_params(s=s, m=m, k=8, seed=3)
    got = torch.empty((m, d), dtype=torch.float32, device="cuda")
    L.lev_sketch_dense(h, to_dev(A), p, got)
    A64 = A.astype(np.float64)
    assert np.all(np.abs(to_np(got) - E.sketch(A64, s, m, 3)) <= 2e-5 * sketch_abs_scale(A64, s, m, 3))
    h.close()
