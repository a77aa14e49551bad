"""The pivoted Cholesky with its columns in registers (csrc/gramqr.cu) at the edges of its sizes: one row a
thread at 256, 512 and 1,024 threads, one to eight columns a CTA, an odd last column."""
import numpy as np
import pytest

from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("twins", [False, True])
@pytest.mark.parametrize("d", [1, 2, 3, 31, 255, 256, 257, 258, 304, 305, 511, 512, 513, 1023, 1024])
def test_factor_and_pivots(d, twins):
    import torch
    L = lev_module()
    h = L.Handle(0)
    rng = np.random.default_rng(d)
    A = rng.standard_normal((2 * d + 9, d)).astype(np.float32)
    if twins:                                              # equal columns: the lower index is the pivot
        A[:, d - d // 2:] = A[:, :d // 2]
    perm = torch.empty(d, dtype=torch.int32, device="cuda")
    R = torch.empty((d, d), dtype=torch.float64, device="cuda")
    r = L.lev_rrqr(h, to_dev(A), 1e-4, perm, R)
    assert L.lev_device_status(h) == 0
    assert r == (d - d // 2 if twins else d)
    p, R = to_np(perm), to_np(R)
    assert sorted(p) == list(range(d))
    if twins:
        assert p[:r].max() < r
    # r subtractions an entry, each within a few 2^-47 of the columns' norms
    P = A[:, p[:r]].astype(np.float64)
    G = P.T @ P
    nrm = np.sqrt(np.diag(G))
    bound = 8 * r * 2.0 ** -47
    assert np.max(np.abs(R[:r, :r].T @ R[:r, :r] - G) / np.outer(nrm, nrm)) <= bound
    # each pivot is the largest remaining diagonal entry
    S = np.cumsum(R[:r, :r][::-1] ** 2, axis=0)[::-1]
    assert np.all(np.diag(R[:r, :r]) ** 2 >= np.triu(S).max(axis=1) - bound * nrm.max() ** 2)
    h.close()
