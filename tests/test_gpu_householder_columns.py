"""The Householder pivoted QR with a column a CTA (small tau) at the edges of its register tiles, and just past
the sizes that it takes."""
import numpy as np
import pytest

from oracle import linalg as OL
from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,d", [(1, 1), (2, 3), (60, 127), (127, 40), (128, 100), (129, 5), (512, 200), (513, 200),
                                 (1024, 304), (1025, 60), (700, 305)])
def test_householder_with_a_column_a_block(m, d):
    import torch
    L = lev_module()
    h = L.Handle(0)
    rs = np.random.default_rng(1000 * m + d)
    At = (rs.standard_normal((m, d)) * np.exp(0.5 * rs.standard_normal(d))[None, :]).astype(np.float32)
    if d > 4:
        At[:, d - 1] = At[:, 1]                                  # a dependent column ends below tau
    perm = torch.empty(d, dtype=torch.int32, device="cuda")
    R = torch.empty((d, d), dtype=torch.float64, device="cuda")
    rank = L.lev_rrqr(h, to_dev(At), 1e-9, perm, R)
    q = OL.pivoted_qr(At.astype(np.float64), 1e-9)
    assert rank == q.rank
    gp = to_np(perm)
    assert np.array_equal(gp[:rank], q.perm[:rank])
    assert np.all(np.diff(gp[rank:]) > 0)
    gR = to_np(R)
    want = np.zeros((rank, d))
    at = {c: t for t, c in enumerate(gp)}
    for t, c in enumerate(q.perm):
        want[:, at[c]] = q.R[:rank, t]
    # O(u kappa) of Householder's R; the bound of the parity tests
    assert np.max(np.abs(gR[:rank] - want)) <= 1e-10 * np.max(np.abs(want))
    assert np.all(gR[rank:] == 0)
    again = torch.empty_like(R)
    L.lev_rrqr(h, to_dev(At), 1e-9, perm, again)
    assert torch.equal(R, again)
    assert L.lev_device_status(h) == 0
    h.close()
