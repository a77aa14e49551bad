"""The right-factor solve at the edges of its blocks of 32 rows and of its column pairs."""
import numpy as np
import pytest

from oracle import estimator as E
from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["omega", "identity", "reduced"])
@pytest.mark.parametrize("d,r", [(1, 1), (32, 31), (33, 32), (64, 33), (65, 65), (100, 7), (257, 256), (1000, 993),
                                 (1024, 1024)])
def test_omega_factor_at_block_edges(d, r, form):
    import torch
    from scipy.linalg import solve_triangular
    L = lev_module()
    h = L.Handle(0)
    k = {"omega": 9, "identity": d, "reduced": d + 3}[form]
    rs = np.random.default_rng(7 * d + r)
    R = np.triu(rs.standard_normal((d, d)) * 0.02) + np.diag(1.0 + rs.random(d))
    gp = rs.permutation(d).astype(np.int32)
    flags = {"omega": 0, "identity": L.LEV_OMEGA_IDENTITY, "reduced": L.LEV_OMEGA_REDUCED}[form]
    Mf = torch.full((d, k), 5.0, dtype=torch.float32, device="cuda")
    d_rank = torch.tensor([r], dtype=torch.int64, device="cuda")
    L.lev_omega_factor(h, to_dev(R), to_dev(gp), d_rank, d, k, 31, flags, Mf)
    got = to_np(Mf).astype(np.float64)
    want = np.zeros((d, k))
    if form == "identity":
        want[gp[:r], :r] = solve_triangular(R[:r, :r], np.eye(r), lower=False)
    elif form == "reduced":
        Om = E.omega_factor(np.eye(r), k, 31)
        want[gp[:r], :r] = solve_triangular(R[:r, :r], np.linalg.cholesky(Om @ Om.T), lower=False)
    else:
        want[gp[:r]] = E.omega_factor(R[:r, :r], k, 31)
    # the bound of the parity tests of this solve
    assert np.max(np.abs(got - want)) <= 1e-6 * np.max(np.abs(want))
    assert np.all(got[want == 0] == 0)
    h.close()
