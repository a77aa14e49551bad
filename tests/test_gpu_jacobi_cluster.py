"""The one-sided Jacobi on a thread-block cluster (csrc/rank.cu) at the edges of its block layout: one to
sixteen CTAs, odd and padded blocks, row paddings to 128 elements, and the first sizes of the grid form."""
import numpy as np
import pytest

from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2, 3, 15, 16, 17, 31, 33, 65, 127, 129, 255, 257, 383, 385])
def test_singular_values_and_rows(d):
    import torch
    L = lev_module()
    h = L.Handle(0)
    rng = np.random.default_rng(d)
    A = (rng.standard_normal((2 * d + 5, d)) * np.geomspace(1.0, 1e-5, d)).astype(np.float32)
    p = L.make_params(s=16, m=A.shape[0], k=8, tau=1e-10, rank_svd=True)
    perm = torch.empty(d, dtype=torch.int32, device="cuda")
    R = torch.empty((d, d), dtype=torch.float64, device="cuda")
    sigma = torch.empty(d, dtype=torch.float64, device="cuda")
    r, _ = L.lev_rrqr_select(h, to_dev(A), p, perm, R, sigma)
    assert r == d and L.lev_device_status(h) == 0
    # a sweep rotates each row d - 1 times, each rotation within a few 2^-48; 12 sweeps and the FP64 QR of A
    want = np.linalg.svd(A.astype(np.float64), compute_uv=False)
    assert np.max(np.abs(to_np(sigma) - want) / want) <= 12 * (d + 1) * 2.0 ** -46
    _, sweeps = L.lev_rank_stats(h)
    assert sweeps <= 20
    h.close()
