"""The pivoted Cholesky with its columns in shared memory (csrc/gramqr.cu), which a partition of a GPU with too few
SMs for the register form, or without room for a cluster, takes: the same pivots, rank and R, bit for bit, as the
cluster (d <= 256) and the register form give. LEV_FAULT=partition launches it on a whole GPU."""
import numpy as np
import pytest

from tests._gpu import lev_module, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("d", [1, 2, 4, 129, 255, 256, 257, 400, 401, 512, 513, 1023, 1024])
def test_same_factor_as_the_other_forms(monkeypatch, d, forced):
    import torch
    L = lev_module()
    h = L.Handle(0)
    rng = np.random.default_rng(d)
    A = rng.standard_normal((4 * d + 9, d)) * np.exp(rng.standard_normal(d))
    A[:, d - d // 4:] = A[:, :d // 4]                      # dependent columns: the rank stops short of d
    A = to_dev(A.astype(np.float32))
    order = torch.from_numpy(rng.permutation(d - d // 4).astype(np.int32)).cuda()
    p = L.make_params(s=8 * d, m=2 * d + 9, k=32, seed=1, perm_in=order, rank_in=order.numel())
    out = []
    for fault in (None, "partition"):
        if fault:
            monkeypatch.setenv("LEV_FAULT", fault)
        perm = torch.empty(d, dtype=torch.int32, device="cuda")
        if forced:                                         # the factor through the scores that it gives
            x = torch.empty(A.shape[0], device="cuda")
            r = L.lev_estimate_dense(h, A, p, x, perm)
        else:
            x = torch.empty((d, d), dtype=torch.float64, device="cuda")
            r = L.lev_rrqr(h, A, 1e-4, perm, x)
        assert L.lev_device_status(h) == 0
        out.append((r, to_np(perm), to_np(x)))
    h.close()
    assert out[0][0] == out[1][0] == d - d // 4
    assert np.array_equal(out[0][1], out[1][1])
    assert np.array_equal(out[0][2], out[1][2])
