"""The tensor-core Gaussian stage where its column tiles are not whole groups of 32 columns: above 256
columns the tiles are equal multiples of 16, and a tile's epilogue must not store past its last column."""
import numpy as np
import pytest

from oracle import estimator as E
from tests._gpu import lev_module, sketch_abs_scale, to_dev, to_np
from workloads import dense_gaussian

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,c", [("bf16x3", 1e-4), ("tf32", 2e-3), ("bf16", 1.6e-2)])
@pytest.mark.parametrize("d", [270, 281, 600, 599])
def test_sketch_with_tiles_of_an_odd_number_of_16_columns(prec, c, d):
    import torch
    L = lev_module()
    h = L.Handle(0)
    n, s, m, seed = 3000, 700, 300, 5
    A = dense_gaussian(n, d, seed=d).astype(np.float32)
    p = L.make_params(s=s, m=m, k=8, seed=seed, sketch_prec=prec)
    got = torch.empty((m, d), dtype=torch.float32, device="cuda")
    L.lev_sketch_dense(h, to_dev(A), p, got)
    A64 = A.astype(np.float64)
    want = E.sketch(A64, s, m, seed)
    # the operand roundings: the bound of the parity tests of this stage (c of |G||S||A| entrywise)
    assert np.all(np.abs(to_np(got) - want) <= c * sketch_abs_scale(A64, s, m, seed))
    again = torch.empty_like(got)
    L.lev_sketch_dense(h, to_dev(A), p, again)
    assert torch.equal(got, again)
    assert L.lev_device_status(h) == 0
    h.close()
