"""The tensor-core Gram matrix (csrc/gram_tc.cu) of tall matrices, where a row split holds many chunks.

R_00 R_0j gives the pivot's row of G back with three roundings of the double-float arithmetic (at most 2^-46
each); 8 x 2^-46 of sqrt(G_pp G_jj) bounds them and the Gram's own error (FP64 grade, 2^-46 allowed). In FP32
pairs over a whole split, sums of equal terms drift past it: 1.6e-12 after 1,000 chunks."""
import numpy as np
import pytest

from tests._gpu import lev_module, to_np

pytestmark = pytest.mark.gpu

BOUND = 8 * 2.0 ** -46


def _first_row(L, A):
    import torch
    d = A.shape[1]
    h = L.Handle(0)
    perm = torch.empty(d, dtype=torch.int32, device="cuda")
    R = torch.empty((d, d), dtype=torch.float64, device="cuda")
    L.lev_rrqr(h, A, 1e-6, perm, R)
    assert L.lev_device_status(h) == 0
    h.close()
    R = to_np(R)
    return to_np(perm).astype(np.int64), R[0, 0] * R[0]


# splits of 1,024 and 38 chunks; of 9, one past the chunks that a pair sums, and of 8
@pytest.mark.parametrize("m,d", [(1 << 20, 1024), (286000, 513), (8200, 1000), (8192, 1000)])
def test_constant_columns(L, m, d):
    import torch
    x = np.random.default_rng(d).uniform(1.0, 2.0, d).astype(np.float32)
    p, row = _first_row(L, torch.from_numpy(x).cuda().repeat(m, 1))
    want = m * x[p[0]].astype(np.longdouble) * x[p].astype(np.longdouble)
    assert p[0] == np.argmax(x)
    assert np.max(np.abs(row - want) / want) <= BOUND


@pytest.mark.parametrize("m,d", [(1000003, 256), (1000003, 130)])
def test_rows_that_differ(L, m, d):
    import torch
    g = torch.Generator(device="cuda").manual_seed(d)
    A = torch.rand(m, d, generator=g, device="cuda") + 0.5
    p, row = _first_row(L, A)
    piv = A[:, int(p[0])].double()
    want = np.zeros(d, dtype=np.longdouble)
    nrm = np.zeros(d)
    for r0 in range(0, m, 1 << 12):                        # FP64 products of short blocks, added in long double
        X = A[r0:r0 + (1 << 12)].double()
        want += to_np(piv[r0:r0 + (1 << 12)] @ X)
        nrm += to_np((X * X).sum(0))
    scale = np.sqrt(nrm[p[0]] * nrm[p])
    assert np.max(np.abs(row - want[p]) / scale) <= BOUND


@pytest.fixture(scope="module")
def L():
    return lev_module()
