"""Estimates in flight on several streams, one handle a stream (include/lev.h, thread safety): the factorisations'
cooperative grids and clusters of different sizes meet on the device; each call gives the scores that it gives
alone, and no bounded wait runs out."""
import pytest

from tests._gpu import lev_module

pytestmark = pytest.mark.gpu

# (d, tau): the cluster, the register grids of 512 and 1,024 threads, the Householder forms (tau < 1e-6)
MIXED = [(64, 1e-4), (256, 1e-4), (300, 1e-4), (512, 1e-4), (1000, 1e-4), (128, 1e-8), (304, 1e-8), (320, 1e-8)]


@pytest.mark.parametrize("kinds", [[(512, 1e-4)] * 6, [(1024, 1e-4)] * 6, [(300, 1e-8)] * 6, MIXED],
                         ids=["d512", "d1024", "householder", "mixed"])
def test_scores_with_batches_in_flight(kinds):
    import torch
    L = lev_module()
    n = 6000
    jobs = []
    for i, (d, tau) in enumerate(kinds):
        g = torch.Generator(device="cuda").manual_seed(i)
        A = torch.randn(n, d, generator=g, device="cuda")
        p = L.make_params(s=2048, m=2 * d, k=32, tau=tau, seed=i, sketch_prec="bf16x3")
        h, st = L.Handle(0), torch.cuda.Stream()
        want, got = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
        assert L.lev_estimate_dense(h, A, p, want) == d
        jobs.append((h, st, A, p, want, got))
    torch.cuda.synchronize()
    for _ in range(5):
        for _ in range(8):
            for h, st, A, p, want, got in jobs:
                with torch.cuda.stream(st):
                    L.lev_estimate_dense(h, A, p, got, want_rank=False)
        torch.cuda.synchronize()
        for h, st, A, p, want, got in jobs:
            assert L.lev_device_status(h) == 0
            assert torch.equal(got, want)
    for job in jobs:
        job[0].close()
