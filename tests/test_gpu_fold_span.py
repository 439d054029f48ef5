"""Calls of one launch fold partial-sum slots that nothing zeroes: a short call
after a long one on the same plan must not see the long call's slots, also
inside a captured graph (the call's kernels are dependent launches)."""
import pytest
import torch

from paper_1411_0436_gb300.vspec import DIRECT, PFB, Plan

pytestmark = pytest.mark.gpu

CASES = [(64, 8, 2, PFB, 1), (1024, 8, 2, PFB, 1), (2048, 12, 2, PFB, 1), (4096, 4, 2, PFB, 1), (8192, 8, 2, PFB, 4),
         (16384, 8, 1, PFB, 1), (32768, 8, 2, PFB, 1), (65536, 1, 2, DIRECT, 3), (131072, 8, 2, PFB, 1),
         (262144, 8, 1, PFB, 1), (524288, 8, 2, PFB, 1), (1048576, 1, 2, DIRECT, 1)]


@pytest.mark.parametrize("nchan,taps,npol,mode,nsub", CASES)
def test_short_call_after_a_long_one(nchan, taps, npol, mode, nsub):
    g = torch.Generator(device="cuda:0")
    g.manual_seed(nchan + taps)
    long, short = max(7, min(300, (1 << 22) // nchan)), 3
    n = (long + taps - 1) * nchan * nsub * npol * 2
    x = torch.randint(-100, 100, (n,), generator=g, dtype=torch.int8, device="cuda:0")

    def plan():
        return Plan(nchan, taps, npol, mode, 1, nsub=nsub)

    with plan() as fresh:
        want = torch.zeros(fresh.out_floats, device="cuda:0")
        fresh.execute(x, short, want)
    with plan() as p:
        acc = torch.zeros(p.out_floats, device="cuda:0")
        p.execute(x, long, acc)
        acc.zero_()
        p.execute(x, short, acc)
        assert torch.equal(acc, want)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            acc.zero_()
            p.execute(x, short, acc, stream=torch.cuda.current_stream())
        p.execute(x, long, torch.zeros_like(acc))
        for _ in range(2):
            graph.replay()
            assert torch.equal(acc, want)
