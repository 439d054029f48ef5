"""The shape that a plan reports, handed back by name, is accepted and gives the
same plan: the same kernels, and bit for bit the same spectrum."""
import pytest

from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HANN

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,npol,mode,flags", [
    (131072, 8, 1, PFB, 0), (262144, 3, 1, PFB, 0), (524288, 12, 1, PFB, 0), (1 << 20, 8, 1, PFB, 0),
    (524288, 1, 1, DIRECT, 0), (4096, 1, 1, DIRECT, 0), (1 << 20, 1, 1, DIRECT, 0),
    (262144, 2, 2, PFB, 0), (262144, 16, 2, PFB, 4), (524288, 9, 2, PFB, 1), (16384, 12, 2, PFB, 1),
    (1 << 20, 8, 2, PFB, 0), (1 << 20, 1, 2, DIRECT, 0),
])
def test_own_shape_gives_the_same_plan(n, p, npol, mode, flags):
    from paper_1411_0436_gb300.vspec import Plan
    s = 5
    g = torch.Generator(device="cuda")
    g.manual_seed(n + p)
    d_in = torch.randint(-90, 91, ((s + p - 1) * n * npol * 2,), dtype=torch.int8, device="cuda", generator=g)
    res = []
    shape = (0, 0)
    for _ in range(2):
        with Plan(n, p, npol, mode, WIN_HANN, flags, col_len=shape[0], tile_cols=shape[1]) as plan:
            acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
            plan.execute(d_in, s, acc)
            torch.cuda.synchronize()
            plan.check()
            res.append((plan.describe(), plan.shape(), acc))
            shape = plan.shape()
    assert res[0][:2] == res[1][:2]
    assert torch.equal(res[0][2], res[1][2])
