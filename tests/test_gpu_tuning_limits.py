"""Launch limits that stored tunings rely on: a plan accepts its largest
kernel-A launch, and the spectrum stays the oracle's."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, WIN_RECT, Bank

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,flags", [(4096, 0), (8192, 1), (16384, 1), (16384, 4)])
def test_direct_plans_accept_two_kernel_a_ctas_per_sm(oracle_mod, n, flags):
    from paper_1411_0436_gb300 import vspec
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bank = Bank(n, 1, 2, DIRECT, WIN_RECT, 301, rho=0.3)
    x = workloads.generate(bank, 5)
    with vspec.Plan(n, 1, 2, DIRECT, WIN_RECT, flags) as plan:
        limit = plan.get_tuning()[1]["blocks_a"]
        assert limit == 4 * 2 * sms, plan.describe()  # four waves
        plan.tune(blocks_a=limit, **({} if flags else {"two_kernel_from": 0}))
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), bank.nspectra, acc)
        torch.cuda.synchronize()
        got = acc.cpu().numpy().astype(np.float64)
    o = oracle_mod.channelize(x, n, 1, 2, bank.nspectra, DIRECT, WIN_RECT)
    assert_close(got.reshape(o.shape), o, what=f"{n} flags {flags}")
