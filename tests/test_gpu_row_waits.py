"""The row kernels' bounded waits for their row copies: vspec_set_wait_limit
governs them, a wait that gives up is reported once, and the plan runs normally
afterwards. A limit of 0 makes every wait give up at once (no GPU fault)."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HANN, WIN_RECT, Bank

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,nsub", [
    ((4096, 8, 2, PFB, WIN_HANN, 6), 1),         # a fused plan's own two-kernel plan
    ((65536, 1, 2, DIRECT, WIN_RECT, 40), 1),    # several rows per CTA: skipped copies
    ((65536, 8, 1, PFB, WIN_HANN, 7), 1),        # pairs of spectra
    ((1 << 19, 8, 2, PFB, WIN_HANN, 5), 1),      # 4096-point rows
    ((4096, 8, 2, PFB, WIN_HANN, 9), 4),         # sub-bands
], ids=lambda c: "-".join(map(str, c)) if isinstance(c, tuple) else f"nsub{c}")
def test_row_wait_that_gives_up_is_reported_once(oracle_mod, cfg, nsub):
    from paper_1411_0436_gb300 import vspec
    n, p, npol, mode, win, s = cfg
    bank = Bank(n, p, npol, mode, win, s, rho=0.3 if npol == 2 else 0.0)
    x = np.ascontiguousarray(np.stack([workloads.generate(bank, 40 + b) for b in range(nsub)], axis=1))
    d_in = torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda()
    with vspec.Plan(n, p, npol, mode, win, nsub=nsub) as plan:
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        try:
            vspec.vspec_set_wait_limit(0)
            plan.execute(d_in, s, acc)
            torch.cuda.synchronize()
        finally:
            vspec.vspec_set_wait_limit(-1)
        with pytest.raises(vspec.VspecError) as e:
            plan.check()
        assert e.value.status == vspec.ERR_DEVICE_TIMEOUT
        plan.check()  # cleared
        plan.dump(acc)
        plan.execute(d_in, s, acc)
        torch.cuda.synchronize()
        plan.check()
        got = acc.cpu().numpy().astype(np.float64).reshape(nsub, -1)
    for b in range(nsub):
        o = oracle_mod.channelize(np.ascontiguousarray(x[:, b]), n, p, npol, s, mode, win)
        assert_close(got[b].reshape(o.shape), o, what=f"{cfg} band {b} after a timeout")
