"""Requested splits of pre-filtered plans too long for a register FIR window
(kernel A's tap-gather form), among them the shapes the autotuner tries and
partial tiles: every tap is applied (against the FP64 oracle)."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import PFB, WIN_HAMMING, WIN_HANN, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,shapes", [
    ((1 << 20, 8, 2, WIN_HANN, 3), [(256, 0), (512, 8), (512, 0)]),
    ((1 << 20, 3, 1, WIN_HANN, 2), [(256, 16)]),
    ((1 << 19, 12, 2, WIN_HAMMING, 3), [(256, 16), (128, 8), (512, 0)]),
    ((1 << 19, 8, 1, WIN_HANN, 4), [(256, 16), (128, 0)]),
    ((1 << 18, 16, 1, WIN_HANN, 5), [(64, 64), (128, 0)]),
], ids=lambda c: "-".join(map(str, c)) if isinstance(c, tuple) else "")
def test_long_shaped_plans_match_oracle(oracle_mod, cfg, shapes):
    from paper_1411_0436_gb300.vspec import Plan
    n, p, npol, win, s = cfg
    bank = Bank(n, p, npol, PFB, win, s, rho=0.3 if npol == 2 else 0.0, tones=(Tone(30.0, n * 0.13 + 0.3, (0,)),))
    x = workloads.generate(bank, 71 + n)
    o = oracle_mod.channelize(x, n, p, npol, s, PFB, win)
    d_in = torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda()
    for n2, cols in shapes:
        with Plan(n, p, npol, PFB, win, col_len=n2, tile_cols=cols) as plan:
            shape, desc = plan.shape(), plan.describe()
            acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
            plan.execute(d_in, s, acc)
            torch.cuda.synchronize()
            got = acc.cpu().numpy().astype(np.float64)
        assert_close(got.reshape(o.shape), o, what=f"{cfg} shape {n2, cols}")
        assert shape[0] == n2 and "A=gather " in desc, desc
