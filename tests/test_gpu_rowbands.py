"""Sub-band calls of one-row transforms, all bands in one launch of the batched
kernel: fewer spectra than CTAs per band, single polarisation, band counts that
do not divide the CTAs, against the FP64 oracle."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HAMMING, WIN_HANN, WIN_RECT, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,blocks_b", [
    ((1024, 8, 2, PFB, WIN_HANN, 19, 8), 0), ((1024, 8, 2, PFB, WIN_HANN, 3, 16), 0), ((512, 1, 1, DIRECT, WIN_RECT, 301, 3), 0),
    ((2048, 8, 2, PFB, WIN_HANN, 5, 4), 0), ((2048, 12, 2, PFB, WIN_HAMMING, 70, 2), 0), ((1024, 16, 1, PFB, WIN_HANN, 41, 7), 0),
    ((512, 8, 2, PFB, WIN_HANN, 33, 4), 5), ((512, 8, 2, PFB, WIN_HANN, 33, 4), 3),
], ids=lambda c: "-".join(map(str, c)) if isinstance(c, tuple) else f"blocks{c}")
def test_bands_in_one_launch_match_oracle(oracle_mod, cfg, blocks_b):
    from paper_1411_0436_gb300.vspec import Plan
    n, p, npol, mode, win, s, nsub = cfg
    bank = Bank(n, p, npol, mode, win, s, rho=0.3 if npol == 2 else 0.0, tones=(Tone(20.0, n * 0.3 + 0.2, (0,)),))
    x = np.ascontiguousarray(np.stack([workloads.generate(bank, 900 + 7 * b) for b in range(nsub)], axis=1))
    with Plan(n, p, npol, mode, win, nsub=nsub) as plan:
        if blocks_b:
            plan.tune(blocks_b=blocks_b)
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), s, acc)
        torch.cuda.synchronize()
        got = acc.cpu().numpy().astype(np.float64).reshape(nsub, -1)
    for b in range(nsub):
        o = oracle_mod.channelize(np.ascontiguousarray(x[:, b]), n, p, npol, s, mode, win)
        assert_close(got[b].reshape(o.shape), o, what=f"{cfg} band {b}")
