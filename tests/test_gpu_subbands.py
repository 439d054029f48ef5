"""Sub-band calls whose kernel-A tiles are words of the interleaved rows
(power-of-two band counts), all bands in one launch per chunk: every column
form, short and long columns, several chunks, against the FP64 oracle."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HAMMING, WIN_HANN, WIN_RECT, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,chunk", [
    ((4096, 8, 2, PFB, WIN_HANN, 19, 8), 0), ((4096, 1, 2, DIRECT, WIN_HANN, 21, 4), 0),
    ((8192, 5, 2, PFB, WIN_HAMMING, 5, 16), 0), ((16384, 8, 2, PFB, WIN_HANN, 37, 2), 8),
    ((32768, 8, 2, PFB, WIN_HANN, 9, 8), 0), ((65536, 8, 2, PFB, WIN_RECT, 6, 4), 0),
    ((131072, 1, 2, DIRECT, WIN_HAMMING, 3, 8), 0), ((32768, 1, 2, DIRECT, WIN_RECT, 1, 2), 0),
], ids=lambda c: "-".join(map(str, c)) if isinstance(c, tuple) else f"chunk{c}")
def test_interleaved_tiles_match_oracle(oracle_mod, cfg, chunk):
    from paper_1411_0436_gb300.vspec import Plan
    n, p, npol, mode, win, s, nsub = cfg
    bank = Bank(n, p, npol, mode, win, s, rho=0.3, tones=(Tone(20.0, n * 0.3 + 0.2, (0,)),))
    x = np.ascontiguousarray(np.stack([workloads.generate(bank, 700 + 7 * b) for b in range(nsub)], axis=1))
    with Plan(n, p, npol, mode, win, nsub=nsub) as plan:
        if chunk:
            plan.tune(chunk_spectra=chunk)
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), s, acc)
        torch.cuda.synchronize()
        got = acc.cpu().numpy().astype(np.float64).reshape(nsub, -1)
    for b in range(nsub):
        o = oracle_mod.channelize(np.ascontiguousarray(x[:, b]), n, p, npol, s, mode, win)
        assert_close(got[b].reshape(o.shape), o, what=f"{cfg} band {b}")
