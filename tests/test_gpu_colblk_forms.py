"""The blocked kernel A in its other forms (direct, more than 8 taps, single
polarisation as pairs of spectra): batch remainders, odd spectrum counts,
leading zero taps, several runs per CTA and several chunks, against the FP64
oracle."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HANN, WIN_RECT, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lg,taps,npol,mode,window,nspectra,blocks_a,chunk", [
    (20, 1, 2, DIRECT, WIN_HANN, 5, 0, 0), (20, 1, 2, DIRECT, WIN_RECT, 7, 16, 3), (20, 12, 2, PFB, WIN_HANN, 5, 8, 0),
    (20, 16, 2, PFB, WIN_HANN, 3, 0, 0), (20, 5, 1, PFB, WIN_HANN, 5, 16, 0), (20, 8, 1, PFB, WIN_HANN, 9, 16, 4),
    (20, 1, 1, DIRECT, WIN_HANN, 3, 0, 0), (19, 8, 1, PFB, WIN_HANN, 11, 8, 0), (19, 16, 1, PFB, WIN_RECT, 4, 0, 3),
    (18, 8, 1, PFB, WIN_HANN, 1, 0, 0), (18, 3, 1, PFB, WIN_HANN, 17, 4, 0), (18, 13, 1, PFB, WIN_HANN, 13, 4, 7),
])
def test_blocked_forms_match_oracle(oracle_mod, lg, taps, npol, mode, window, nspectra, blocks_a, chunk):
    from paper_1411_0436_gb300.vspec import Plan
    N = 1 << lg
    bank = Bank(N, taps, npol, mode, window, nspectra, rho=0.3 if npol == 2 else 0.0,
                tones=(Tone(25.0, N * 0.3 + 0.4, (0, 1) if npol == 2 else (0,)),))
    x = workloads.generate(bank, 6100 + lg + taps)
    o = oracle_mod.channelize(x, N, taps, npol, nspectra, mode, window)
    with Plan(N, taps, npol, mode, window) as plan:
        tuning = {"blocks_a": blocks_a}
        if chunk:
            tuning["chunk_spectra"] = chunk
        plan.tune(**tuning)
        assert "A=gather-blocked" in plan.describe() and "N1=2048" in plan.describe()
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), nspectra, acc)
        torch.cuda.synchronize()
    got = acc.cpu().numpy().astype(np.float64)
    assert_close(got.reshape(N, 4) if npol == 2 else got, o, what=f"2^{lg} P{taps} pol{npol} S{nspectra}")
