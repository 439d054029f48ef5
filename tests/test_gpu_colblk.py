"""The blocked kernel A of the longest pre-filtered transforms (2^20 channels):
batch remainders, ring rotation over several batches, leading zero taps,
several runs per CTA and several chunks, against the FP64 oracle."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import PFB, WIN_HAMMING, WIN_HANN, WIN_RECT, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N = 1 << 20


@pytest.mark.parametrize("taps,window,nspectra,blocks_a,chunk", [
    (8, WIN_HANN, 1, 0, 0), (8, WIN_HANN, 4, 8, 0), (8, WIN_HAMMING, 13, 16, 0), (5, WIN_HANN, 7, 24, 0),
    (1, WIN_RECT, 3, 0, 0), (8, WIN_HANN, 6, 0, 5),
])
def test_blocked_kernel_matches_oracle(oracle_mod, taps, window, nspectra, blocks_a, chunk):
    from paper_1411_0436_gb300.vspec import Plan
    bank = Bank(N, taps, 2, PFB, window, nspectra, rho=0.3, tones=(Tone(25.0, N * 0.3 + 0.4, (0, 1)),))
    x = workloads.generate(bank, 5200 + nspectra)
    o = oracle_mod.channelize(x, N, taps, 2, nspectra, PFB, window)
    with Plan(N, taps, 2, PFB, window) as plan:
        tuning = {"blocks_a": blocks_a}
        if chunk:
            tuning["chunk_spectra"] = chunk
        plan.tune(**tuning)
        if taps > 4:
            assert "A=gather-blocked" in plan.describe()
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), nspectra, acc)
        torch.cuda.synchronize()
    assert_close(acc.cpu().numpy().astype(np.float64).reshape(N, 4), o, what=f"P{taps} S{nspectra}")
