"""The 4096-point row kernel (524288 channels with a pre-filter): one spectrum,
both groups and one, the ends of summation runs, several tiles per CTA and
several chunks, against the FP64 oracle."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import PFB, WIN_HAMMING, WIN_HANN, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N = 1 << 19


@pytest.mark.parametrize("taps,window,nspectra,blocks_b,chunk", [
    (8, WIN_HANN, 1, 0, 0), (8, WIN_HANN, 2, 100, 0), (8, WIN_HAMMING, 5, 3, 0), (4, WIN_HANN, 7, 0, 3),
    (8, WIN_HANN, 32, 128, 0), (8, WIN_HANN, 35, 1, 0),
])
def test_row4096_matches_oracle(oracle_mod, taps, window, nspectra, blocks_b, chunk):
    from paper_1411_0436_gb300.vspec import Plan
    bank = Bank(N, taps, 2, PFB, window, nspectra, rho=0.3, tones=(Tone(25.0, N * 0.3 + 0.4, (0, 1)),))
    x = workloads.generate(bank, 8800 + nspectra)
    o = oracle_mod.channelize(x, N, taps, 2, nspectra, PFB, window)
    with Plan(N, taps, 2, PFB, window) as plan:
        tuning = {"blocks_b": blocks_b}
        if chunk:
            tuning["chunk_spectra"] = chunk
        plan.tune(**tuning)
        assert "B=row4096" in plan.describe()
        outs = []
        for _ in range(2):
            acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
            plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), nspectra, acc)
            torch.cuda.synchronize()
            plan.check()
            outs.append(acc.cpu().numpy())
    assert np.array_equal(outs[0], outs[1])  # fixed summation order
    assert_close(outs[0].astype(np.float64).reshape(N, 4), o, what=f"P{taps} S{nspectra}")
