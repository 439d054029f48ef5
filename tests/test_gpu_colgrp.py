"""The grouped kernel A: every column length, tap class and polarisation count,
batch remainders, odd chunks of single-polarisation pairs, several runs per
group and several chunks, against the FP64 oracle."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HAMMING, WIN_HANN, WIN_RECT, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,taps,npol,mode,window,nspectra,blocks_a,chunk", [
    # dual-pol pre-filter: up to 4, 8 and 16 taps
    (4096, 3, 2, PFB, WIN_HANN, 13, 2, 0), (8192, 4, 2, PFB, WIN_HANN, 9, 0, 0), (16384, 1, 2, PFB, WIN_RECT, 5, 0, 0),
    (32768, 2, 2, PFB, WIN_HAMMING, 7, 3, 0), (65536, 4, 2, PFB, WIN_HANN, 6, 0, 4), (131072, 4, 2, PFB, WIN_HANN, 3, 0, 0),
    (262144, 3, 2, PFB, WIN_HANN, 2, 0, 0), (65536, 8, 2, PFB, WIN_HANN, 11, 2, 0), (262144, 8, 2, PFB, WIN_HANN, 5, 8, 0),
    (4096, 16, 2, PFB, WIN_HANN, 37, 1, 0), (8192, 9, 2, PFB, WIN_HAMMING, 8, 0, 0), (32768, 12, 2, PFB, WIN_HANN, 19, 2, 7),
    (131072, 16, 2, PFB, WIN_HANN, 9, 4, 0), (262144, 12, 2, PFB, WIN_HANN, 18, 16, 0), (524288, 16, 2, PFB, WIN_HANN, 2, 0, 0),
    # single-pol pre-filter and direct mode: odd and even counts
    (4096, 8, 1, PFB, WIN_HANN, 1, 0, 0), (8192, 5, 1, PFB, WIN_HANN, 13, 2, 5), (65536, 8, 1, PFB, WIN_HANN, 7, 0, 0),
    (131072, 2, 1, PFB, WIN_HAMMING, 4, 0, 0), (131072, 8, 1, PFB, WIN_HANN, 5, 16, 0), (16384, 16, 1, PFB, WIN_HANN, 35, 1, 0),
    (4096, 1, 1, DIRECT, WIN_HANN, 9, 1, 0), (32768, 1, 1, DIRECT, WIN_RECT, 12, 0, 0), (65536, 1, 1, DIRECT, WIN_HAMMING, 5, 2, 3),
    (524288, 1, 1, DIRECT, WIN_HANN, 3, 0, 0),
    # dual-pol direct
    (4096, 1, 2, DIRECT, WIN_HANN, 11, 1, 0), (32768, 1, 2, DIRECT, WIN_HAMMING, 6, 2, 0), (65536, 1, 2, DIRECT, WIN_RECT, 9, 1, 4),
    (524288, 1, 2, DIRECT, WIN_HANN, 5, 8, 0),
])
def test_grouped_kernel_matches_oracle(oracle_mod, n, taps, npol, mode, window, nspectra, blocks_a, chunk):
    from paper_1411_0436_gb300.vspec import PLAN_TWO_KERNEL, Plan
    bank = Bank(n, taps, npol, mode, window, nspectra, rho=0.3 if npol == 2 else 0.0,
                tones=(Tone(25.0, n * 0.3 + 0.4, (0,)),))
    x = workloads.generate(bank, 7400 + nspectra)
    o = oracle_mod.channelize(x, n, taps, npol, nspectra, mode, window)
    with Plan(n, taps, npol, mode, window, PLAN_TWO_KERNEL) as plan:
        tuning = {"blocks_a": blocks_a}
        if chunk:
            tuning["chunk_spectra"] = chunk
        plan.tune(**tuning)
        d = plan.describe()
        assert ("A=general-paired" in d) if npol == 1 else ("A=col" in d), d
        outs = []
        for _ in range(2):
            acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
            plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), nspectra, acc)
            torch.cuda.synchronize()
            outs.append(acc.cpu().numpy())
    assert np.array_equal(outs[0], outs[1])  # fixed summation order
    got = outs[0].astype(np.float64)
    assert_close(got.reshape(n, 4) if npol == 2 else got, o, what=f"N{n} P{taps} pol{npol} S{nspectra}")
