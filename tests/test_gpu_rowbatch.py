"""The batched kernel of the one-row transforms (512 .. 2048 channels): batch
remainders, odd single-polarisation pairs, the ends of its summation runs,
every tap class, several chunks, against the FP64 oracle."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HAMMING, WIN_HANN, WIN_RECT, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,taps,npol,mode,window,nspectra,blocks_b,chunk", [
    (1024, 8, 2, PFB, WIN_HANN, 1, 0, 0), (1024, 8, 2, PFB, WIN_HANN, 9, 1, 0), (1024, 8, 2, PFB, WIN_HANN, 150, 1, 0),
    (1024, 5, 2, PFB, WIN_HAMMING, 31, 2, 11), (1024, 16, 2, PFB, WIN_HANN, 17, 2, 0),
    (1024, 1, 2, DIRECT, WIN_HANN, 23, 3, 0), (1024, 1, 2, PFB, WIN_RECT, 8, 1, 0),
    (1024, 8, 1, PFB, WIN_HANN, 1, 0, 0), (1024, 8, 1, PFB, WIN_HANN, 15, 1, 0), (1024, 8, 1, PFB, WIN_HANN, 131, 1, 0),
    (1024, 12, 1, PFB, WIN_HANN, 18, 1, 0), (1024, 1, 1, DIRECT, WIN_RECT, 33, 2, 10),
    (512, 8, 2, PFB, WIN_HANN, 300, 1, 0), (512, 3, 1, PFB, WIN_HANN, 45, 1, 0), (512, 16, 2, PFB, WIN_RECT, 19, 1, 0),
    (512, 9, 1, PFB, WIN_HAMMING, 301, 1, 0), (512, 1, 2, DIRECT, WIN_RECT, 37, 2, 0),
    (2048, 8, 2, PFB, WIN_HANN, 71, 1, 0), (2048, 8, 2, PFB, WIN_HANN, 5, 1, 3), (2048, 1, 2, DIRECT, WIN_HAMMING, 6, 1, 0),
    (2048, 8, 1, PFB, WIN_HANN, 7, 1, 0), (2048, 16, 1, PFB, WIN_HANN, 73, 1, 0), (2048, 1, 1, DIRECT, WIN_HANN, 3, 1, 0),
    (2048, 12, 2, PFB, WIN_HANN, 9, 0, 0), (2048, 16, 2, PFB, WIN_HANN, 75, 1, 0), (2048, 9, 2, PFB, WIN_RECT, 5, 1, 2),
])
def test_batched_rows_match_oracle(oracle_mod, n, taps, npol, mode, window, nspectra, blocks_b, chunk):
    from paper_1411_0436_gb300.vspec import PLAN_TWO_KERNEL, Plan
    bank = Bank(n, taps, npol, mode, window, nspectra, rho=0.3 if npol == 2 else 0.0,
                tones=(Tone(25.0, n * 0.3 + 0.4, (0,)),))
    x = workloads.generate(bank, 6300 + nspectra)
    o = oracle_mod.channelize(x, n, taps, npol, nspectra, mode, window)
    with Plan(n, taps, npol, mode, window, PLAN_TWO_KERNEL) as plan:
        tuning = {"blocks_b": blocks_b}
        if chunk:
            tuning["chunk_spectra"] = chunk
        plan.tune(**tuning)
        assert "-batched" in plan.describe()
        outs = []
        for _ in range(2):
            acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
            plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), nspectra, acc)
            torch.cuda.synchronize()
            outs.append(acc.cpu().numpy())
    assert np.array_equal(outs[0], outs[1])  # fixed summation order
    got = outs[0].astype(np.float64)
    assert_close(got.reshape(n, 4) if npol == 2 else got, o, what=f"N{n} P{taps} pol{npol} S{nspectra}")
