"""The 2048-point row kernel with tensor-memory sums, at the sizes where its
item split can go wrong: fewer spectra than groups, group remainders, run
ends, ring wraps of the row buffers, several row tiles per CTA, several
chunks. Every case against the FP64 oracle within the FP32 tolerance."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import PFB, WIN_HANN, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nchan,nspectra,blocks_b,chunk", [
    (4096, 1, 0, 0), (4096, 3, 1, 0), (4096, 4, 0, 0), (4096, 5, 1, 0), (4096, 7, 1, 0), (4096, 8, 2, 0),
    (4096, 64, 1, 0), (4096, 65, 1, 0), (4096, 131, 1, 0), (4096, 131, 3, 0), (8192, 29, 1, 7),
    (16384, 11, 5, 0), (32768, 13, 3, 5),
])
def test_row_groups_match_oracle(oracle_mod, nchan, nspectra, blocks_b, chunk):
    from paper_1411_0436_gb300.vspec import PLAN_TWO_KERNEL, Plan
    bank = Bank(nchan, 8, 2, PFB, WIN_HANN, nspectra, rho=0.3, tones=(Tone(25.0, nchan * 0.3 + 0.4, (0, 1)),))
    x = workloads.generate(bank, 4100 + nspectra)
    o = oracle_mod.channelize(x, nchan, 8, 2, nspectra, PFB, WIN_HANN)
    d_in = torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda()
    with Plan(nchan, 8, 2, PFB, WIN_HANN, PLAN_TWO_KERNEL) as plan:
        assert "B=row2048" in plan.describe()
        tuning = {"blocks_b": blocks_b}
        if chunk:
            tuning["chunk_spectra"] = chunk
        plan.tune(**tuning)
        outs = []
        for _ in range(2):
            acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
            plan.execute(d_in, nspectra, acc)
            torch.cuda.synchronize()
            outs.append(acc.cpu().numpy())
        plan.check()
    assert np.array_equal(outs[0], outs[1])  # fixed summation order
    assert_close(outs[0].astype(np.float64).reshape(nchan, 4), o, what=f"N{nchan} S{nspectra} b{blocks_b} c{chunk}")
