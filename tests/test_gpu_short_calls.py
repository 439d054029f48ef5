"""Calls of one to a few spectra of the longest pre-filters, on either side of
the length below which they take the tap-gather kernel: every count gives the
oracle's spectrum, the two paths' calls add up in one accumulator, a tuned plan
keeps its own kernels, a captured call replays, and a scratch that was replaced is
the one that the next call uses."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import PFB, WIN_HANN, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,npol,counts", [(1 << 19, 3, 1, "1,3"), (1 << 19, 12, 2, "1,2,3"), (1 << 20, 7, 1, "1,2,3"),
                                             (1 << 20, 6, 1, "1"), (1 << 20, 9, 2, "1"), (1 << 19, 9, 1, "1,2,3")])
def test_short_calls_match_oracle_and_add_up(oracle_mod, n, p, npol, counts):
    from paper_1411_0436_gb300.vspec import Plan
    s = int(counts[-1]) + 2
    bank = Bank(n, p, npol, PFB, WIN_HANN, s, rho=0.3 if npol == 2 else 0.0, tones=(Tone(30.0, n * 0.13 + 0.3, (0,)),))
    x = workloads.generate(bank, 17 + p)
    d_in = torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda()
    frame = n * npol * 2  # bytes

    def oracle(first, count):
        part = x.reshape(-1)[first * frame:(first + count + p - 1) * frame].reshape((-1,) + x.shape[1:])
        return oracle_mod.channelize(np.ascontiguousarray(part), n, p, npol, count, PFB, WIN_HANN)

    with Plan(n, p, npol, PFB, WIN_HANN) as plan:
        assert f" | spectra={counts} two-kernel " in plan.describe() and " A=gather " in plan.describe()
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")

        def spectrum():
            torch.cuda.synchronize()
            plan.check()
            return acc.cpu().numpy().astype(np.float64)

        for count in range(1, s + 1):
            plan.dump(acc)
            plan.execute(d_in, count, acc)
            o = oracle(0, count)
            assert_close(spectrum().reshape(o.shape), o, what=f"{count} spectra")
        plan.dump(acc)  # one short call, then the rest
        plan.execute(d_in, 1, acc)
        plan.execute(d_in[frame:], s - 1, acc)
        o = oracle(0, s)
        assert_close(spectrum().reshape(o.shape), o, what="1 + rest")
        plan.dump(acc)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            plan.execute(d_in, 1, acc)
        graph.replay()
        o = oracle(0, 1)
        assert_close(spectrum().reshape(o.shape), o, what="captured")
        plan.tune(blocks_a=76)
        plan.dump(acc)
        plan.execute(d_in, 1, acc)
        assert_close(spectrum().reshape(o.shape), o, what="tuned")
        for chunk in (2, 8):  # the scratch that both plans use, smaller and larger than before
            plan.tune(blocks_a=0, chunk_spectra=chunk)
            plan.trim_scratch()
            for count in (1, 3):
                plan.dump(acc)
                plan.execute(d_in, count, acc)
                o = oracle(0, count)
                assert_close(spectrum().reshape(o.shape), o, what=f"{count} spectra, chunks of {chunk}")
