"""A batch whose banks run in one graph reports a row copy's wait that gave up
in any bank, once, and runs correctly afterwards."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HANN, WIN_RECT, Bank

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BANKS = [Bank(1024, 8, 2, PFB, WIN_HANN, 9), Bank(32768, 8, 2, PFB, WIN_HANN, 5),
         Bank(65536, 1, 2, DIRECT, WIN_RECT, 4)]


def test_batch_check_reports_a_banks_wait_once(oracle_mod):
    from paper_1411_0436_gb300 import vspec
    xs = [workloads.generate(b, 60 + i) for i, b in enumerate(BANKS)]
    d_in = [torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda() for x in xs]
    ns = [b.nspectra for b in BANKS]
    with vspec.Batch([(b.nchan, b.ntaps, b.npol, b.mode, b.window) for b in BANKS]) as batch:
        def accumulators():
            return [torch.zeros(batch.out_floats(i), dtype=torch.float32, device="cuda") for i in range(len(BANKS))]
        try:
            vspec.vspec_set_wait_limit(0)
            incomplete = accumulators()
            batch.execute(d_in, ns, incomplete)
            torch.cuda.synchronize()
        finally:
            vspec.vspec_set_wait_limit(-1)
        with pytest.raises(vspec.VspecError) as e:
            batch.check()
        assert e.value.status == vspec.ERR_DEVICE_TIMEOUT
        batch.check()  # cleared
        accs = accumulators()
        batch.execute(d_in, ns, accs)
        torch.cuda.synchronize()
        batch.check()
        for b, x, a in zip(BANKS, xs, accs):
            o = oracle_mod.channelize(x, b.nchan, b.ntaps, b.npol, b.nspectra, b.mode, b.window)
            assert_close(a.cpu().numpy().astype(np.float64).reshape(o.shape), o, what=f"bank {b.nchan} after a timeout")


def test_recorded_batch_follows_the_wait_limit():
    """A batch called again on the same buffers takes the limit in force, in
    either direction."""
    from paper_1411_0436_gb300 import vspec
    b = BANKS[1]
    d_in = torch.from_numpy(workloads.generate(b, 60).view(np.uint8).reshape(-1)).cuda()
    with vspec.Batch([(b.nchan, b.ntaps, b.npol, b.mode, b.window)]) as batch:
        acc = torch.zeros(batch.out_floats(0), dtype=torch.float32, device="cuda")

        def call():
            batch.execute([d_in], [b.nspectra], [acc])
            torch.cuda.synchronize()

        call()
        batch.check()
        try:
            vspec.vspec_set_wait_limit(0)
            call()
        finally:
            vspec.vspec_set_wait_limit(-1)
        with pytest.raises(vspec.VspecError) as e:
            batch.check()
        assert e.value.status == vspec.ERR_DEVICE_TIMEOUT
        call()
        batch.check()
