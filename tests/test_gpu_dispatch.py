"""Which kernels a call runs: plan forms by whole tokens of describe() (the
general forms' names are parts of others), the sub-band path of interleaved
tiles for every tap class, and the band-by-band path that a small scratch takes."""
import numpy as np
import pytest

from parity_util import assert_close
from paper_1411_0436_gb300 import workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HAMMING, WIN_HANN, Bank, Tone

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,tokens", [
    ((1024, 8, 1, PFB), "A=none B=general-batched fir-in-B"),
    ((2048, 8, 2, PFB), "A=none B=row2048-batched fir-in-B"),
    ((65536, 4, 1, PFB), "A=general-paired B=row2048"),
    ((65536, 1, 1, DIRECT), "A=general-paired B=row2048"),
    ((16384, 4, 2, PFB), "A=colreg4 B=row2048"),
    ((16384, 12, 2, PFB), "A=colreg16 B=row2048"),
    ((1 << 20, 2, 2, PFB), "A=gather-blocked B=row2048"),
    ((1 << 20, 8, 1, PFB), "A=gather-blocked B=row2048"),
    ((1 << 20, 1, 1, DIRECT), "A=gather-blocked B=row2048"),
    ((262144, 8, 1, PFB), "A=gather-blocked B=row2048"),
    ((1 << 20, 12, 1, PFB), "A=gather B=general"),
], ids=lambda c: "-".join(map(str, c)) if isinstance(c, tuple) else "")
def test_plan_forms_by_whole_token(cfg, tokens):
    from paper_1411_0436_gb300.vspec import Plan
    with Plan(*cfg, WIN_HANN) as plan:
        d = plan.describe()
    assert not set(tokens.split()) - set(d.split()), (cfg, d)


def run_sub(cfg, prepare=lambda plan: None):
    """(per-band spectra, kernel-A launches, input) of one call."""
    from paper_1411_0436_gb300.vspec import Plan
    n, p, npol, mode, win, s, nsub = cfg
    bank = Bank(n, p, npol, mode, win, s, rho=0.3, tones=(Tone(20.0, n * 0.3 + 0.2, (0,)),))
    x = np.ascontiguousarray(np.stack([workloads.generate(bank, 130 + 7 * b) for b in range(nsub)], axis=1))
    with Plan(n, p, npol, mode, win, nsub=nsub) as plan:
        prepare(plan)
        plan.set_profiling(True)
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), s, acc)
        torch.cuda.synchronize()
        launches = {r[0]: r[1] for r in plan.kernel_stats()}["fir_colfft"]
        return acc.cpu().numpy().astype(np.float64).reshape(nsub, -1), launches, x


def assert_bands(oracle_mod, cfg, got, x):
    n, p, npol, mode, win, s, nsub = cfg
    for b in range(nsub):
        o = oracle_mod.channelize(np.ascontiguousarray(x[:, b]), n, p, npol, s, mode, win)
        assert_close(got[b].reshape(o.shape), o, what=f"{cfg} band {b}")


@pytest.mark.parametrize("cfg,chunk", [
    ((4096, 3, 2, PFB, WIN_HANN, 19, 8), 0), ((8192, 12, 2, PFB, WIN_HAMMING, 21, 4), 0),
    ((16384, 16, 2, PFB, WIN_HANN, 37, 2), 8), ((4096, 9, 2, PFB, WIN_HANN, 33, 16), 64),
    ((16384, 1, 2, PFB, WIN_HANN, 5, 4), 0), ((8192, 2, 2, PFB, WIN_HANN, 1, 8), 0),
    ((32768, 12, 2, PFB, WIN_HANN, 7, 8), 0),
], ids=lambda c: "-".join(map(str, c)) if isinstance(c, tuple) else f"chunk{c}")
def test_interleaved_tiles_of_other_tap_counts(oracle_mod, cfg, chunk):
    got, launches, x = run_sub(cfg, lambda plan: plan.tune(chunk_spectra=chunk) if chunk else None)
    assert launches == (1 if not chunk else -(-cfg[5] // chunk))  # every band in each launch
    assert_bands(oracle_mod, cfg, got, x)


@pytest.mark.parametrize("cfg", [
    (16384, 8, 2, PFB, WIN_HANN, 5, 3), (16384, 1, 2, DIRECT, WIN_HANN, 5, 5), (8192, 3, 2, PFB, WIN_HANN, 5, 4),
    (32768, 12, 2, PFB, WIN_HAMMING, 5, 8),
], ids=lambda c: "-".join(map(str, c)))
def test_small_scratch_runs_band_by_band(oracle_mod, cfg):
    def small(plan):  # fewer scratch spectra than bands
        plan.tune(chunk_spectra=2)
        plan.trim_scratch()
    got, launches, x = run_sub(cfg, small)
    assert launches == cfg[6] * 3  # ceil(5 / 2) chunks of each band
    assert_bands(oracle_mod, cfg, got, x)
