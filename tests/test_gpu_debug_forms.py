"""The bounds-checked debug build over the kernel forms that plans run by
default: grouped columns for every tap class, direct columns, blocked columns,
pairs of single-pol spectra (odd counts), one-row kernels, sub-bands in every
staging, the short folds; several chunks. Every result matches the FP64 oracle
and no bounds check fires; describe() names the form that is meant to run."""
import json
import os
import subprocess
import sys

import pytest

from paper_1411_0436_gb300 import build as vbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, os, sys
import numpy as np
import torch
sys.path.insert(0, os.environ["VSPEC_ROOT"]); sys.path.insert(0, os.path.join(os.environ["VSPEC_ROOT"], "tests"))
import oracle
from parity_util import metrics
from paper_1411_0436_gb300 import vspec, workloads
from paper_1411_0436_gb300.workloads import DIRECT, PFB, WIN_HANN, WIN_RECT, Bank, Tone
lib = vspec.load()
assert lib._name.endswith("libvspec_debug.so"), lib._name
vspec.vspec_debug_flags(clear=True)
# (nchan, taps, npol, mode, window, spectra, flags, sub-bands, chunk), whole tokens of describe()
shapes = [
    ((16384, 3, 2, PFB, WIN_HANN, 21, 0, 1, 8), "A=colreg4 B=row2048"),
    ((131072, 8, 2, PFB, WIN_HANN, 19, 0, 1, 0), "A=colreg B=row2048"),
    ((262144, 12, 2, PFB, WIN_HANN, 6, 0, 1, 0), "A=colreg16 B=row2048"),
    ((1 << 19, 10, 2, PFB, WIN_HANN, 4, 0, 1, 0), "A=colreg16 B=row4096"),
    ((1 << 20, 8, 2, PFB, WIN_HANN, 3, 0, 1, 0), "A=gather-blocked B=row2048"),
    ((1 << 20, 1, 2, DIRECT, WIN_HANN, 3, 0, 1, 0), "A=gather-blocked B=row2048"),
    ((16384, 1, 2, DIRECT, WIN_HANN, 40, 1, 1, 16), "A=coldir B=row2048"),
    ((4096, 8, 1, PFB, WIN_HANN, 33, 0, 1, 0), "A=general-paired B=row2048"),
    ((65536, 12, 1, PFB, WIN_HANN, 9, 0, 1, 5), "A=general-paired B=row2048"),
    ((262144, 5, 1, PFB, WIN_HANN, 5, 0, 1, 0), "A=gather-blocked B=row2048"),
    ((1 << 19, 16, 1, PFB, WIN_HANN, 3, 0, 1, 0), "A=gather-blocked B=row2048"),
    ((8192, 1, 1, DIRECT, WIN_HANN, 21, 0, 1, 0), "A=general-paired B=row2048"),
    ((262144, 1, 1, DIRECT, WIN_RECT, 3, 0, 1, 2), "A=general-paired B=row2048"),
    ((512, 8, 2, PFB, WIN_HANN, 300, 0, 1, 0), "A=none B=general-batched fir-in-B"),
    ((1024, 12, 1, PFB, WIN_HANN, 77, 0, 1, 0), "A=none B=general-batched fir-in-B"),
    ((2048, 8, 2, PFB, WIN_RECT, 90, 1, 1, 0), "A=none B=row2048-batched fir-in-B"),
    ((2048, 16, 2, PFB, WIN_HANN, 31, 0, 1, 0), "A=none B=row2048-batched fir-in-B"),
    ((1024, 8, 2, PFB, WIN_HANN, 25, 0, 8, 0), "A=none B=general-batched fir-in-B"),
    ((4096, 8, 2, PFB, WIN_HANN, 19, 1, 8, 0), "A=colreg B=row2048"),
    ((8192, 12, 2, PFB, WIN_HANN, 13, 0, 4, 0), "A=colreg16 B=row2048"),
    ((16384, 3, 2, PFB, WIN_HANN, 11, 0, 2, 8), "A=colreg4 B=row2048"),
    ((16384, 8, 2, PFB, WIN_HANN, 9, 1, 3, 0), "A=colreg B=row2048"),
    ((65536, 1, 2, DIRECT, WIN_HANN, 5, 0, 8, 0), "A=coldir B=row2048"),
    ((32768, 1, 2, DIRECT, WIN_RECT, 5, 1, 5, 0), "A=coldir B=row2048"),
    ((4096, 8, 1, PFB, WIN_HANN, 7, 0, 3, 0), "A=general-paired B=row2048"),
]
out = []
for (n, p, npol, mode, win, s, flags, nsub, chunk), tokens in shapes:
    bank = Bank(n, p, npol, mode, win, s, rho=0.3 if npol == 2 else 0.0, tones=(Tone(30.0, n * 0.3 + 0.4, (0,)),))
    x = np.ascontiguousarray(np.stack([workloads.generate(bank, 90 + b) for b in range(nsub)], axis=1))
    with vspec.Plan(n, p, npol, mode, win, flags, nsub=nsub) as plan:
        if chunk:
            plan.tune(chunk_spectra=chunk)
        acc = torch.zeros(plan.out_floats, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x.view(np.uint8).reshape(-1)).cuda(), s, acc)
        torch.cuda.synchronize()
        g = acc.cpu().numpy().astype(np.float64).reshape(nsub, -1)
        desc = plan.describe()
    ratio = 0.0
    for b in range(nsub):
        o = oracle.channelize(np.ascontiguousarray(x[:, b]), n, p, npol, s, mode, win)
        ratio = max(ratio, metrics(g[b].reshape(o.shape), o)["ratio"])
    out.append({"shape": [n, p, npol, mode, win, s, flags, nsub, chunk], "plan": desc, "ratio": ratio,
                "missing": [t for t in tokens.split() if t not in desc.split()],
                "flags": vspec.vspec_debug_flags(clear=True)})
print(json.dumps(out))
"""


@pytest.mark.gpu
def test_every_default_form_stays_in_bounds():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vbuild.build()
    env = dict(os.environ, VSPEC_LIBRARY="debug", VSPEC_ROOT=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    for case in json.loads(r.stdout.strip().splitlines()[-1]):
        assert not case["missing"] and case["ratio"] <= 1.0 and case["flags"] == 0, case
