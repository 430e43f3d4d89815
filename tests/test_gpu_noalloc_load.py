"""hsweep_apply_noalloc in a fresh process: CUDA loads a kernel into device memory at its first use,
so a call after hsweep_apply must not be the first to ask for any kernel."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROG = """
import sys
import numpy as np, torch
import synth
import paper_1007_4290_gb300 as hs
taken = 0
for n, prec, strong in ((64, 0, 0), (64, 1, 0), (127, 1, 2), (127, 0, 2)):
    c = torch.tensor(synth.velocity_constant(n), device="cuda")
    h = hs.hsweep_setup(c, 2 * np.pi * (n + 1) / 12, 8, 1e-6, hs.default_opts(precision=prec, strong_rank=strong))
    for nrhs in (1, 2, 3):
        r = torch.randn(nrhs, n * n, dtype=torch.complex128, device="cuda")
        z = torch.empty_like(r)
        ref = h.apply(r)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        hs.hsweep_apply_noalloc(h, r, z)
        torch.cuda.synchronize()
        taken += free - torch.cuda.mem_get_info()[0]
        assert torch.equal(z, ref)
print("taken", taken)
"""


def test_noalloc_after_apply_loads_nothing():
    r = subprocess.run([sys.executable, "-c", PROG], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.strip() == "taken 0", r.stdout
