"""Layers imported into a handle without a setup: layers not imported are empty (T~_m = 0)."""
import numpy as np
import pytest
import torch

from oracle.assemble import Discretization
from oracle.sweep_exact import solve_exact
from tests.helpers import layer_to_dense, random_layer
from tests.test_gpu_apply import _problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    import paper_1007_4290_gb300 as m
    return m


# slabs of one, two and sixteen CTAs, the team sweep (an explicit team size) and the basic sweep
@pytest.mark.parametrize("n,opts", [(9, {}), (65, {}), (257, {}), (64, dict(precision=0)), (65, dict(team=4)),
                                    (65, dict(sweep_kernel=1))])
def test_apply_with_some_layers_imported(hs, n, opts):
    c, omega, pml = _problem(n, 2)
    disc = Discretization(c, omega, pml)
    h = hs.hsweep_create(torch.tensor(c, device="cuda"), omega, pml, 1e-6, hs.default_opts(r_max=12, **opts))
    mixed = opts.get("precision", 1) == 1
    rng = np.random.default_rng(n)
    scale = 0.3 / np.max(np.abs(disc.north)) / np.sqrt(n)
    r = rng.standard_normal((2, n * n)) + 1j * rng.standard_normal((2, n * n))
    rt = torch.tensor(r, device="cuda")
    T = [np.zeros((n, n), complex) for _ in range(n)]
    for m in (0, n // 2, n // 2 + 1):
        lv, fac, rk = random_layer(n, 8, 12, rng, scale)
        h.import_layer(m, lv, fac, rk)
        if mixed:
            lv = lv.astype(np.complex64).astype(np.complex128)
            fac = fac.astype(np.complex64).astype(np.complex128)
        T[m] = layer_to_dense(n, 8, 12, lv, fac, rk)
        z = h.apply(rt).cpu().numpy()
        assert h.status()[0] == 0
        for s in (0, 1):
            ref = solve_exact(disc, T, r[s])
            err = np.linalg.norm(z[s] - ref) / np.linalg.norm(ref)
            assert err < (2e-5 if mixed else 1e-12), (m, s, err)      # the sweeps' parity bounds
    h.free()
