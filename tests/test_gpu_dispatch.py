"""Which sweep runs for which options: the automatic choice, and the kernels a caller asks for."""
import numpy as np
import pytest
import torch

from oracle.assemble import Discretization
from oracle.sweep_exact import solve_exact
from tests.helpers import layer_to_dense
from tests.test_gpu_setup import _problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    import paper_1007_4290_gb300 as m
    return m


# plan entry 7: 0 or 1 on slabs, the column slices of a row (more) in the team sweep
@pytest.mark.parametrize("n,prec,strong,nrhs", [(100, 1, 0, 3), (100, 0, 0, 1), (127, 1, 2, 2), (260, 1, 0, 9)])
def test_sweep_kernel_2_is_the_team_sweep(hs, n, prec, strong, nrhs):
    c, omega, pml = _problem(n, 3)
    h = hs.hsweep_setup(torch.tensor(c, device="cuda"), omega, pml, 1e-6,
                        hs.default_opts(precision=prec, strong_rank=strong, sweep_kernel=2))
    p = h.sweep_plan(nrhs)
    assert p["tma"] == 2 and p["leaves_per_chunk"] > 1, p
    rng = np.random.default_rng(n)
    r = rng.standard_normal((nrhs, n * n)) + 1j * rng.standard_normal((nrhs, n * n))
    z = h.apply(torch.tensor(r, device="cuda")).cpu().numpy()
    assert h.status()[0] == 0
    r_max = h.info()["r_max"]
    T = [layer_to_dense(n, 8, r_max, *h.export_layer(m)) for m in range(n)]
    disc = Discretization(c, omega, pml)
    for s in {0, nrhs - 1}:
        ref = solve_exact(disc, T, r[s])
        err = np.linalg.norm(z[s] - ref) / np.linalg.norm(ref)
        assert err < (1e-11 if prec == 0 else 1e-4), (s, err)      # as for the automatic choice
    h.free()
