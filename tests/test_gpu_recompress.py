"""The setup's recompression (pivoted Gram-Schmidt and Jacobi SVD of the cores) at the edges of
its paths, against the oracle's exact sweep: one pair of leaves, ragged blocks, no truncation
(strongly graded cores in complex128), and blocks of 128 rows (dense cores in complex64) and
one more (QR of the factors)."""
import numpy as np
import pytest
import torch

from oracle.assemble import Discretization
from oracle.sweep_exact import setup_exact
from tests.test_gpu_setup import _dense_layers, _problem

pytestmark = pytest.mark.gpu


# tolerances: those of the setup's parity tests without truncation; with eps_H = 1e-6, a bound of
# 2e-4 as there for truncated complex64 layers
@pytest.mark.parametrize("n,prec,eps,tol", [(9, 0, 0.0, 1e-10), (9, 1, 0.0, 2e-4), (47, 0, 0.0, 1e-10),
                                            (90, 0, 0.0, 1e-9), (90, 1, 0.0, 2e-4), (256, 1, 1e-6, 2e-4),
                                            (258, 1, 1e-6, 2e-4)])
def test_recompressed_layers_match_the_exact_sweep(n, prec, eps, tol):
    import paper_1007_4290_gb300 as hs
    c, omega, pml = _problem(n, 1)
    T = setup_exact(Discretization(c, omega, pml))
    r_max = min(56, max(4, (n + 1) // 2))
    h = hs.hsweep_setup(torch.tensor(c, device="cuda"), omega, pml, eps,
                        hs.default_opts(precision=prec, r_max=r_max))
    assert h.status()[0] == 0
    ms = [0, 1, n // 2, n - 1]
    D = _dense_layers(h, n, 8, r_max, ms)
    for m in ms:
        err = np.linalg.norm(D[m] - T[m]) / np.linalg.norm(T[m])
        assert err < tol, (m, err)
    h.free()
