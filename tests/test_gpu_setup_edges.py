"""The setup where a depth of the cluster tree has blocks of 128 and of 129 rows (n = 257, 513 to
515, 1025 and on): the smaller ones take the dense path of the recompression in complex64, the
larger ones the QR of their factors, in one launch."""
import numpy as np
import pytest
import torch

from oracle.assemble import Discretization
from tests.helpers import layer_to_dense
from tests.test_gpu_setup import _problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    import paper_1007_4290_gb300 as m
    return m


def exact_layers(disc, ms):
    """T_m of Algorithm 2.1 for the layers ms, dense in complex128 (on the GPU, by torch)."""
    out, T = {}, None
    for m in range(max(ms) + 1):
        S = torch.tensor(disc.A_mm(m), device="cuda")
        if m:
            D = torch.tensor(disc.A_off(m), device="cuda")
            S = S - D[:, None] * T * D[None, :]
        T = torch.linalg.inv(S)
        if m in ms:
            out[m] = T.cpu().numpy()
    return out


# the tolerance of the setup's parity tests for truncated complex64 layers
@pytest.mark.parametrize("n", [257, 515])
def test_layers_with_blocks_of_128_and_129_rows(hs, n):
    c, omega, pml = _problem(n, 1)
    ms = [0, 1, n // 2, n - 1]
    T = exact_layers(Discretization(c, omega, pml), ms)
    h = hs.hsweep_setup(torch.tensor(c, device="cuda"), omega, pml, 1e-6, hs.default_opts(precision=hs.MIXED, r_max=56))
    assert h.status()[0] == 0
    for m in ms:
        D = layer_to_dense(n, 8, 56, *h.export_layer(m))
        err = np.linalg.norm(D - T[m]) / np.linalg.norm(T[m])
        assert err < 2e-4, (m, err)
    h.free()


# small rank caps, where every other buffer of the recompression is small: the preconditioner is
# as good as the one of complex128 (whose blocks take neither path at these ranks)
@pytest.mark.parametrize("n,r_max", [(257, 12), (514, 24), (1025, 24)])
def test_small_rank_caps(hs, n, r_max):
    c, omega, pml = _problem(n, 2)
    ct = torch.tensor(c, device="cuda")
    f = torch.zeros(1, n * n, dtype=torch.complex128, device="cuda")
    f[0, (n // 2) * n + n // 3] = (n + 1.0) ** 2
    steps, u = [], []
    for prec in (hs.FP64, hs.MIXED):
        h = hs.hsweep_setup(ct, omega, pml, 1e-3, hs.default_opts(precision=prec, r_max=r_max))
        x, it, rr = h.solve(f, 1e-6)
        assert h.status()[0] == 0 and rr[0] < 1e-4
        steps.append(it[0])
        u.append(x)
        h.free()
    # one Arnoldi step more for the complex64 sweep's rounding, one for the last refinement step
    assert steps[1] <= steps[0] + 2, steps
    # both within tol of the solution in the preconditioned residual
    assert ((u[0] - u[1]).norm() / u[0].norm()).item() < 1e-3
