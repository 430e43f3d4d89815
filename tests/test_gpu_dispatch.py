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


# complex128 with more right-hand sides than clusters of 16 fit: eight and nine beyond 16 rows a
# slab run as teams of one right-hand side each, ten on slabs again; each can be captured after a
# call with more of them
@pytest.mark.parametrize("n,plans", [(255, {7: 0, 8: 0, 10: 0, 16: 8}), (300, {7: 0, 8: 8, 9: 8, 10: 0, 14: 0, 16: 8}),
                                     (511, {4: 0, 8: 8, 10: 0})])
def test_complex128_plans_between_slabs_and_teams(hs, n, plans):
    c, omega, pml = _problem(n, 3, ppw=16)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = hs.hsweep_setup(torch.tensor(c, device="cuda"), omega, pml, 1e-6, hs.default_opts(precision=0))
        got = {k: h.sweep_plan(k)["leaves_per_chunk"] for k in plans}
        assert got == plans
        r = torch.randn(max(plans), n * n, dtype=torch.complex128, device="cuda")
        top = max(k for k in plans if plans[k] == 0)
        z = h.apply(r[:top])
    s.synchronize()
    for k in plans:
        if k > top:
            continue
        with torch.cuda.stream(s):
            rk = r[:k].clone()
            zk = torch.zeros_like(rk)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            code = hs._lib.hsweep_apply(h.raw, hs._ptr(rk, torch.complex128), hs._ptr(zk, torch.complex128), k)
        assert code == hs.OK
        with torch.cuda.stream(s):
            g.replay()
            ref = h.apply(rk)
        s.synchronize()
        assert torch.equal(zk, ref), k
        # any two plans: rounding apart (the sweeps' parity bound in complex128, each)
        assert ((zk - z[:k]).norm() / z[:k].norm()).item() < 2e-11, k
    assert h.status()[0] == 0
    h.free()
