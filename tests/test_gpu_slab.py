"""The sweep on dense-diagonal slabs (the automatic choice up to n = 1024): parity with the
oracle's exact sweep on the same layers at the edges of its tiles (ragged slabs, one CTA, empty
blocks, every right-hand-side group and its remainders), its two exchanges against the basic
kernel, and its bounded waits."""
import numpy as np
import pytest
import torch

from oracle.assemble import Discretization
from oracle.sweep_exact import solve_exact
from tests.test_gpu_apply import _import_random, _problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    import paper_1007_4290_gb300 as m
    return m


# n, precision, right-hand sides, rank cap: 9 one CTA; 33, 65, 130, 257 slabs of unequal rows;
# 64, 256 full ones; rank cap 3 leaves many empty blocks
CASES = [(9, 0, 1, 4), (9, 1, 3, 4), (33, 1, 1, 12), (64, 0, 2, 12), (65, 1, 4, 12), (65, 0, 5, 3), (100, 1, 8, 3),
         (127, 0, 3, 12), (130, 1, 2, 20), (130, 1, 16, 12), (200, 0, 1, 20), (256, 1, 9, 12), (257, 1, 33, 12)]


@pytest.mark.parametrize("n,prec,nrhs,r_max", CASES)
def test_slab_sweep_matches_exact_sweep_on_the_same_layers(hs, n, prec, nrhs, r_max):
    c, omega, pml = _problem(n, 2)
    disc = Discretization(c, omega, pml)
    h = hs.hsweep_create(torch.tensor(c, device="cuda"), omega, pml, 1e-6,
                         hs.default_opts(precision=prec, r_max=r_max))
    T = _import_random(hs, h, disc, n, 8, r_max, seed=n, mixed=prec == 1)
    rng = np.random.default_rng(n)
    R = rng.standard_normal((nrhs, n * n)) + 1j * rng.standard_normal((nrhs, n * n))
    Z = h.apply(torch.tensor(R, device="cuda")).cpu().numpy()
    assert h.status()[0] == 0
    for s in {0, nrhs // 2, nrhs - 1}:
        ref = solve_exact(disc, T, R[s])
        err = np.linalg.norm(Z[s] - ref) / np.linalg.norm(ref)
        assert err < (1e-12 if prec == 0 else 2e-5), (s, err)
    h.free()


@pytest.mark.parametrize("nrhs", [3, 61])
def test_both_exchanges_match_the_basic_sweep(hs, nrhs):
    # 16 CTAs a team; 61 right-hand sides are more groups than clusters of 16 fit at a time, and
    # go to the teams that exchange through L2 (plan entry 7)
    n = 530
    c, omega, pml = _problem(n, 4)
    ct = torch.tensor(c, device="cuda")
    R = torch.randn(nrhs, n * n, dtype=torch.complex128, device="cuda")
    Z = []
    for kernel in (0, 1):
        h = hs.hsweep_setup(ct, omega, pml, 1e-6, hs.default_opts(sweep_kernel=kernel, core_kernel=1))
        if kernel == 0:
            p = h.sweep_plan(nrhs)
            assert p["tma"] == 2 and p["team_ctas"] == 16 and p["leaves_per_chunk"] == (1 if nrhs > 56 else 0), p
        Z.append(h.apply(R))
        assert h.status()[0] == 0
        if kernel == 0:
            assert torch.equal(h.apply(R), Z[0])
        h.free()
    err = (torch.linalg.norm(Z[0] - Z[1]) / torch.linalg.norm(Z[1])).item()
    assert err < 2e-5, err


@pytest.mark.parametrize("n,prec,nrhs", [(127, 0, 1), (127, 1, 1), (530, 1, 61)])
def test_withheld_sums_time_out_and_every_cta_returns(hs, n, prec, nrhs, monkeypatch):
    c, omega, pml = _problem(n, 2)
    ct = torch.tensor(c, device="cuda")
    opts = hs.default_opts(precision=prec, core_kernel=1)
    h = hs.hsweep_setup(ct, omega, pml, 1e-6, opts)
    r = torch.randn(nrhs, n * n, dtype=torch.complex128, device="cuda")
    ref = h.apply(r)
    assert h.status()[0] == 0
    monkeypatch.setenv("HSWEEP_TEST_WAIT_LIMIT", "20000")
    monkeypatch.setenv("HSWEEP_TEST_WITHHOLD", "1")
    h.apply(r)
    code, layer = h.status()
    monkeypatch.delenv("HSWEEP_TEST_WAIT_LIMIT")
    monkeypatch.delenv("HSWEEP_TEST_WITHHOLD")
    assert code == hs.ERR_TIMEOUT and layer >= 0, (code, layer)
    h.free()
    h = hs.hsweep_setup(ct, omega, pml, 1e-6, opts)
    z = h.apply(r)
    assert h.status()[0] == 0
    assert torch.equal(z, ref)
    h.free()


# n, R, right-hand sides: ragged slabs of 2, 4, 8 and 16 CTAs, the rank from 1 to the largest
# that n = 127 takes, remainders of the right-hand-side groups
@pytest.mark.parametrize("n,R,nrhs", [(40, 2, 1), (63, 5, 3), (127, 1, 9), (127, 5, 2), (200, 2, 35), (260, 3, 5)])
def test_strong_format_slabs_match_the_exact_sweep_of_their_layers(hs, n, R, nrhs):
    # the slabs that the setup packs from the strongly admissible factors (plan kernel 3, plan
    # entry 7 at most 1), the records of the same layers, and the slabs packed anew from the
    # store once a layer is imported
    from tests.helpers import strong_to_dense
    import synth
    c, omega, pml = synth.velocity_lens(n), 2 * np.pi * (n + 1) / 8, 6
    h = hs.hsweep_setup(torch.tensor(c, device="cuda"), omega, pml, 1e-6, hs.default_opts(strong_rank=R))
    p = h.sweep_plan(nrhs)
    assert p["tma"] == 3 and p["leaves_per_chunk"] <= 1, p
    rng = np.random.default_rng(n + R)
    V = rng.standard_normal((nrhs, n * n)) + 1j * rng.standard_normal((nrhs, n * n))
    Vt = torch.tensor(V, device="cuda")
    Z = h.apply(Vt).cpu().numpy()
    assert h.status()[0] == 0
    Ts = [strong_to_dense(n, 8, R, *h.strong_export(m)) for m in range(n)]
    disc = Discretization(c, omega, pml)
    for s in {0, nrhs - 1}:
        ref = solve_exact(disc, Ts, V[s])
        assert np.linalg.norm(Z[s] - ref) / np.linalg.norm(ref) < 2e-5, s
    h.import_layer(0, *h.export_layer(0))
    p = h.sweep_plan(nrhs)
    assert p["tma"] == 2 and p["leaves_per_chunk"] <= 1, p
    Zs = h.apply(Vt)
    h.free()
    h = hs.hsweep_setup(torch.tensor(c, device="cuda"), omega, pml, 1e-6, hs.default_opts(strong_rank=R, sweep_kernel=2))
    Zw = h.apply(Vt)
    assert h.status()[0] == 0
    h.free()
    assert ((Zs - Zw).norm() / Zw.norm()).item() < 4e-5      # two sweeps, 2e-5 each
