"""The slab sweep where its teams exchange through L2 (more groups of right-hand sides than clusters
of 16 CTAs fit): hsweep_apply_noalloc at the edge of its scratch, and capture into a CUDA graph,
also of launches in turn and of fewer right-hand sides than the buffers were sized for."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hs():
    import paper_1007_4290_gb300 as m
    return m


def _setup(hs, n, **opts):
    c = torch.tensor(synth.velocity_random(n, 1 / 8, 1), device="cuda")
    return hs.hsweep_setup(c, 2 * np.pi * (n + 1) / 12, 12, 1e-6, hs.default_opts(core_kernel=1, **opts))


def _l2(h, nrhs):
    p = h.sweep_plan(nrhs)
    return p["tma"] in (2, 3) and p["leaves_per_chunk"] == 1


@pytest.mark.parametrize("n", [258, 264, 270])
def test_noalloc_gives_the_bits_of_apply_up_to_the_end_of_its_scratch(hs, n):
    # the cache takes n * n * 8 bytes a right-hand side: the last few counts that are admitted
    # leave less behind it than the exchange slots need
    h = _setup(hs, n)
    most = hs.NOALLOC_SCRATCH_BYTES // (n * n * 8)
    seen = 0
    for nrhs in range(most + 1, most - 4, -1):
        r = torch.randn(nrhs, n * n, dtype=torch.complex128, device="cuda")
        z = torch.empty_like(r)
        code = hs._lib.hsweep_apply_noalloc(h.raw, hs._ptr(r, torch.complex128), hs._ptr(z, torch.complex128), nrhs)
        if code == hs.ERR_ARG:
            assert nrhs >= most
            continue
        assert code == hs.OK
        assert torch.equal(z, h.apply(r)), nrhs
        seen += _l2(h, nrhs)
    assert seen >= 1 and h.status()[0] == 0
    h.free()


# 61: one launch; 130: teams in turn; each captured after a call with `first` right-hand sides
@pytest.mark.parametrize("n,strong,nrhs,first", [(530, 0, 61, 61), (530, 0, 61, 100), (530, 0, 130, 130), (300, 2, 60, 64)])
def test_captured_exchange_through_l2_replays_the_eager_apply(hs, n, strong, nrhs, first):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = _setup(hs, n, strong_rank=strong)
        assert strong or _l2(h, nrhs)
        h.apply(torch.randn(first, n * n, dtype=torch.complex128, device="cuda"))
        r = torch.randn(nrhs, n * n, dtype=torch.complex128, device="cuda")
        z = torch.zeros_like(r)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        code = hs._lib.hsweep_apply(h.raw, hs._ptr(r, torch.complex128), hs._ptr(z, torch.complex128), nrhs)
    assert code == hs.OK
    for k in range(2):
        with torch.cuda.stream(s):
            r.copy_(torch.randn_like(r))
            ref = h.apply(r)
            g.replay()
        s.synchronize()
        assert torch.equal(z, ref), k
    assert h.status()[0] == 0
    h.free()
