"""hsweep_setup and hsweep_import_layer end with their work done: the handle may be used on another
stream directly afterwards."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _apply(h, r, stream):
    h.set_stream(stream)
    with torch.cuda.stream(stream):
        z = h.apply(r)
    torch.cuda.synchronize()
    return z


@pytest.mark.parametrize("n,prec,strong", [(511, 1, 0), (255, 0, 0), (255, 1, 2)])
def test_setup_and_import_return_when_their_stream_is_idle(n, prec, strong):
    import paper_1007_4290_gb300 as hs
    c = torch.tensor(synth.velocity_lens(n), device="cuda")
    r = torch.randn(2, n * n, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s1):
        h = hs.hsweep_setup(c, 2 * np.pi * (n + 1) / 8, 8, 1e-6,
                            hs.default_opts(precision=prec, strong_rank=strong, core_kernel=1))
    idle = s1.query()
    z = _apply(h, r, s2)
    assert idle and torch.equal(z, _apply(h, r, s1))
    # import the same layer again (on a strong handle every layer is packed anew from the store)
    h.import_layer(n // 2, *h.export_layer(n // 2))
    idle = s1.query()
    zi = _apply(h, r, s2)
    assert idle and torch.equal(zi, _apply(h, r, s1))
    assert strong or torch.equal(zi, z)
    assert h.status()[0] == 0
    h.free()
