"""Device memory that a handle reserves: the dense-diagonal slabs only where its options can use them."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _reserved(n, **opts):
    """Bytes a handle holds after its creation and one imported layer."""
    import paper_1007_4290_gb300 as hs
    c = torch.tensor(synth.velocity_constant(n), device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    h = hs.hsweep_create(c, 2 * np.pi * (n + 1) / 8, 8, 1e-6, hs.default_opts(**opts))
    h.import_layer(0, *h.export_layer(0))
    used = free - torch.cuda.mem_get_info()[0]
    assert h.status()[0] == 0
    h.free()
    return used


@pytest.mark.parametrize("n,prec,strong", [(300, 1, 0), (200, 0, 0), (200, 0, 2)])
def test_slabs_are_reserved_only_where_the_options_can_use_them(n, prec, strong):
    es, leaf = (8, 16)[prec == 0], 8
    slack = 64 << 20                       # allocation granularity, buffers of the library's first call
    _reserved(n, precision=prec, strong_rank=strong)
    others = [_reserved(n, precision=prec, strong_rank=strong, **o)
              for o in (dict(sweep_kernel=1), dict(sweep_kernel=2), dict(team=4), dict(groups=2), dict(team_threads=256),
                        dict(sweep_tc=1))]
    assert max(others) - min(others) < slack // 8, others
    auto = _reserved(n, precision=prec, strong_rank=strong)
    # every slab holds its rows' dense diagonal and room for 48 columns a depth
    slabs = n * n * 48 * (4 if n > 256 or prec == 0 else 3) * es
    assert slabs > slack
    if strong:
        assert auto - min(others) < slack // 8, (auto, others)
    else:
        assert auto - min(others) > slabs, (auto, others)
