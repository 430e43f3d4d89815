"""Single kernels of the strongly admissible projection on constructed inputs, through
tests/kernels/strong_entries.cu."""
import ctypes

import numpy as np
import pytest

from tests.kernels import kernel_library

pytestmark = pytest.mark.gpu

U32, U64 = 2.0 ** -24, 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return kernel_library(tmp_path_factory, "strong")


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


# one row, a CTA's worth and one more, a large block; P = 16 and 10 vectors
@pytest.mark.parametrize("P,m,seed", [(16, 0, 0), (10, 77, 5)])
def test_test_vectors_are_the_library_s_normals_rounded(lib, P, m, seed):
    import paper_1007_4290_gb300 as hs
    rows = np.array([1, 16, 17, 128, 301], np.int32)
    host = []
    for blk, r in enumerate(rows):
        out = np.zeros((P, r, 2))
        assert hs._lib.hsweep_rsvd_normals(blk, m, seed, int(r), P, _p(out)) == hs.OK
        host.append((out[..., 0] + 1j * out[..., 1]).reshape(-1))
    host = np.concatenate(host)
    d64, d32 = np.zeros(len(host), np.complex128), np.zeros(len(host), np.complex64)
    assert lib.normals_f64(len(rows), _p(rows), P, m, seed, _p(d64)) == 0
    assert lib.normals_f32(len(rows), _p(rows), P, m, seed, _p(d32)) == 0
    # two libraries' logarithm, sine and square root: a few units in the last place (2 pi u is rounded
    # before the host's sine)
    assert np.abs(d64 - host).max() < 40 * U64 * 6
    for a, b in ((d32.real, d64.real), (d32.imag, d64.imag)):
        assert np.array_equal(a, b.astype(np.float32))
