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


def _far(lib, prec, Fa, Fb, R, eps, shared):
    ct = np.complex64 if prec == 32 else np.complex128
    (su, k), sw = Fa.shape, Fb.shape[0]
    Fa, Fb = Fa.astype(ct), Fb.astype(ct)
    F = np.concatenate([Fa.T.reshape(-1), Fb.T.reshape(-1)])
    O = np.zeros((su + sw) * R, ct)
    fn = lib.far_f32 if prec == 32 else lib.far_f64
    rc = fn(su, sw, k, R, ctypes.c_double(eps), int(shared), _p(F), _p(O))
    assert rc == 0, rc
    O = O.astype(complex)
    return (Fa.astype(complex) @ Fb.astype(complex).T, O[:su * R].reshape(R, su).T, O[su * R:].reshape(R, sw).T)


# a block of exact rank R whose singular values form a cluster: the projection is the block itself, as
# far as the right factor's columns are orthogonal (the rotations' tolerance, twice, and their rounding)
@pytest.mark.parametrize("prec,spread", [(32, 1e-4), (32, 1e-3), (32, 0.0), (64, 1e-8), (64, 1e-4), (64, 0.0)])
@pytest.mark.parametrize("su,sw,R,shared", [(16, 17, 8, True), (64, 60, 8, True), (128, 128, 7, False)])
def test_projection_of_a_cluster_is_the_block(lib, prec, spread, su, sw, R, shared):
    u = U32 if prec == 32 else U64
    rng = np.random.default_rng(su + R)
    q = [np.linalg.qr(rng.standard_normal((n, R)) + 1j * rng.standard_normal((n, R)))[0] for n in (su, sw)]
    s = 1 + spread * rng.standard_normal(R)
    S, A, B = _far(lib, prec, q[0] * s, q[1], R, 1e-9 if prec == 64 else 1e-6, shared)
    P = B / np.linalg.norm(B, axis=0)
    tol = 2 * (4e-7 if prec == 32 else 1e-15) + 60 * u
    assert np.abs(P.conj().T @ P - np.eye(R)).max() < tol
    assert np.linalg.norm(S - A @ B.T, 2) < R * tol
