"""Single kernels of the setup on constructed inputs, against NumPy in complex128: launched through
tests/kernels/setup_entries.cu, which is compiled with the library's own flags and objects."""
import ctypes

import numpy as np
import pytest

from tests.kernels import kernel_library

pytestmark = pytest.mark.gpu

U32, U64 = 2.0 ** -24, 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return kernel_library(tmp_path_factory, "setup")


def _types(prec):
    return (np.complex64, U32) if prec == 32 else (np.complex128, U64)


def _svd(lib, prec, C, eps, r_max=56, qcap=None):
    ct, _ = _types(prec)
    qa, qb = C.shape
    qcap = qcap or max(qa, qb)
    Cf = np.asfortranarray(C.astype(ct))
    Ta, Tb = np.zeros((r_max, qcap), ct), np.zeros((r_max, qcap), ct)
    rank = ctypes.c_int(-1)
    fn = lib.svd_f32 if prec == 32 else lib.svd_f64
    rc = fn(qa, qb, qcap, r_max, ctypes.c_double(eps), Cf.ctypes.data_as(ctypes.c_void_p),
            Ta.ctypes.data_as(ctypes.c_void_p), Tb.ctypes.data_as(ctypes.c_void_p), ctypes.byref(rank))
    assert rc == 0, rc
    k = rank.value
    return Ta[:k, :qa].T.astype(complex), Tb[:k, :qb].T.astype(complex), np.array(Cf, dtype=complex)


def _unitary(rng, n, k):
    return np.linalg.qr(rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k)))[0]


# eps, and sizes: one column, a leaf pair, ragged cores, the largest dense core of complex64
@pytest.mark.parametrize("prec,eps", [(32, 1e-6), (32, 1e-7), (32, 1e-3), (64, 1e-6), (64, 1e-12)])
@pytest.mark.parametrize("qa,qb", [(1, 1), (8, 7), (49, 98), (98, 49), (97, 97), (112, 112), (128, 127)])
def test_svd_keeps_the_singular_values_above_eps(lib, prec, eps, qa, qb):
    if prec == 64 and max(qa, qb) > 112:
        pytest.skip("beyond the cores of complex128")
    _, u = _types(prec)
    rng = np.random.default_rng(qa * 1000 + qb)
    q = min(qa, qb)
    s = 0.5 ** np.arange(q)
    C = (_unitary(rng, qa, q) * s) @ _unitary(rng, qb, q).conj().T
    Ta, Tb, C = _svd(lib, prec, C, eps)
    s = np.linalg.svd(C, compute_uv=False)
    # rounding of a column update and of a rotation: a few u of the largest value, each of up to 40
    noise = 40 * u
    k = Ta.shape[1]
    # at most eps / 2 is out of the expansion's reach: sqrt(1 + 1/4) < 1.2
    assert k >= min(56, np.sum(s > 1.2 * eps * s[0] + noise * s[0])), (k, s[:k + 3])
    assert k <= np.sum(s > 0.9 * eps * s[0] - noise * s[0])
    left = s[k] if k < q else 0.0
    assert np.linalg.norm(C - Ta @ Tb.T, 2) <= 1.2 * left + (noise + (0.5 * eps if k < q else 0)) * s[0]


@pytest.mark.parametrize("prec,eps", [(32, 1e-6), (64, 1e-6), (64, 1e-10)])
def test_svd_keeps_a_value_spread_over_many_small_columns(lib, prec, eps):
    # every column but the first is a fifth of eps; 100 of them aligned make a singular value of 2 eps
    C = np.zeros((112, 112), complex)
    C[0, 0] = 1
    C[1, 1:101] = 0.2 * eps
    Ta, Tb, C = _svd(lib, prec, C, eps)
    assert Ta.shape[1] == 2
    assert np.linalg.norm(C - Ta @ Tb.T, 2) < 0.1 * eps


# cosines between the columns of T_b: the rotations' tolerance (4e-7, 1e-15), twice, and the rounding
# of the sweeps' rotations, a few u each of at most 20 sweeps
@pytest.mark.parametrize("prec,spread", [(32, 1e-4), (32, 1e-2), (32, 0.0), (64, 1e-8), (64, 1e-4), (64, 0.0)])
def test_svd_columns_of_a_cluster_are_orthogonal(lib, prec, spread):
    _, u = _types(prec)
    rng = np.random.default_rng(7)
    q, m = 96, 40
    s = np.concatenate([1 + spread * rng.standard_normal(m), 1e-2 * (1 + spread * rng.standard_normal(m // 2))])
    k = len(s)
    C = (_unitary(rng, q, k) * s) @ _unitary(rng, q, k).conj().T
    Ta, Tb, C = _svd(lib, prec, C, 1e-4, r_max=56)
    assert Ta.shape[1] == 56
    P = Tb / np.linalg.norm(Tb, axis=0)
    G = np.abs(P.conj().T @ P - np.eye(56))
    tol = 2 * (4e-7 if prec == 32 else 1e-15) + 60 * u
    assert G.max() < tol, (G.max(), tol)


def _qr(lib, prec, F, qsh):
    ct, _ = _types(prec)
    s, w = F.shape
    Fq = np.asfortranarray(F.astype(ct))
    Rm, qc = np.zeros((w, w), ct), ctypes.c_int(-1)
    fn = lib.qr_f32 if prec == 32 else lib.qr_f64
    F0 = np.array(Fq, dtype=complex)
    rc = fn(s, w, int(qsh), Fq.ctypes.data_as(ctypes.c_void_p), Rm.ctypes.data_as(ctypes.c_void_p), ctypes.byref(qc))
    assert rc == 0, rc
    return F0, Fq[:, :qc.value].astype(complex), Rm[:qc.value].astype(complex)


# remainders of the columns down to near the drop threshold (2e-6, 1e-13), and below it
@pytest.mark.parametrize("prec,least", [(32, 1e-1), (32, 5e-6), (32, 1e-9), (64, 1e-1), (64, 5e-13), (64, 1e-18)])
@pytest.mark.parametrize("s,w,qsh", [(9, 3, True), (130, 57, True), (256, 98, True), (130, 57, False), (512, 49, False)])
def test_qr_is_orthogonal_also_for_columns_with_small_remainders(lib, prec, least, s, w, qsh):
    _, u = _types(prec)
    if qsh and s * w * (8 if prec == 32 else 16) > 220 * 1024:
        qsh = False
    rng = np.random.default_rng(s + w)
    B = _unitary(rng, s, w)
    F = np.empty((s, w), complex)
    for j in range(w):
        v = B[:, :j] @ (rng.standard_normal(j) + 1j * rng.standard_normal(j)) if j else B[:, 0]
        F[:, j] = (v / np.linalg.norm(v) + np.exp(rng.uniform(np.log(least), 0)) * B[:, j]) * np.exp(rng.uniform(-3, 3))
    F, Q, R = _qr(lib, prec, F, qsh)
    # a column keeps at least half of itself in its last pass: 2 u for each rounding, a few of them,
    # from up to w updates added at random, and as much again a few times over from the columns before
    tol = 2 * u * 3 * np.sqrt(w) * 5
    assert np.abs(Q.conj().T @ Q - np.eye(Q.shape[1])).max() < tol
    # rounding of w updates, and the dropped remainders
    drop = 4e-6 if prec == 32 else 2e-13
    err = np.linalg.norm(F - Q @ R, axis=0) / np.linalg.norm(F, axis=0)
    assert err.max() < 4 * np.sqrt(w) * u + (drop if Q.shape[1] < w else 0)
    if least > drop:
        assert Q.shape[1] == w


@pytest.mark.parametrize("m,size", [(97, 1.5e-7), (97, 0.5e-7), (128, 2.2e-7)])
def test_svd_tells_noise_from_a_value_spread_over_columns(lib, m, size):
    # unrelated columns, whose squares sum to about (eps / 2)^2 and more while none of their singular values
    # (about twice a column's norm) reaches eps; and with them one value of 1.3 eps spread over all columns
    eps = 1e-6
    rng = np.random.default_rng(m)
    N = rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))
    N *= size / np.sqrt(2 * m)
    a = rng.standard_normal(m) + 1j * rng.standard_normal(m)
    for spread in (0.0, 1.3e-6):
        C = np.zeros((m, m), complex)
        C[:, 0] = a / np.linalg.norm(a)
        b = np.exp(2j * np.pi * rng.uniform(size=m)) / np.sqrt(m)
        b[0] = 0
        v = _unitary(rng, m, 2)[:, 0]
        C[:, 1:] += (N + spread * np.outer(v, b))[:, 1:]
        Ta, Tb, Cr = _svd(lib, 32, C, eps)
        s = np.linalg.svd(Cr, compute_uv=False)
        assert Ta.shape[1] == np.sum(s > eps * s[0]) == (2 if spread else 1), (s[:4], Ta.shape[1])
        # what is left: at most the largest value not kept and half of eps
        k = Ta.shape[1]
        assert np.linalg.norm(Cr - Ta @ Tb.T, 2) < 1.2 * s[k] + 0.5 * eps
