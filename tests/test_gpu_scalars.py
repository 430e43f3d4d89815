"""The integer conversions between double and float and the Newton reciprocals of csrc/common.cuh, through
tests/kernels/common_entries.cu."""
import ctypes

import numpy as np
import pytest

from tests.kernels import kernel_library

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return kernel_library(tmp_path_factory, "common")


def _map(fn, x, out, op):
    assert fn(len(x), x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), op) == 0
    return out


def test_double_to_float_has_the_compiler_s_bits(lib):
    rng = np.random.default_rng(1)
    any_bits = rng.integers(0, 2 ** 64, 1 << 22, dtype=np.uint64).view(np.float64)
    e = rng.integers(1023 - 155, 1023 + 130, 1 << 22).astype(np.uint64) << np.uint64(52)      # FP32's range and its edges
    near = ((rng.integers(0, 2 ** 52, 1 << 22, dtype=np.uint64) | e) | (rng.integers(0, 2, 1 << 22).astype(np.uint64) << np.uint64(63))).view(np.float64)
    # ties and their neighbours: 29 bits are dropped
    ties = (near.view(np.uint64) & ~np.uint64(0x1fffffff)) | rng.choice(np.array([0, 1, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff], np.uint64), 1 << 22)
    odd = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -126, 2.0 ** -149, 2.0 ** -150, 2.0 ** -151, 1.5 * 2.0 ** -150,
                    3.4028234663852886e38, 3.4028235677973366e38, 3.4028235677973362e38, 5e-324, -5e-324, 1.7976931348623157e308])
    x = np.concatenate([any_bits, near, ties.view(np.float64), odd, -odd])
    a, b = (_map(lib.narrow, x, np.zeros(len(x), np.float32), op) for op in (0, 1))
    nan = np.isnan(x)
    assert np.array_equal(a[~nan].view(np.uint32), b[~nan].view(np.uint32)) and np.isnan(a[nan]).all()


def test_float_to_double_has_the_compiler_s_bits(lib):
    rng = np.random.default_rng(2)
    bits = np.concatenate([rng.integers(0, 2 ** 32, 1 << 22, dtype=np.uint64).astype(np.uint32),
                           np.arange(1 << 16, dtype=np.uint32), (np.arange(1 << 16, dtype=np.uint32) + np.uint32(0x007f8000)),
                           (np.arange(1 << 16, dtype=np.uint32) + np.uint32(0x7f7f8000))])
    x = np.concatenate([bits, bits | np.uint32(0x80000000)]).view(np.float32)
    a, b = (_map(lib.widen, x, np.zeros(len(x)), op) for op in (0, 1))
    nan = np.isnan(x)
    assert np.array_equal(a[~nan].view(np.uint64), b[~nan].view(np.uint64)) and np.isnan(a[nan]).all()


# two Newton steps from FP32: 2^-22 squares to 2^-43 and 2^-86, and each of the last step's two or three
# operations rounds once: 4 * 2^-53
@pytest.mark.parametrize("op,lo,hi", [(0, -120, 120), (1, -120, 120), (2, -1021, 1024), (3, -1021, 1024)])
def test_newton_reciprocals(lib, op, lo, hi):
    rng = np.random.default_rng(3)
    x = np.ldexp(rng.uniform(0.5, 1.0, 1 << 20), rng.integers(lo, hi + 1, 1 << 20))
    x = np.concatenate([x, np.ldexp(1.0, np.arange(lo, hi)), np.ldexp(1.0 - 2.0 ** -53, np.arange(lo + 1, hi + 1))])
    y = _map(lib.newton, x, np.zeros(len(x)), op).astype(np.longdouble)
    xl = x.astype(np.longdouble)
    one = np.longdouble(1)
    ref = one / xl if op in (0, 2) else one / np.sqrt(xl)
    # (1 / x below 2^-1022 is rounded to the subnormals' spacing)
    err = np.abs(y - ref) / np.maximum(ref, np.longdouble(2.0) ** -1022)
    assert err.max() < 4 * 2.0 ** -53, float(err.max())
