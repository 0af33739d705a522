"""hr_math.cuh: reciprocal, square roots and conversions of the FP64 kernels.

In the range of the seeds (biased exponents 1 to 2044) the iteration leaves a
truncation of e^3 (1/x, e = 1 - x y) or 5 e^3/16 (roots, e = 1 - x y^2) beside
the rounding of the last operation.  The seeds y hold 20 bits, so that |e| is
about 2^-20 or 2^-19: 2^-60 and 2^-58.7 of the result, less than 0.01 and 0.02 of
its last place: at most 0.51 and 0.52 ulp, against extended precision.  Everywhere else (zero, subnormal,
infinite, NaN, negative under the root) the bits of the language's operation.
The conversions: the bits of the language's for every pattern, ties, carries
into the next binade, overflow and underflow of FP32 among them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1312_6127_gb300 import _build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
RCP, SQRT, RSQRT, SQRT_OF_PAIR, RSQRT_OF_PAIR, NARROW, WIDEN = range(7)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("math") / "math_probe.so")
    subprocess.check_call([_build.nvcc(), "-shared", "-I", _build.CSRC] + _build.ARCH + _build.FLAGS +
                          [os.path.join(HERE, "cuda", "math_probe.cu"), "-o", so])
    lib = ctypes.CDLL(so)

    def run(op, own, bits):
        src = torch.from_numpy(bits.view(np.int64)).cuda()
        dst = torch.empty_like(src)
        assert lib.math_probe(op, own, len(bits), ctypes.c_void_p(src.data_ptr()), ctypes.c_void_p(dst.data_ptr()),
                              ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        return dst.cpu().numpy().view(np.uint64)

    return run


def patterns():
    """Every sign and exponent with mantissas at and beside its ends, and random ones."""
    g = np.random.default_rng(7)
    e = np.arange(2048, dtype=np.uint64) << np.uint64(52)
    m = np.array([0, 1, 2, 3, 2 ** 51 - 1, 2 ** 51, 2 ** 51 + 1, 2 ** 52 - 2, 2 ** 52 - 1], dtype=np.uint64)
    ends = (e[:, None] | m[None, :]).ravel()
    return np.concatenate([ends, ends | np.uint64(1 << 63), g.integers(0, 2 ** 64, 1 << 20, dtype=np.uint64)])


@pytest.mark.parametrize("op", [RCP, SQRT, RSQRT, SQRT_OF_PAIR, RSQRT_OF_PAIR])
def test_reciprocal_and_roots(probe, op):
    bits = patterns()
    x = bits.view(np.float64)
    own = probe(op, 1, bits)
    exponent = (bits >> np.uint64(52)) & np.uint64(2047)
    seeded = (exponent >= 1) & (exponent <= 2044)
    if op != RCP:
        seeded &= bits >> np.uint64(63) == 0
    other = probe(op, 0, bits[~seeded])
    assert np.array_equal(own[~seeded], other)
    X = x[seeded].astype(np.longdouble)
    root = np.sqrt(X) if op != RCP else None
    exact = 1.0 / X if op == RCP else (root if op in (SQRT, SQRT_OF_PAIR) else 1.0 / root)
    ulp = np.ldexp(np.longdouble(1.0), np.frexp(exact)[1] - 53)
    err = np.abs(own[seeded].view(np.float64).astype(np.longdouble) - exact) / ulp
    print("op %d: %d arguments, largest error %.4f ulp" % (op, seeded.sum(), float(err.max())))
    assert err.max() <= (0.51 if op == RCP else 0.52)


def test_narrow(probe):
    g = np.random.default_rng(8)
    # around FP32's roundings: exact, one off, ties, for every exponent that FP32 reaches and its neighbours
    e = np.arange(1023 - 152, 1023 + 131, dtype=np.uint64) << np.uint64(52)
    top = np.concatenate([[0, 1, 2 ** 23 - 2, 2 ** 23 - 1], g.integers(0, 2 ** 23, 40)]).astype(np.uint64) << np.uint64(29)
    low = np.array([0, 1, 2 ** 28 - 1, 2 ** 28, 2 ** 28 + 1, 2 ** 29 - 1], dtype=np.uint64)
    b = (e[:, None, None] | top[None, :, None] | low[None, None, :]).ravel()
    bits = np.concatenate([patterns(), b, b | np.uint64(1 << 63)])
    assert np.array_equal(probe(NARROW, 1, bits), probe(NARROW, 0, bits))


def test_widen(probe):
    g = np.random.default_rng(9)
    e = np.arange(512, dtype=np.uint64) << np.uint64(23)
    m = np.concatenate([[0, 1, 2 ** 22 - 1, 2 ** 22, 2 ** 23 - 1], g.integers(0, 2 ** 23, 200)]).astype(np.uint64)
    bits = (e[:, None] | m[None, :]).ravel()
    assert np.array_equal(probe(WIDEN, 1, bits), probe(WIDEN, 0, bits))
