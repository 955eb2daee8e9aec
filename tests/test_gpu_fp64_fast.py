"""GPU tests of the short FP64 quotient, reciprocal and square root against CUDA's operators."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2505_20375_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
NAMES = ("divide", "reciprocal", "root", "reciprocal_near")


@pytest.fixture(scope="module")
def apply(fci_lib, tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("probe") / "probe.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "static",
                    "-I", build.CSRC, "-o", lib, os.path.join(HERE, "fp64_fast_probe.cu")], check=True)
    fn = ctypes.CDLL(lib).fp64_fast_apply
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p, ctypes.c_void_p]

    def run(a, b):
        a, b = (torch.from_numpy(np.ascontiguousarray(v, np.float64)).cuda() for v in (a, b))
        fast, op = (torch.empty(len(a), 4, dtype=torch.float64, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        assert fn(a.data_ptr(), b.data_ptr(), len(a), fast.data_ptr(), op.data_ptr()) == 0
        return fast.cpu().numpy(), op.cpu().numpy()

    return run


def _equal(fast, op):
    both_nan = np.isnan(fast) & np.isnan(op)
    return both_nan | (fast.view(np.int64) == op.view(np.int64))


def test_random_operands_give_the_bits_of_the_operators(apply):
    """Mantissas over all bits, exponents over the range of the short forms and past it."""
    r = np.random.default_rng(5)
    for spread in (1, 40, 390, 1000):
        m = r.integers(0, 1 << 52, size=(2, 1 << 21), dtype=np.int64)
        e = r.integers(1023 - spread, 1023 + spread + 1, size=m.shape)
        sign = r.integers(0, 2, size=m.shape)
        a, b = (m | (e << 52) | (sign << 63)).view(np.float64)
        fast, op = apply(a, b)
        ok = _equal(fast, op)
        assert ok.all(), {n: int((~ok[:, i]).sum()) for i, n in enumerate(NAMES)}


def test_special_operands_give_the_bits_of_the_operators(apply):
    """Zeros, infinities, NaN, subnormals, the ends of the exponent range and of the range of the
    short forms, powers of two and squares (mantissas of ones only are in the next test)."""
    v = [0.0, np.inf, np.nan, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308, 1e-300, 1e300, 1.0, 2.0, 3.0, 0.1,
         1.0 + 2.0 ** -52, 4.0, 9.0, 1.5, 2.0 ** 399, 2.0 ** 400, 2.0 ** -399, 2.0 ** -400, 2.0 ** 401, 1e154]
    v = np.array(v + [-x for x in v])
    a, b = np.meshgrid(v, v)
    fast, op = apply(a.ravel(), b.ravel())
    assert _equal(fast, op).all()


def test_quotients_next_to_a_midpoint(apply):
    """Quotients as close to the midpoint of two neighbours as they get (n / d = m / 2^53 (1 +- tiny)
    with odd m), where the error of the last correction decides the rounding: with a reciprocal
    of 2^-45 there 44% of them miss."""
    r = np.random.default_rng(6)
    num, den = [], []
    while len(num) < 20000:
        d = int(r.integers(1 << 52, 1 << 53)) | 1
        for sign in (1, -1):
            m = (sign * pow(d, -1, 1 << 53)) % (1 << 53) + (1 << 53)
            n, rest = divmod(m * d - sign, 1 << 53)
            assert rest == 0
            if 1 << 52 <= n < 1 << 53:
                num.append(float(n))
                den.append(float(d))
    fast, op = apply(num, den)
    assert _equal(fast[:, 0], op[:, 0]).all()


def test_mantissas_of_ones_are_within_one_unit(apply):
    """The class that the reciprocal's last correction does not cover."""
    ones = np.array([2.0 ** k * (2.0 - 2.0 ** -52) for k in range(-50, 51)])
    fast, op = apply(np.concatenate([np.ones_like(ones), ones]), np.concatenate([ones, ones[::-1]]))
    assert np.abs(fast.view(np.int64) - op.view(np.int64)).max() <= 1
