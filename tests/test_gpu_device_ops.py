"""The step kernels' own quotients, reciprocals and roots against CUDA's.

FP64: before its one rounding a value is good to 2^-85 of itself, so it is the
IEEE operation's or, where the exact value is that close to the middle of two
numbers, the other of the two.  Of n operands without a pattern 2 n 2^-85 /
2^-53 are so close, n / 2^31.

FP32: for normal operands the bare instructions are the full functions."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1204_4098_gb300 import build

pytestmark = pytest.mark.gpu
TESTS = os.path.dirname(os.path.abspath(__file__))
N = 1 << 22


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("ops") / "ops.so")
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v")]
    subprocess.run([build._nvcc(), *build.ARCH, *flags, "-shared", "-o", so,
                    os.path.join(TESTS, "device_ops.cu"), "-lcudart"],
                   check=True, capture_output=True, text=True)
    return ctypes.CDLL(so)


def fp64(ops, a, b):
    a, b = (np.ascontiguousarray(v, dtype=np.float64) for v in (a, b))
    out = (ctypes.c_ulonglong * 6)()
    P = ctypes.c_void_p
    assert ops.fp64_ops(P(a.ctypes.data), P(b.ctypes.data), ctypes.c_size_t(len(a)), out) == 0
    return list(out[:3]), list(out[3:])


def test_fp64_of_random_operands_is_ieee(ops):
    rng = np.random.default_rng(1)
    a, b = (rng.uniform(1.0, 2.0, N) * 2.0 ** rng.integers(-99, 99, N) for _ in range(2))
    assert fp64(ops, a, b) == ([0, 0, 0], [0, 0, 0])


def near_ones(rng, lead):
    """Mantissas of `lead` ones, then random bits: their reciprocals lie near
    the middle of two numbers."""
    m = rng.integers(0, 1 << (52 - lead), N, dtype=np.uint64)
    bits = np.uint64(((1 << lead) - 1) << (52 - lead)) | m | np.uint64(1023 << 52)
    return bits.view(np.float64)


@pytest.mark.parametrize("lead", [8, 20, 26, 28, 30, 40])
def test_fp64_near_the_middle_of_two_numbers_is_one_of_them(ops, lead):
    rng = np.random.default_rng(lead)
    a, b = near_ones(rng, lead), near_ones(rng, lead)
    scale = 2.0 ** rng.integers(-90, 90, N)
    for x, y in ((a, b), (a * scale, b), (a, b * scale), (1.0 / b, b)):
        worst, differ = fp64(ops, x, y)
        print(lead, worst, differ)
        assert max(worst) <= 1


def pairs(x, y):
    return (np.concatenate([v, -v]) for v in (g.ravel() for g in np.meshgrid(x, y)))


POWERS = [2.0 ** k for k in range(-1074, 1024)]
LIMITS = [v * 2.0 ** e for e in (-100, 100) for v in (1.0, 1.0 + 2.0 ** -52, 1.5)]
ODD = [0.0, np.inf, np.nan, 5e-324, 2.2e-308, 1.7e308]


def test_fp64_at_and_beyond_the_limits_is_ieee(ops):
    # beyond 2^-100 and 2^100 (by an ulp, and mantissas of all ones with it) the
    # IEEE operations run
    beyond = [(1.0 - 2.0 ** -53) * 2.0 ** -100, (2.0 - 2.0 ** -52) * 2.0 ** 100]
    x = np.array(POWERS + LIMITS + ODD)
    for a, b in (pairs(x, x), pairs(x, beyond), pairs(beyond, x)):
        assert fp64(ops, a, b) == ([0, 0, 0], [0, 0, 0])


def test_fp64_mantissas_of_all_ones_within_the_limits(ops):
    # 1 / (2 - 2^-52) lies 2^-107 of itself from the middle of two numbers
    ones = [(2.0 - 2.0 ** -52) * 2.0 ** e for e in (-100, -1, 0, 99)]
    x = np.array(POWERS + LIMITS)
    for a, b in (pairs(x, ones), pairs(ones, x), pairs(ones, ones)):
        assert max(fp64(ops, a, b)[0]) <= 1


def test_fp32_bare_forms_are_the_full_ones_for_normal_operands(ops):
    out = (ctypes.c_ulonglong * 3)()
    first, last = (127 - 110) << 23, (127 + 110) << 23  # every one from 2^-110 to 2^110
    assert ops.fp32_ops(ctypes.c_uint(first), ctypes.c_uint(last), out) == 0
    assert list(out) == [0, 0, 0]
