"""The division in the Rayleigh-Ritz solve's triangular inverse is a product
with the reciprocal and two corrections; it has to be the division itself,
rounded to nearest, for every operand it meets."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1907_07410_gb300", "csrc")


@pytest.fixture(scope="module")
def quotients(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotient")
    src, lib = str(d / "q.cpp"), str(d / "q.so")
    with open(src, "w") as f:
        f.write('#include "quotient.h"\n'
                'extern "C" void quotients(long n, const float *a, const float '
                '*b, float *q) {\n'
                '  for (long i = 0; i < n; ++i)\n'
                '    q[i] = bsvd::quotient(a[i], b[i], 1.0f / b[i]);\n}\n')
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off",
                           "-shared", "-fPIC", "-I", CSRC, "-o", lib, src])
    f = ctypes.CDLL(lib).quotients
    f.argtypes = [ctypes.c_long] + [ctypes.c_void_p] * 3

    def run(a, b):
        a, b = (np.ascontiguousarray(v, np.float32) for v in (a, b))
        q = np.empty(a.size, np.float32)
        f(a.size, a.ctypes.data, b.ctypes.data, q.ctypes.data)
        return q
    return run


def floats(rng, n, lo, hi):
    """Any mantissa, exponents lo .. hi - 1."""
    m = rng.integers(0, 1 << 23, n)
    at = rng.integers(0, 4, n) == 0              # mantissas near the ends
    m[at] = rng.choice([0, 1, 2, 3, (1 << 23) - 1, (1 << 23) - 2,
                        (1 << 22) - 1, 1 << 22, (1 << 22) + 1], at.sum())
    return ((1.0 + m / 2.0 ** 23) * 2.0 ** rng.integers(lo, hi, n)
            ).astype(np.float32)


# the divisor is the root of a pivot of a matrix with unit diagonal, between
# its drop limit and 1 or a little above; the dividend an entry of an inverse
@pytest.mark.parametrize("seed", range(4))
def test_rounds_as_the_division(quotients, seed):
    rng = np.random.default_rng(seed)
    n = 1 << 20
    b = floats(rng, n, -24, 2)
    a = floats(rng, n, -60, 40) * rng.choice([-1, 1], n).astype(np.float32)
    assert np.array_equal(quotients(a, b), a / b)


def test_exact_and_zero_quotients(quotients):
    rng = np.random.default_rng(9)
    b = floats(rng, 1 << 18, -24, 2)
    k = rng.integers(0, 64, b.size).astype(np.float32)
    a = (k * b).astype(np.float32)                # exact for small k, or near
    assert np.array_equal(quotients(a, b), a / b)
    assert not quotients(np.zeros(b.size), b).any()


def test_every_mantissa_against_a_few(quotients):
    m = (1.0 + np.arange(1 << 23) / 2.0 ** 23).astype(np.float32)
    for b in (1.0, 1.0 + 2.0 ** -23, 1.5, 2.0 - 2.0 ** -23, 4.0 / 3.0):
        b = np.full(m.size, b, np.float32)
        assert np.array_equal(quotients(m, b), m / b)
        assert np.array_equal(quotients(b, m), b / m)
