"""The fixed-point roots of unity of the integer transform passes (host code)."""

import ctypes
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_1206_0675_gb300 import build

EXTENTS = sorted(2 ** a * 3 ** b for a in range(8) for b in range(5) if 2 <= 2 ** a * 3 ** b <= 128)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    (d / "roots.cpp").write_text('#include "lgf_roots.h"\nextern "C" int roots(int N, int* hl) '
                                 '{ return lgf::fixed_roots(N, hl); }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(d / "libroots.so"),
                    str(d / "roots.cpp")], check=True)
    return ctypes.CDLL(str(d / "libroots.so"))


def cos_sin(m, N):
    """cos and sin of 2 pi m / N to 40 digits, by their power series."""
    getcontext().prec = 60
    pi = Decimal("3.14159265358979323846264338327950288419716939937510582097494")
    t = 2 * pi * m / N
    c, s, term = Decimal(0), Decimal(0), Decimal(1)
    for n in range(0, 80):
        if n % 2 == 0:
            c += term if n % 4 == 0 else -term
        else:
            s += term if n % 4 == 1 else -term
        term = term * t / (n + 1)
    return c, s


@pytest.mark.parametrize("N", EXTENTS)
def test_fixed_roots(lib, N):
    """Each limb pair is the root rounded to 2^-60 (an eighth of a unit more where long double has 64 bits), and the
    angles evaluated are those of one octant, not all N."""
    hl = np.zeros((N, 2, 2), dtype=np.int32)
    n = lib.roots(N, ctypes.c_void_p(hl.ctypes.data))
    assert n <= (N // 8 + 1 if N % 8 == 0 else N // 2 + 1)
    assert np.all(np.abs(hl[..., 1]) <= 2 ** 29)
    for m in range(N):
        c, s = cos_sin(m, N)
        for k, want in enumerate((c, -s)):
            got = int(hl[m, k, 0]) * 2 ** 30 + int(hl[m, k, 1])
            assert abs(Decimal(got) - want * 2 ** 60) <= Decimal("0.625")
