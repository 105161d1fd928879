"""String values of complex128 states are FP64 sums (GPU).

A thread of the 128 adds its products one by one and the partial sums meet in
seven additions, so a value is off by at most (p + 7 + 4) u times the sum of
the absolute values: p products a thread (4 per entry of a leaf, 2 of a
string across the middle), 4 for the leaf's weights, u = 2^-53.  The reference
multiplies and sums exactly.  The entries have all 53 bits: 49 of them, as
double-float holds, would be off by more wherever few products are summed.
"""

import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2303_03681_gb300 import build as _build
from paper_2303_03681_gb300.inputs import MASTER_SEED, make_rng

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
PAULI = [np.eye(2), np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.diag([1, -1])]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    path = str(tmp_path_factory.mktemp("strings") / "strings.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-I", _build.CSRC,
                    os.path.join(HERE, "native", "strings.cu"), "-o", path], check=True)
    return ctypes.CDLL(path)


def _ptr(a):
    return ctypes.c_void_p(None if a is None else a.ctypes.data)


def _entries(rng, *shape):
    """Doubles with all 53 bits in use."""
    return rng.uniform(-1, 1, shape) + 1j * rng.uniform(-1, 1, shape)


def _exact(terms):
    """Sum of products of doubles, exactly, and of their absolute values."""
    exact = [math.prod(map(Fraction, t)) for t in terms]
    return sum(exact), float(sum(map(abs, exact)))


@pytest.mark.parametrize("chi_l,chi_r", [(1, 1), (1, 2), (3, 5), (16, 8), (11, 12)])
@pytest.mark.parametrize("op", range(4))
@pytest.mark.parametrize("weighted", [False, True])
def test_leaf(lib, chi_l, chi_r, op, weighted):
    rng = make_rng(MASTER_SEED + 1800 + chi_l + 20 * op)
    B, M = _entries(rng, chi_l, 2, chi_r), _entries(rng, chi_l, 2, chi_r)
    w = rng.uniform(0, 1, chi_r) if weighted else None
    out = np.zeros(1)
    assert lib.leaf_c128(chi_l, chi_r, op, _ptr(B), _ptr(M), _ptr(w), _ptr(out)) == 0
    terms = []
    for i in range(2):
        j = int(np.argmax(np.abs(PAULI[op][i])))
        y = PAULI[op][i, j] * M[:, j, :]
        for a in range(chi_l):
            for b in range(chi_r):
                ww = (w[b], w[b]) if weighted else ()
                terms += [(*ww, B[a, i, b].real, y[a, b].real), (*ww, B[a, i, b].imag, y[a, b].imag)]
    value, size = _exact(terms)
    p = 4 * -(-chi_l * chi_r // 128)
    assert abs(float(Fraction(float(out[0])) - value)) <= (p + 7 + 4) * 2.0 ** -53 * size


@pytest.mark.parametrize("chi", [1, 2, 7, 16, 17])
@pytest.mark.parametrize("n", [1, 8])
def test_across_the_middle(lib, chi, n):
    rng = make_rng(MASTER_SEED + 1900 + chi)

    def hermitian():
        x = _entries(rng, chi, chi)
        return np.triu(x, 1) + np.triu(x, 1).conj().T + np.diag(x.diagonal().real)

    L, R = hermitian(), np.array([hermitian() for _ in range(n)])
    out = np.zeros(n)
    assert lib.cross_c128(chi, n, _ptr(L), _ptr(R), _ptr(out)) == 0
    for k in range(n):
        terms = []
        for b in range(chi):
            for d in range(b, chi):
                f = 1.0 if b == d else 2.0
                terms += [(f * L[b, d].real, R[k, b, d].real), (-f * L[b, d].imag, R[k, b, d].imag)]
        value, size = _exact(terms)
        p = 2 * -(-chi * (chi + 1) // 2 // 128)
        assert abs(float(Fraction(float(out[k])) - value)) <= (p + 7 + 4) * 2.0 ** -53 * size
