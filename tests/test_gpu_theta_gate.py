"""The gate's product in the theta of complex128 states is an FP64 one (GPU).

The site tensors hold small powers of two, so the contraction over the middle
bond is exact and what is left are the 4 complex products of an entry with the
gate: 8 real products each for re and im, and an error of at most 8 u times the
sum of their absolute values (u = 2^-53).  Real gates take a path of their own.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_03681_gb300 import build as _build
from paper_2303_03681_gb300.inputs import MASTER_SEED, haar_su4, make_rng

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def theta(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("theta") / "theta.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-I", _build.CSRC,
                    os.path.join(HERE, "native", "theta.cu"), "-o", lib], check=True)
    fn = ctypes.CDLL(lib).theta_c128
    fn.argtypes = [ctypes.c_int] * 3 + [ctypes.c_void_p] * 4

    def call(bl, br, gate):
        out = np.zeros((2 * bl.shape[0], 2 * br.shape[2]), np.complex128)
        assert fn(bl.shape[0], bl.shape[2], br.shape[2], bl.ctypes.data, br.ctypes.data, gate.ctypes.data,
                  out.ctypes.data) == 0
        return out

    return call


@pytest.mark.parametrize("chi_l,chi_m,chi_r", [(1, 1, 1), (2, 1, 2), (15, 3, 17), (16, 16, 16), (33, 18, 5)])
@pytest.mark.parametrize("real", [False, True])
def test_gate_product(theta, chi_l, chi_m, chi_r, real):
    rng = make_rng(MASTER_SEED + 1700 + chi_l)
    bl, br = (2.0 ** rng.integers(-2, 3, s) * rng.choice([1, -1, 1j, -1j], s)
              for s in ((chi_l, 2, chi_m), (chi_m, 2, chi_r)))
    gate = haar_su4(rng)
    if real:
        gate = np.linalg.qr(gate.real)[0] + 0j
    gate = np.ascontiguousarray(gate, np.complex128)
    out = theta(np.ascontiguousarray(bl), np.ascontiguousarray(br), gate).reshape(chi_l, 2, 2, chi_r)
    t = np.einsum("lim,mjr->lijr", bl, br)  # exact
    # the reference in extended precision where numpy has it, else within another 8 u
    g = gate.reshape(2, 2, 2, 2).astype(np.clongdouble)
    ref = np.einsum("ijkl,aklb->aijb", g, t.astype(np.clongdouble))
    size = np.einsum("ijkl,aklb->aijb", np.abs(gate.real.reshape(2, 2, 2, 2)) + np.abs(gate.imag.reshape(2, 2, 2, 2)),
                     np.abs(t.real) + np.abs(t.imag))
    assert np.all(np.abs(out - ref) <= 16 * 2.0 ** -53 * size)
