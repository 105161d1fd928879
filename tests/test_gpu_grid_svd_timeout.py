"""The co-resident-grid SVD when a wait at its barrier is given up (GPU).

The kernel is launched with the barrier's abort flag already set, as a CTA
whose wait ran out leaves it.  Every CTA then has to leave at its first barrier
that the others have not reached, without reading what they published: the
launch ends at once, reports the timeout and leaves the bond dimension alone.
No wait in it is longer than the barrier's own limit of about two seconds.
"""

import ctypes
import os
import subprocess
import time

import numpy as np
import pytest

from paper_2303_03681_gb300 import build as _build
from paper_2303_03681_gb300.inputs import MASTER_SEED, make_rng

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def grid_svd(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("grid_svd") / "grid_svd.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-I", _build.CSRC,
                    os.path.join(HERE, "native", "grid_svd.cu"), "-o", lib], check=True)
    fn = ctypes.CDLL(lib).grid_svd
    fn.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def call(n, C, abort):
        out = np.zeros(2, np.int32)
        assert fn(n, np.ascontiguousarray(C).ctypes.data, abort, out.ctypes.data) == 0
        return int(out[0]), int(out[1])

    return call


@pytest.mark.parametrize("rank", [340, 3])  # 3: the residuals below the noise floor are scaled up, step after step
def test_given_up_wait_ends_the_kernel(grid_svd, rank):
    n = 340
    rng = make_rng(MASTER_SEED + 1300 + rank)
    C = (rng.normal(size=(n, rank)) + 1j * rng.normal(size=(n, rank))) @ (
        rng.normal(size=(rank, n)) + 1j * rng.normal(size=(rank, n)))
    error, k = grid_svd(n, C, 0)
    assert error == 0 and k >= rank
    t0 = time.perf_counter()
    error, k = grid_svd(n, C, 1)
    assert error == 1 and k == -1
    assert time.perf_counter() - t0 < 2.0
