"""A bounded wait that ran out on the device reaches the caller as MPS_ETIMEOUT.

The GPU tests set the flag in a state's report as the kernels do (no wait has
to run out) and then make the calls a user makes.  The status of a whole
report, which mps_truncated_svd returns too, is checked without a GPU.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_03681_gb300 import build as _build
from paper_2303_03681_gb300.inputs import (MASTER_SEED, brickwork_circuit, hf_bits, jw_molecular_hamiltonian, make_rng,
                                           random_integrals, uccsd_template)

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def flags(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("flags") / "report_flags.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-I", _build.CSRC,
                    os.path.join(HERE, "native", "report_flags.cu"), _build.build(), "-o", lib,
                    "-Xlinker", "-rpath," + os.path.dirname(_build.LIB)], check=True)
    lib = ctypes.CDLL(lib)
    lib.set_timeout_flag.argtypes = [ctypes.c_void_p]
    return lib


def test_status_of_a_report(flags):
    from paper_2303_03681_gb300 import mps

    assert flags.status_of(0, 0) == mps.MPS_OK
    assert flags.status_of(0, 2) == mps.MPS_ENOTCONV
    assert flags.status_of(1, 0) == flags.status_of(1, 2) == mps.MPS_ETIMEOUT


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32", "tf32x3"])
def test_every_call_reports_the_timeout(flags, precision):
    from paper_2303_03681_gb300 import mps

    n = 6
    rng = make_rng(MASTER_SEED + 1400)
    h, g = random_integrals(n // 2, rng)
    ctx = mps.Context(0)
    bits = hf_bits(n, 2)
    tmpl = uccsd_template(n, 2)
    ham = mps.Hamiltonian(ctx, jw_molecular_hamiltonian(h, g))
    circ = mps.Circuit(ctx, tmpl)
    gates = brickwork_circuit(n, 2, rng)
    st = mps.State(ctx, n, bits, chi_max=8, precision=precision, trunc_rel=1e-5)
    st.apply_gates(gates)
    before = st.energy(ham)
    ctx.synchronize()
    assert flags.set_timeout_flag(st.handle) == 0
    for call in (lambda: st.energy(ham), lambda: st.expectations(ham), lambda: st.apply_gates(gates)):
        with pytest.raises(mps.MpsError) as err:
            call()
        assert err.value.status == mps.MPS_ETIMEOUT
    with pytest.raises(mps.MpsError) as err:  # the gates may rest on an unfinished result
        st.apply_gates(gates)
    assert err.value.status == mps.MPS_ESTATE
    # a reset clears it
    e, status = mps.vqe_eval(ctx, [(st, circ, ham, np.zeros(tmpl.n_params), bits)])
    assert status[0] == 0 and np.isfinite(e[0])
    st.reset(bits)
    st.apply_gates(gates)
    assert st.energy(ham) == before
