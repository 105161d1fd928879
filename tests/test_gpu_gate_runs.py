"""Whole circuits as runs of gates (GPU): batches of more than eight streams.

``vqe_eval_batch`` issues the circuits of more than eight contexts as runs of
gates on one CTA, then on clusters of 4 and of 8.  Each case below is a batch
of nine whose circuit reaches another of these forms, with one-qubit gates in
between, against the same evaluations one at a time (gate by gate).

Tolerance: both forms sum the same products with the same error bound, in
another order.  A double-float sum of K <= 128 products is good to K 2^-47 of
the sum of their absolute values (1e-12), an FP32 one to K 2^-24 (8e-6), and
each gate adds its part to the state, whose strings have absolute value <= 1.
"""

import numpy as np
import pytest

from paper_2303_03681_gb300.inputs import MASTER_SEED, jw_molecular_hamiltonian, make_rng, random_integrals
from paper_2303_03681_gb300.inputs.circuits import CircuitTemplate, brickwork_circuit, uccsd_template

pytestmark = pytest.mark.gpu


# qubits, brickwork layers (0: UCCSD), chi_max, precision, svd_fp64; the widest theta is 2 chi
CASES = [
    (4, 0, 4, "fp64", 1),     # thetas of at most 8 columns: FP64 SVD, one CTA
    (8, 8, 16, "fp64", 1),    # 32 columns: double-float SVD, one CTA
    (8, 8, 16, "fp64", 2),    # the FP64 SVD of 32 columns
    (8, 8, 16, "fp32", 1),    # complex64 storage
    (10, 8, 32, "fp64", 1),   # 64 columns: clusters of 4
    (14, 10, 120, "fp64", 1),  # 240 columns: clusters of 8, and truncation
]


@pytest.mark.parametrize("n,layers,chi,precision,svd_fp64", CASES)
def test_runs_equal_gate_by_gate(n, layers, chi, precision, svd_fp64):
    from paper_2303_03681_gb300 import mps

    rng = make_rng(MASTER_SEED + 1200 + 10 * n + layers)
    h, g = random_integrals(n // 2, rng)
    ham = jw_molecular_hamiltonian(h, g)
    tmpl = uccsd_template(n, n // 2)
    if layers:
        gl = brickwork_circuit(n, layers, rng)
        gl.arity[5::7] = 1  # a unitary block of two: one-qubit gates in between
        gl.u[5::7] = 0
        gl.u[5::7, :2, :2] = np.linalg.qr(rng.normal(size=(len(gl.q[5::7]), 2, 2)) + 1j * rng.normal(size=(2, 2)))[0]
        tmpl = CircuitTemplate.from_gates(gl)
    bits = np.array([i < n // 2 for i in range(n)], np.uint8)
    thetas = [rng.uniform(-0.3, 0.3, tmpl.n_params) for _ in range(9)]
    ctxs = [mps.Context(0) for _ in thetas]
    circ, H = mps.Circuit(ctxs[0], tmpl), mps.Hamiltonian(ctxs[0], ham)
    states = [mps.State(c, n, bits, chi_max=chi, precision=precision, svd_fp64=svd_fp64,
                        trunc_rel=1e-10 if precision == "fp64" else 1e-5) for c in ctxs]
    batch, status = mps.vqe_eval_batch([(s, circ, H, th, bits) for s, th in zip(states, thetas)])
    assert not np.any(status)
    runs = [(s.bond_dims(), s.report()) for s in states]
    tol = tmpl.n_gates * (1e-12 if precision == "fp64" else 8e-6) * np.abs(ham.coeffs).sum()
    for i in (0, 8):
        alone, st = mps.vqe_eval(ctxs[i], [(states[i], circ, H, thetas[i], bits)])
        assert st[0] == 0 and abs(alone[0] - batch[i]) <= tol
        dims, rep = runs[i]
        assert np.array_equal(dims, states[i].bond_dims())
        one = states[i].report()
        for key in ("max_chi", "two_qubit_gates"):
            assert rep[key] == one[key]
        assert abs(rep["discarded_weight"] - one["discarded_weight"]) <= tmpl.n_gates * (
            1e-12 if precision == "fp64" else 8e-6)
