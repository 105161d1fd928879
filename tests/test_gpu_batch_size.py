"""A request's result does not depend on how many others are in its batch (GPU).

Up to eight streams ``vqe_eval_batch`` feeds gate by gate, beyond that it gives
them whole circuits as runs of gates.  The number of CTAs that a theta gets, the order of
its column pairs and the order of every sum follow from its sizes alone, so
both forms give the same bits.  The cases take a circuit through the sizes on
both sides of each change: one CTA up to 48 columns, clusters of 4 and of 8,
and rows past a tile of the product.
"""

import numpy as np
import pytest

from paper_2303_03681_gb300.inputs import MASTER_SEED, hf_bits, jw_molecular_hamiltonian, make_rng, random_integrals
from paper_2303_03681_gb300.inputs.circuits import CircuitTemplate, brickwork_circuit

pytestmark = pytest.mark.gpu


# qubits, layers, chi_max, precision, svd_fp64, CTAs of the widest theta
CASES = [
    (8, 6, 16, "fp64", 1, 1),     # 32 columns
    (10, 7, 24, "fp64", 1, 1),    # 48 columns
    (10, 7, 28, "fp64", 1, 4),    # 56 columns: would fit one CTA's shared memory
    (10, 7, 28, "fp64", 2, 4),
    (12, 8, 42, "fp64", 1, 4),    # 84 columns
    (12, 8, 64, "fp64", 1, 4),    # 128 columns, two tiles of product rows
    (14, 9, 120, "fp64", 1, 4),   # 64 x 240 and 128 x 128
    (16, 9, 120, "fp64", 1, 8),   # 240 x 240
    (12, 8, 64, "fp32", 1, 4),
]


@pytest.mark.parametrize("n,layers,chi,precision,svd_fp64,ctas", CASES)
def test_batches_of_nine_and_one_give_the_same_bits(n, layers, chi, precision, svd_fp64, ctas):
    from paper_2303_03681_gb300 import mps

    rng = make_rng(MASTER_SEED + 1500 + 10 * n + chi)
    h, g = random_integrals(n // 2, rng)
    tmpl = CircuitTemplate.from_gates(brickwork_circuit(n, layers, rng))
    bits = hf_bits(n, n // 2)
    ctxs = [mps.Context(0) for _ in range(9)]
    circ = mps.Circuit(ctxs[0], tmpl)
    ham = mps.Hamiltonian(ctxs[0], jw_molecular_hamiltonian(h, g))
    states = [mps.State(c, n, bits, chi_max=chi, precision=precision, svd_fp64=svd_fp64, trunc_rel=1e-6)
              for c in ctxs]
    reqs = [(s, circ, ham, np.zeros(0), bits) for s in states]
    for c in ctxs:
        c.profile_read(reset=True)
    energies, status = mps.vqe_eval_batch(reqs)
    assert not np.any(status)
    # a run is one launch of one CTA, one of 4 and one of 8, as far as its widest theta asks for
    launches = ctxs[8].profile_read(reset=True)["svd"][0]
    assert launches == {1: 1, 4: 2, 8: 3}[ctas]
    dims, (B, lam) = states[8].bond_dims(), states[8].export()
    assert dims.max() == chi  # the widest theta was met
    alone, st = mps.vqe_eval_batch(reqs[8:])
    assert st[0] == 0 and alone[0] == energies[8]
    B1, lam1 = states[8].export()
    for x, y in zip(B + lam, B1 + lam1):
        assert np.array_equal(x, y)
