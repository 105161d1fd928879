"""Expectation values through environments from both ends (GPU).

Prefixes of the strings are contracted from the left, suffixes from the right,
and they meet at the bond with the least work.  Each family of strings below
puts that bond elsewhere or leaves one side empty; every string is compared
with its own transfer-matrix chain on the exported state.

Tolerance: a level's sum of at most 2 chi products errs by 2 chi u of the sum
of their absolute values, environments have Frobenius norm up to sqrt(chi), and
there are n levels: 2 n chi^1.5 u with u = 2^-47 (double-float) or 2^-24.
"""

import numpy as np
import pytest

from gpu_helpers import to_oracle
from oracle import mps as om
from paper_2303_03681_gb300.inputs import MASTER_SEED, brickwork_circuit, make_rng
from paper_2303_03681_gb300.inputs.hamiltonian import PauliSum

pytestmark = pytest.mark.gpu


def _strings(family, n, rng):
    if family == "mixed":  # any support, all four operators inside, the identity, single sites
        ops = rng.integers(0, 4, (150, n))
        for row in ops:
            a, b = sorted(rng.integers(0, n + 1, 2))
            row[:a] = 0
            row[b:] = 0
        ops[:n] = np.diag(rng.integers(1, 4, n))
        ops[n] = 0
    else:
        ops = np.repeat(rng.integers(1, 4, (1, n)), 60, axis=0)
        free = slice(n - 3, n) if family == "tails" else slice(0, 3)  # all but these sites in common
        ops[:, free] = rng.integers(0, 4, (60, 3))
    if family == "left":
        ops[:, n // 2 - 1:] = 0
    return np.unique(ops, axis=0).astype(np.uint8)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("family", ["mixed", "heads", "tails", "left"])
@pytest.mark.parametrize("n,chi", [(2, 2), (9, 13), (10, 17)])
def test_every_string(n, chi, family, precision):
    from paper_2303_03681_gb300 import mps

    if n == 2 and family != "mixed":
        pytest.skip("two sites")
    rng = make_rng(MASTER_SEED + 1300 + n)
    ops = _strings(family, n, rng)
    ctx = mps.Context(0)
    st = mps.State(ctx, n, None, chi_max=chi, precision=precision)
    st.apply_gates(brickwork_circuit(n, 8, rng))
    vals = st.expectations(mps.Hamiltonian(ctx, PauliSum(n, ops, np.ones(len(ops)))))
    got = to_oracle(st)
    want = np.array([om.expect_pauli(got, row) for row in ops])
    u = 2.0 ** -47 if precision == "fp64" else 2.0 ** -24
    assert np.max(np.abs(vals - want)) <= 2 * n * chi ** 1.5 * u
