"""Thetas that need the co-resident grid, replayed as a graph and on several streams (GPU).

18 qubits at chi_max = 176: the middle theta is 352 x 352, past a cluster's
shared memory.  A graph replay, launches from the host and concurrent
evaluations run the same kernels in the same order, so the bits agree.
"""

import numpy as np
import pytest

from paper_2303_03681_gb300.inputs import MASTER_SEED, hf_bits, jw_molecular_hamiltonian, make_rng, random_integrals
from paper_2303_03681_gb300.inputs.circuits import CircuitTemplate, brickwork_circuit

pytestmark = pytest.mark.gpu


def test_grid_svds_in_a_graph_and_on_streams():
    from paper_2303_03681_gb300 import mps

    n = 18
    rng = make_rng(MASTER_SEED + 2100)
    h, g = random_integrals(n // 2, rng)
    ham = jw_molecular_hamiltonian(h, g)
    tmpl = CircuitTemplate.from_gates(brickwork_circuit(n, 9, rng))
    bits = hf_bits(n, n // 2)
    ctxs = [mps.Context(0) for _ in range(3)]
    circ, H = mps.Circuit(ctxs[0], tmpl), mps.Hamiltonian(ctxs[0], ham)
    states = [mps.State(c, n, bits, chi_max=176, precision="fp64", trunc_rel=1e-8) for c in ctxs]
    reqs = [(s, circ, H, np.zeros(0), bits) for s in states]
    energies = []
    for graphs in (False, True, True):
        ctxs[0].set_graphs(graphs)
        e, status = mps.vqe_eval(ctxs[0], reqs[:1])
        assert status[0] == 0
        energies.append(e[0])
    dims = states[0].bond_dims()
    assert dims[8] == dims[10] == 176
    batch, status = mps.vqe_eval_batch(reqs)
    assert not np.any(status)
    assert len(set(energies) | set(batch.tolist())) == 1
