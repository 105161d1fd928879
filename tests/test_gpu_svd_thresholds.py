"""Truncation thresholds at the rounding level (GPU).

Diagonal thetas whose entries are powers of two: every step of the
factorisation is exact on them, so the kept count has to be the rule's, s_i >
trunc_rel s_1, even where the threshold lies below the arithmetic's noise
floor (8 u: 1.1e-13 in double-float, 8.9e-16 in FP64).
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _svd(A, trunc, mode):
    import torch

    from paper_2303_03681_gb300 import mps

    n = A.shape[0]
    ctx = mps.Context(0)
    d = torch.from_numpy(np.ascontiguousarray(A, dtype=np.complex128)).cuda()
    s = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    vh = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
    k, rep, rc = mps.truncated_svd(ctx, "fp64", n, n, d.data_ptr(), n, trunc, mode, s.data_ptr(), vh.data_ptr())
    assert rc == mps.MPS_OK
    return k, s.cpu().numpy()[:k], vh.cpu().numpy()[:k], rep


# mode, columns, small entries, threshold between them and the others
@pytest.mark.parametrize("mode,n,small,trunc", [
    (1, 32, 2.0 ** -53, 1e-14),   # double-float, one CTA
    (1, 64, 2.0 ** -53, 1e-14),   # a cluster
    (1, 340, 2.0 ** -52, 1e-14),  # a grid
    (1, 16, 2.0 ** -54, 2e-16),   # FP64
    (2, 64, 2.0 ** -54, 2e-16),
])
def test_directions_below_a_tiny_threshold_are_dropped(mode, n, small, trunc):
    big = 2.0 ** -(np.arange(n // 2) % 4)
    k, s, V, _ = _svd(np.diag(np.r_[big, np.full(n - n // 2, small)]), trunc, mode)
    assert k == n // 2
    assert np.array_equal(np.abs(V).sum(axis=0) > 0, np.arange(n) < n // 2)
    assert np.max(np.abs(s - np.sort(big)[::-1])) <= 4 * np.sqrt(n) * 2.0 ** (-46 if mode == 1 and n >= 32 else -53)


@pytest.mark.parametrize("mode,n", [(1, 16), (2, 16), (2, 64), (1, 64), (1, 340)])
def test_rounding_level_singular_values_without_a_threshold(mode, n):
    """Directions that count as zero columns are kept, their values moved by at most 4e-17 of the largest entry.

    (They are scaled up to just above 1e-17 of it, a quarter of FP64's unit
    roundoff.)  All other values are their own, exact to the roots' rounding.
    """
    tiny = [2.0 ** -58, 2.0 ** -64, 2.0 ** -70]
    d = np.r_[2.0 ** -(np.arange(n - 6) % 4), 2.0 ** -50, 2.0 ** -52, 2.0 ** -54, tiny]
    k, s, V, rep = _svd(np.diag(d), 0.0, mode)
    assert k == n
    err = np.abs(s - np.sort(d)[::-1])
    tol = 8 * 2.0 ** -46 if mode == 1 and n >= 32 else 16 * 2.0 ** -53
    assert np.max(err[:-4] / s[:-4]) <= tol
    assert np.max(err[-4:]) <= 4e-17
    assert np.max(np.abs(V @ V.conj().T - np.eye(n))) <= tol
    assert rep["min_kept_sv"] * np.linalg.norm(d) <= 4e-17


def test_fp64_svd_normalises_in_fp64():
    """svd_fp64 = 2: the kept singular values of every bond have norm one to FP64 rounding.

    Each value's own roundings (root, quotient: 4 u) and those of the norm's sum
    of k <= 64 squares over 32 lanes (7 u, halved by the root) give 2 (4 + 4) u,
    and the check's sum another 7 u; 2^-53 = u.
    """
    from paper_2303_03681_gb300 import mps
    from paper_2303_03681_gb300.inputs import MASTER_SEED, brickwork_circuit, make_rng

    n = 12
    ctx = mps.Context(0)
    for seed in range(4):
        st = mps.State(ctx, n, None, chi_max=64, precision="fp64", svd_fp64=2)
        st.apply_gates(brickwork_circuit(n, 10, make_rng(MASTER_SEED + 1600 + seed)))
        for lam in st.export()[1]:
            assert abs(float(np.sum(lam * lam)) - 1.0) <= 24 * 2.0 ** -53
