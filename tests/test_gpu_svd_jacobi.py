"""The FP64-accurate truncation SVD at the edges of its launch plans (GPU).

``mps_truncated_svd`` with svd_fp64 = 1 and 2 at the sizes where the plan
changes: the smallest thetas, the last and first sizes of the single-CTA, the
4-CTA, the 8-CTA and the co-resident-grid forms, and long or wide thetas; then
thetas of every scale, a zero theta, and exact low rank without a truncation
threshold.

Tolerances: the sweeps stop when every pair is orthogonal to 4 sqrt(max(m, n))
u with u = 2^-46 (double-float) or 2^-53 (FP64), so the kept rows are held to
that, and the singular values to it times s_1; LAPACK's own error, a few
2^-53 sqrt(max(m, n)), is far inside the double-float bound and doubles the
FP64 one.
"""

import numpy as np
import pytest

from paper_2303_03681_gb300.inputs import MASTER_SEED, make_rng

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mps():
    from paper_2303_03681_gb300 import mps as m

    return m


@pytest.fixture(scope="module")
def ctx(mps):
    return mps.Context(0)


def _unitary(rng, n, r):
    q, _ = np.linalg.qr(rng.normal(size=(n, r)) + 1j * rng.normal(size=(n, r)))
    return q


def _svd(mps, ctx, A, chi_max, trunc, mode):
    import torch

    m, n = A.shape
    d = torch.from_numpy(np.ascontiguousarray(A)).cuda()
    s = torch.full((min(m, n),), float("nan"), dtype=torch.float64, device="cuda")
    vh = torch.zeros((min(chi_max, m, n), n), dtype=torch.complex128, device="cuda")
    k, rep, rc = mps.truncated_svd(ctx, "fp64", m, n, d.data_ptr(), chi_max, trunc, mode, s.data_ptr(), vh.data_ptr())
    assert rc == mps.MPS_OK and rep["svd_not_converged"] == 0
    return k, s.cpu().numpy()[:k], vh.cpu().numpy()[:k]


def _tol(m, n, mode):
    double_float = mode == 1 and n >= 32  # smaller thetas are swept in FP64
    return 4 * np.sqrt(max(m, n)) * 2.0 ** -46 if double_float else 8 * np.sqrt(max(m, n)) * 2.0 ** -53


SIZES = [(2, 2), (2, 4), (6, 2), (30, 30), (34, 32), (48, 48), (50, 50), (2, 52), (52, 2), (20, 190), (190, 20),
         (232, 232), (238, 238), (326, 330), (340, 336), (600, 340), (338, 500)]


@pytest.mark.parametrize("m,n", SIZES)
@pytest.mark.parametrize("mode", [1, 2])
def test_plan_edges(mps, ctx, m, n, mode):
    rng = make_rng(MASTER_SEED + 900 + 7 * m + n)
    r = min(m, n)
    s0 = np.repeat(10.0 ** -np.linspace(0, 7, (r + 1) // 2), 2)[:r]  # degenerate pairs over seven decades
    A = (_unitary(rng, m, r) * s0) @ _unitary(rng, n, r).conj().T
    chi = max(2, r // 4 * 2)
    k, s, V = _svd(mps, ctx, A, chi, 1e-9, mode)
    u, sr, vr = np.linalg.svd(A, full_matrices=False)
    kr = max(1, min(chi, int(np.sum(sr > 1e-9 * sr[0]))))
    tol = _tol(m, n, mode)
    assert k == kr and np.all(np.diff(s) <= 0)
    assert np.max(np.abs(s - sr[:k])) <= tol * sr[0]
    assert np.max(np.abs(V @ V.conj().T - np.eye(k))) <= tol
    # the truncated theta is unique as long as no pair is cut (chi is even)
    best = (u[:, :k] * sr[:k]) @ vr[:k]
    assert np.linalg.norm(A @ V.conj().T @ V - best) <= 4 * tol * np.linalg.norm(sr)


@pytest.mark.parametrize("scale", [1e-250, 1e-40, 1e25, 1e250])
@pytest.mark.parametrize("n", [12, 40, 64])
def test_any_scale(mps, ctx, n, scale):
    rng = make_rng(MASTER_SEED + 901 + n)
    A = (_unitary(rng, n, n) * 10.0 ** -np.linspace(0, 9, n)) @ _unitary(rng, n, n).conj().T
    k, s, V = _svd(mps, ctx, A * scale, n // 2, 1e-8, 1)
    sr = np.linalg.svd(A, compute_uv=False)
    tol = _tol(n, n, 1)
    assert k == min(n // 2, int(np.sum(sr > 1e-8 * sr[0])))
    assert np.max(np.abs(s / scale - sr[:k])) <= tol * sr[0]
    assert np.max(np.abs(V @ V.conj().T - np.eye(k))) <= tol


@pytest.mark.parametrize("n", [8, 40, 60, 400])
def test_zero_and_low_rank_without_a_threshold(mps, ctx, n):
    k, s, V = _svd(mps, ctx, np.zeros((n, n), complex), n, 0.0, 1)
    assert k == 1 and s[0] == 0.0 and abs(np.linalg.norm(V) - 1.0) == 0.0
    # rank 3: whatever rounding-level directions are kept are orthonormal too
    rng = make_rng(MASTER_SEED + 902 + n)
    A = (_unitary(rng, n, 3) * np.array([1.0, 0.5, 1e-6])) @ _unitary(rng, n, 3).conj().T
    k, s, V = _svd(mps, ctx, A, n, 0.0, 1)
    tol = _tol(n, n, 1)
    assert k >= 3 and np.max(np.abs(s[:3] - [1.0, 0.5, 1e-6])) <= tol
    assert np.all(s[3:] <= tol)
    assert np.max(np.abs(V @ V.conj().T - np.eye(k))) <= tol
