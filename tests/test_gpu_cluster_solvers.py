"""The cluster solves of the step (pivoted Cholesky with one-sided Jacobi; the range basis
with its columns spread over the CTAs) through qlb_eig_check, at the sizes where their split
over CTAs changes and on matrices with exact structure.

Bars, in units of the working precision's eps (2.2e-16, and 2^-46 for double-float): the
backward error of a Hermitian solve and the loss of orthogonality of n vectors are both
bounded by a small multiple of n eps ||G||; 40 n eps is the bar of the other solver tests.
Scaling G by a power of two scales the arithmetic exactly, so the kept vectors must not
change by a bit."""
import numpy as np
import pytest

from paper_2605_27515_gb300 import qlb as Q

pytestmark = pytest.mark.gpu

EPS = {Q.PREC_F64: 2.220446049250313e-16, Q.PREC_MIXED: 1.4210854715202004e-14}
# one below, at and above every size where the number of CTAs changes, and the last sizes
EDGES = [1, 3, 8, 9, 16, 17, 24, 25, 32, 33, 48, 49, 64, 65, 88, 89, 96, 97, 128, 129, 241, 256, 257]
PRECS = [Q.PREC_F64, Q.PREC_MIXED]


def _gram(n, rank, spread, seed):
    rng = np.random.default_rng(seed)
    M = rng.normal(size=(n, rank)) + 1j * rng.normal(size=(n, rank))
    M = M * np.logspace(0, -spread, rank)[None, :]
    G = M @ M.conj().T
    return 0.5 * (G + G.conj().T)


def _check_eig(prec, G, lam, V, k):
    n = G.shape[0]
    scale = np.linalg.norm(G, 2)
    ref = np.maximum(np.sort(np.linalg.eigvalsh(G))[::-1], 0)
    tol = 40 * n * EPS[prec] * scale
    assert np.max(np.abs(lam - ref)) <= tol
    assert np.max(np.abs(V.conj().T @ V - np.eye(k))) <= 40 * n * EPS[prec]
    assert np.max(np.linalg.norm(G @ V - V * lam[:k][None, :], axis=0)) <= tol


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n", EDGES)
def test_solves_at_the_edges_of_their_split(prec, n):
    rank = max(1, (2 * n) // 3)
    G = _gram(n, rank, 4, seed=100 + n)
    lam, V, k, _ = Q.qlb_eig_check(0, prec, Q.SOLVER_STEP, G, tol=1e-10, cap=n)
    _check_eig(prec, G, lam, V, k)
    assert k <= rank
    _, U, r, _ = Q.qlb_eig_check(0, prec, Q.SOLVER_RANGE, G, tol=1e-10, cap=n)
    assert 1 <= r <= rank
    assert np.max(np.abs(U.conj().T @ U - np.eye(r))) <= 40 * n * EPS[prec]
    left = np.trace(G).real - np.trace(U.conj().T @ G @ U).real
    assert left <= 1e-10 * np.trace(G).real + 40 * n * EPS[prec] * np.linalg.norm(G)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n", [9, 33, 100])
def test_structured_matrices(prec, n):
    """Equal eigenvalues, exact zeros, one direction, and nothing at all."""
    half = np.diag((np.arange(n) % 2).astype(np.complex128))
    one = np.ones((n, n), dtype=np.complex128)
    for G, rank in ((np.eye(n, dtype=np.complex128), n), (half, n // 2), (one, 1)):
        lam, V, k, _ = Q.qlb_eig_check(0, prec, Q.SOLVER_STEP, G, tol=1e-12, cap=n)
        assert k == rank
        _check_eig(prec, G, lam, V, k)
        _, U, r, _ = Q.qlb_eig_check(0, prec, Q.SOLVER_RANGE, G, tol=1e-12, cap=n)
        assert r == rank
        assert np.max(np.abs(U @ (U.conj().T @ G) - G)) <= 40 * n * EPS[prec] * np.linalg.norm(G, 2)
    zero = np.zeros((n, n), dtype=np.complex128)
    for solver in (Q.SOLVER_STEP, Q.SOLVER_RANGE):
        _, V, k, _ = Q.qlb_eig_check(0, prec, solver, zero, tol=1e-12, cap=n)
        assert k == 1 and abs(np.linalg.norm(V) - 1.0) <= 4 * EPS[prec]


@pytest.mark.parametrize("solver", [Q.SOLVER_STEP, Q.SOLVER_RANGE])
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n", [12, 40, 100])
def test_power_of_two_scale_changes_nothing(prec, n, solver):
    """G scaled by 2^-300 and 2^300 (outside FP32's range): the same vectors bit for bit."""
    G = _gram(n, n, 3, seed=n)
    _, V0, k0, _ = Q.qlb_eig_check(0, prec, solver, G, tol=1e-9, cap=n)
    for s in (2.0 ** -300, 2.0 ** 300):
        _, V, k, _ = Q.qlb_eig_check(0, prec, solver, G * s, tol=1e-9, cap=n)
        assert k == k0
        np.testing.assert_array_equal(V, V0)
