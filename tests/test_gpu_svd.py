"""The operator builder's SVD on its own (qlb_svd_check): orthonormal factors and U R = A on tall
and wide matrices whose rows or columns are graded down to, and past, the rounding level.

Bars: U or R holds vectors of up to 520 entries, each rotated fewer than 6 * 520 times or
projected twice, so 40 k eps bounds their loss of orthogonality as in the other solver tests;
1e-12 relative Frobenius for U R (rotations' roundings, as for whole operators)."""
import numpy as np
import pytest

from paper_2605_27515_gb300 import qlb as Q

pytestmark = pytest.mark.gpu

EPS = 2.220446049250313e-16


@pytest.fixture(scope="module")
def ctx():
    c = Q.Ctx(device=0)
    yield c
    c.close()


def _unitary(rng, n, k):
    return np.linalg.qr(rng.normal(size=(n, k)) + 1j * rng.normal(size=(n, k)))[0]


def _graded(m, n, decades, seed):
    """Singular values falling evenly over `decades`."""
    rng = np.random.default_rng(seed)
    k = min(m, n)
    return (_unitary(rng, m, k) * np.logspace(0, -decades, k)) @ _unitary(rng, n, k).conj().T


def _deficient(m, n, rank, seed):
    """Exact rank `rank` up to rounding, as the stacked cores of a sum of operators have."""
    rng = np.random.default_rng(seed)
    return rng.normal(size=(m, rank)) @ (rng.normal(size=(rank, n)) + 1j * rng.normal(size=(rank, n)))


SHAPES = [(4, 1), (8, 2), (40, 10), (64, 16), (41, 40), (172, 43), (1000, 12), (3000, 100), (560, 520)]
CASES = ["graded 14", "graded 30", "rank 1", "rank half", "equal columns"]


def _matrix(m, n, case, seed=3):
    if case.startswith("graded"):
        return _graded(m, n, int(case.split()[1]), seed)
    if case == "equal columns":
        return np.repeat(_graded(m, 1, 0, seed), n, axis=1)
    return _deficient(m, n, 1 if case == "rank 1" else max(1, min(m, n) // 2), seed)


def _check(ctx, A, u_scale, tol):
    U, R = Q.qlb_svd_check(ctx, A, tol=tol, u_scale=u_scale, r_unscale=u_scale)
    k = U.shape[1]
    assert 1 <= k <= min(A.shape)
    assert np.linalg.norm(U @ R - A) <= 1e-12 * np.linalg.norm(A)
    return U, R, k


@pytest.mark.parametrize("tol", [1e-32, 0.0])
@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("m,n", SHAPES)
def test_tall_left_factor_is_orthonormal(ctx, m, n, case, tol):
    """The left factor of a left-canonical sweep (singular values in R)."""
    U, R, k = _check(ctx, _matrix(m, n, case), False, tol)
    assert np.max(np.abs(U.conj().T @ U - np.eye(k))) <= 40 * k * EPS


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("m,n", [(64, 16), (16, 64), (172, 43), (43, 172)])
def test_unitary_side(ctx, m, n, case):
    """The factor that the accumulated rotations give: U of a wide matrix, R of a tall one."""
    tall = m > n
    U, R, k = _check(ctx, _matrix(m, n, case), tall, 1e-32)
    Z = R.conj().T if tall else U
    assert np.max(np.abs(Z.conj().T @ Z - np.eye(k))) <= 40 * k * EPS


@pytest.mark.parametrize("m,n", [(40, 39), (39, 40), (64, 16), (300, 250)])
def test_memory(m, n):
    """Device memory beside the matrix: at most the rotations and a left factor of m x m and a
    right factor of m x n (and 4 KB of counts and scratch), the budget the rows' own rotation needs."""
    budget = 16 * (2 * m * n + 2 * m * m) + 4096
    c = Q.Ctx(device=0, hbm_budget=budget)
    U, R = Q.qlb_svd_check(c, _graded(m, n, 3, 1), tol=1e-32)
    assert U.shape[1] == min(m, n)
    c.close()


@pytest.mark.parametrize("power", [0, -440, -455, -500, 455])
@pytest.mark.parametrize("m,n", [(2, 3), (9, 20), (20, 9), (40, 40)])
def test_orthogonal_rows_of_any_size(ctx, m, n, power):
    """Rows without a common entry, one of them zero: their couplings are exact zeros, so nothing is
    rotated however small the entries are (squares down to 2^-1000), and the factors are exact (a
    tall matrix's to rounding)."""
    rng = np.random.default_rng(m + n)
    A = np.zeros((m, n), dtype=np.complex128)
    d = min(m, n)
    A[np.arange(d), rng.permutation(n)[:d]] = np.arange(2.0, d + 2.0) * 2.0 ** power
    A[d // 2] = 0.0
    U, R = Q.qlb_svd_check(ctx, A)
    assert U.shape[1] == d - 1
    if m > n:  # through a QR, whose column norms round
        k = d - 1
        assert np.max(np.abs(U @ R - A)) <= 40 * k * EPS * np.max(np.abs(A))
        assert np.max(np.abs(np.sort(np.abs(U), axis=0)[-1] - 1.0)) <= 40 * k * EPS
        assert np.count_nonzero(np.abs(U) > 40 * k * EPS) == k
    else:
        np.testing.assert_array_equal(U @ R, A)
        np.testing.assert_array_equal(np.sort(np.abs(U), axis=0)[-1], 1.0)
        assert np.count_nonzero(U) == d - 1


# beyond one CTA's rows, a column's shared memory, and the cluster's; a row more than columns
@pytest.mark.parametrize("m,n", [(2, 1), (33, 32), (257, 5), (13000, 2), (14000, 20), (900, 400), (4200, 60)])
def test_tall_shapes(ctx, m, n):
    rng = np.random.default_rng(m)
    A = rng.normal(size=(m, n)) + 1j * rng.normal(size=(m, n))
    A[:, n // 2] = 0.0  # a column without a reflector
    U, R = Q.qlb_svd_check(ctx, A, tol=1e-28)
    k = U.shape[1]
    assert k == (n - 1 if n > 1 else 1)
    assert np.linalg.norm(U @ R - A) <= 1e-12 * max(np.linalg.norm(A), 1e-300)
    assert np.max(np.abs(U.conj().T @ U - np.eye(k))) <= 40 * k * EPS


def test_operator_ranks():
    """Ranks of the transmon-resonator Hamiltonian, whose sum of five terms has cores of up to
    100 x 25 of lower rank: rounding must not pass for content (those of rotating a tall core's
    own rows, which leaves exact zeros where the operator has them)."""
    from paper_2605_27515_gb300 import inputs, systems

    cfg = inputs.config("transmon")
    c = Q.Ctx(device=0)
    b = systems.build_transmon(c, cfg, nsteps=1)
    assert b.ops["H0"].bond_dims() == [4, 5, 5, 5, 5, 5, 3, 6, 8, 12, 12, 12, 12, 11, 7, 4]
    assert b.ops["H1"].bond_dims() == [1, 1, 1, 1, 1, 1, 1, 4, 6, 10, 11, 11, 11, 9, 5, 2]
    c.close()


@pytest.mark.parametrize("R", [3, 6, 9])
def test_far_levels_stay_uncoupled(R):
    """a^2 - alpha^2 couples levels n and n - 2 only: every other off-diagonal entry of its MPO is an
    exact zero, as the supports of the cores' rows do not meet."""
    c = Q.Ctx(device=0)
    s = Q.System(c, [R])
    D = s.op([(1.0, [(0, Q.F_A, 2)]), (-16.0, [])]).to_dense()
    i, j = np.indices(D.shape)
    assert np.count_nonzero(D[(i != j) & (j != i + 2)]) == 0
    c.close()
