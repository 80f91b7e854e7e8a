"""The operator builder's one-sided Jacobi SVD over its whole range of shapes: one CTA and a
cluster, 4 to 256 lanes per pair, slices in shared memory and outside, rows of X or of its
conjugate transpose, and the launches per round of the largest.  A dense 2^R x 2^R factor's
TT-SVD has 4^i x 4^(R-i) unfoldings and its recompression tall and wide cores.

Bar 1e-12 relative Frobenius: a row takes part in fewer than 6 * 256 rotations an SVD, whose
roundings of ~4 eps add like a random walk (sqrt(1536) * 4 eps = 3.5e-14), over fewer than 18 SVDs
(another sqrt(18): 1.5e-13)."""
import numpy as np
import pytest

from paper_2605_27515_gb300 import qlb as Q

pytestmark = pytest.mark.gpu

BAR = 1e-12


@pytest.fixture(scope="module")
def ctx():
    c = Q.Ctx(device=0)
    yield c
    c.close()


def _op(ctx, R, F, tol=0.0):
    s = Q.System(ctx, [R])
    op = s.op([(1.0, [(0, Q.F_DENSE, F)])], tol=tol)
    out = op.to_dense(), op.bond_dims()
    op.close()
    s.close()
    return out


@pytest.mark.parametrize("R", [1, 2, 3, 4, 5, 6, 7, 8])
def test_full_rank(ctx, R):
    rng = np.random.default_rng(R)
    N = 2 ** R
    F = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
    got, dims = _op(ctx, R, F)
    assert np.linalg.norm(got - F) <= BAR * np.linalg.norm(F)
    assert max([1] + dims) == 4 ** (R // 2)


@pytest.mark.parametrize("R", [4, 7, 9])
@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e60])
def test_graded_low_rank(ctx, R, scale):
    """Three products of single-site factors with weights 1, 1e-3, 1e-6: exact ranks 3, the
    rows beyond them rounding noise that must not be rotated for ever."""
    rng = np.random.default_rng(R)
    F = 0
    for w in (1.0, 1e-3, 1e-6):
        T = np.ones((1, 1))
        for _ in range(R):
            T = np.kron(T, rng.normal(size=(2, 2)) + 1j * rng.normal(size=(2, 2)))
        F = F + w * T / np.linalg.norm(T)
    got, dims = _op(ctx, R, F * scale, tol=1e-24)
    assert np.linalg.norm(got - F * scale) <= BAR * np.linalg.norm(F) * scale
    assert max(dims) == 3


def test_zero(ctx):
    got, dims = _op(ctx, 4, np.zeros((16, 16)))
    assert not got.any() and max(dims) == 1
