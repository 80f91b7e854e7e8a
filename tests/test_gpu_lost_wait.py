"""A wait between the CTAs of a cluster kernel that runs out: whichever CTA it happens in, the
solve returns QLB_ETIMEOUT with every CTA gone, and the device works on as before."""
import numpy as np
import pytest

from paper_2605_27515_gb300 import qlb as Q

pytestmark = pytest.mark.gpu


def _usable(prec, n):
    rng = np.random.default_rng(n)
    M = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
    G = M @ M.conj().T
    lam, V, k, _ = Q.qlb_eig_check(0, prec, Q.SOLVER_STEP, G, tol=0.0, cap=n)
    # backward error of a Hermitian solve, as in the other solver tests
    eps = 2.220446049250313e-16 if prec == Q.PREC_F64 else 1.4210854715202004e-14
    assert k == n and np.max(np.abs(lam - np.linalg.eigvalsh(G)[::-1])) <= 40 * n * eps * np.linalg.norm(G, 2)


@pytest.mark.parametrize("prec", [Q.PREC_F64, Q.PREC_MIXED])
@pytest.mark.parametrize("kernel", [Q.WAIT_FACTOR, Q.WAIT_EXCHANGE, Q.WAIT_RANGE])
@pytest.mark.parametrize("n,cta", [(64, 0), (64, 3), (256, 15)])
def test_lost_wait_of_a_solve(kernel, prec, n, cta):
    with pytest.raises(Q.QlbError) as e:
        Q.qlb_lost_wait_check(0, kernel, prec, n, cta)
    assert e.value.status == Q.ETIMEOUT
    _usable(prec, n)


@pytest.mark.parametrize("cta", [0, 1])
def test_lost_wait_of_the_operator_svd(cta):
    with pytest.raises(Q.QlbError) as e:
        Q.qlb_lost_wait_check(0, Q.WAIT_SVD, Q.PREC_F64, 32, cta)
    assert e.value.status == Q.ETIMEOUT
    ctx = Q.Ctx(device=0)
    F = np.random.default_rng(1).normal(size=(16, 16)).astype(np.complex128)
    s = Q.System(ctx, [4])
    op = s.op([(1.0, [(0, Q.F_DENSE, F)])])
    assert np.linalg.norm(op.to_dense() - F) <= 1e-12 * np.linalg.norm(F)
    ctx.close()


@pytest.mark.parametrize("kernel", [Q.WAIT_FACTOR, Q.WAIT_RANGE])
def test_no_such_cta(kernel):
    """A CTA that has no part in a small problem holds nobody up."""
    Q.qlb_lost_wait_check(0, kernel, Q.PREC_F64, 6, 5)


@pytest.mark.parametrize("n,cta", [(43, 0), (200, 1)])
def test_lost_wait_of_the_qr(n, cta):
    with pytest.raises(Q.QlbError) as e:
        Q.qlb_lost_wait_check(0, Q.WAIT_QR, Q.PREC_F64, n, cta)
    assert e.value.status == Q.ETIMEOUT
    _usable(Q.PREC_F64, 64)
