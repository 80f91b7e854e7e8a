"""The step's GEMM about the size where its tiles are chosen by work instead of waves (8e6
products): both sides of the line, K splits that fill the chip and that do not, and padding that
makes tiles of 8 the cheaper ones.  Bars as for the other engine tests: relative Frobenius error
8 eps sqrt(k) in FP64, 2^-44 sqrt(k) in double-float."""
import numpy as np
import pytest

from paper_2605_27515_gb300 import qlb as Q

pytestmark = pytest.mark.gpu

SHAPES = [(200, 200, 200), (200, 199, 200), (128, 128, 600), (162, 161, 496), (192, 192, 257), (7, 5000, 300),
          (300, 17, 1601), (64, 64, 4096), (513, 31, 600), (2049, 64, 64)]
BAR = {Q.GEMM_FP64: 8 * 2.2e-16, Q.GEMM_DF64: 2.0 ** -44}


@pytest.mark.parametrize("engine", [Q.GEMM_FP64, Q.GEMM_DF64])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_large_products(engine, m, n, k):
    rng = np.random.default_rng(m + 1000 * n + k)
    A = rng.normal(size=(m, k)) + 1j * rng.normal(size=(m, k))
    B = rng.normal(size=(k, n)) + 1j * rng.normal(size=(k, n))
    ref = A @ B
    C, _ = Q.qlb_zgemm_check(0, engine, A, B)
    assert np.linalg.norm(C - ref) <= BAR[engine] * np.sqrt(k) * np.linalg.norm(ref)
