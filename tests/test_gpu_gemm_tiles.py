"""The step's GEMM at the edges of its decomposition: tiles of 8 and 16, chunks of 32 in K, the
onset of the K split, and double-float operands beyond the range that the bit-pattern
conversion takes.  Bars as for the other engine tests: relative Frobenius error 8 eps sqrt(k)
in FP64, 2^-44 sqrt(k) in double-float (a ~48-bit significand per operation)."""
import numpy as np
import pytest

from paper_2605_27515_gb300 import qlb as Q

pytestmark = pytest.mark.gpu

SHAPES = [(8, 8, 32), (9, 7, 33), (16, 16, 31), (17, 15, 64), (24, 40, 65), (8, 8, 257), (40, 40, 513), (250, 9, 96),
          (3, 1000, 2), (129, 127, 128)]
BAR = {Q.GEMM_FP64: 8 * 2.2e-16, Q.GEMM_DF64: 2.0 ** -44}


def _mats(m, n, k, seed):
    rng = np.random.default_rng(seed)
    return (rng.normal(size=(m, k)) + 1j * rng.normal(size=(m, k)),
            rng.normal(size=(k, n)) + 1j * rng.normal(size=(k, n)))


@pytest.mark.parametrize("engine", [Q.GEMM_FP64, Q.GEMM_DF64])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_tile_edges(engine, m, n, k):
    A, B = _mats(m, n, k, seed=m + 1000 * n + k)
    ref = A @ B
    C, _ = Q.qlb_zgemm_check(0, engine, A, B)
    assert np.linalg.norm(C - ref) <= BAR[engine] * np.sqrt(k) * np.linalg.norm(ref)


@pytest.mark.parametrize("power", [-80, -73, -60, 60])
def test_double_float_operand_range(power):
    """Operands whose low halves fall below 2^-73 take the conversions: the same accuracy
    there (powers of two whose products stay in FP32's range)."""
    A, B = _mats(20, 20, 40, seed=7)
    A[3, 5] = 0.0
    A[4, :] *= 2.0 ** -8
    C0, _ = Q.qlb_zgemm_check(0, Q.GEMM_DF64, A, B)
    C, _ = Q.qlb_zgemm_check(0, Q.GEMM_DF64, A * 2.0 ** power, B)
    ref = A @ B
    assert np.linalg.norm(C * 2.0 ** -power - ref) <= BAR[Q.GEMM_DF64] * np.sqrt(40) * np.linalg.norm(ref)
    assert np.linalg.norm(C0 - ref) <= BAR[Q.GEMM_DF64] * np.sqrt(40) * np.linalg.norm(ref)
