"""Length of the FP64 GEMM's chains of additions where K is long or the columns
are few.  A row holds a one and otherwise 2^-54, its columns ones: a chain that
has met the one loses every later term of 2^-54, and nothing else is lost but
roundings of whole chains.  A chain of 32 loses 31 2^-54; the chains, thread
groups and K slices on the way of the one add at most 8 roundings of 2^-53 or
less (sums of 4 and more terms are exact beside the one).  Rows differ in where
the one stands.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M, N, K", [(1800, 4, 1800), (2400, 2, 1200), (5000, 1, 5000),
                                     (64, 48, 22000), (157, 6, 123245), (100, 24, 50000),
                                     (300, 300, 4160), (700, 200, 9000)])
def test_terms_lost_beside_a_one(M, N, K):
    import paper_2604_27451_gb300 as pkg

    A = np.full((M, K), 2.0 ** -54, dtype=np.complex128)
    A[np.arange(M), np.arange(M) % K] = 1.0
    ctx = pkg.Context(0)
    C = ctx.zgemm(A, np.ones((K, N), dtype=np.complex128), "fp64")
    ctx.close()
    assert (C.imag == 0).all()
    lost = (1.0 + (K - 1) * 2.0 ** -54 - C.real) * 2.0 ** 54  # within one
    assert np.abs(lost).max() <= 31 + 16 + 1
