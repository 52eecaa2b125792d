"""Small outputs of a long K are FP64 in the slice precisions too: entries that
are small beside the largest one of their row, infinities and not-a-numbers,
and rows and columns whose largest entries multiply beyond the range although
the sums are finite.

FP64 sums are within (K + 4) 2^-53 of the sum of moduli, per component of two
products and on both sides: 4 (K + 4) 2^-53 |A||B| together.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M, N, K = 100, 24, 20000


def _product(A, B, prec):
    import paper_2604_27451_gb300 as pkg

    ctx = pkg.Context(0)
    C = ctx.zgemm(A, B, prec)
    ctx.close()
    return C


def _inputs(seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((K, N)) + 1j * rng.standard_normal((K, N))
    return A, B


def _close(C, A, B):
    bound = 4.0 * (K + 4) * 2.0 ** -53 * (np.abs(A) @ np.abs(B))
    return (np.abs(C - A @ B) <= bound).all()


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
@pytest.mark.parametrize("big", [1e18, 1e200])
def test_wide_rows_and_columns(prec, big):
    A, B = _inputs(1)
    A[::7, 0] = big
    B[0] = 0.0
    A[:, 1] = 0.0
    B[1, ::5] = big
    assert _close(_product(A, B, prec), A, B)


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
def test_infinite_and_nan_entries(prec):
    A, B = _inputs(2)
    ref_A = A.copy()
    A[3, 11] = complex(np.nan, 1.0)
    A[4, 12] = complex(-np.inf, 1.0)
    C = _product(A, B, prec)
    assert np.isnan(C[3].real).all() and np.isnan(C[3].imag).all()
    assert (C[4].real == -np.inf * B[12].real).all()
    assert (C[4].imag == -np.inf * B[12].imag).all()
    rest = [m for m in range(M) if m not in (3, 4)]
    assert _close(C[rest], ref_A[rest], B)
