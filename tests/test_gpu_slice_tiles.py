"""The exact-slice GEMMs at the edges of their tiles (128 x 64 and 256 x 128
or 64 columns, K blocks of 64, runs of 512 products, K slices) and with the
digits that bring every exact run to its bound.

Bounds, relative to 2^(e_m + f_n) (the power-of-two scales, at most twice the
largest component of the row and column) and per real product: 4 slices
leave 2^-29 of either operand (2 2^-29) and drop the pairs of order 4 and
more (3.1 2^-30), together below 2^-27; 7 slices leave 2 2^-50 and drop 6.1
2^-51, below 2^-47.6.  A component of a complex product is a sum of 2 K real
ones; the float-float sums of the runs add less than 2^-42 of it.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(33, 300, 1100), (128, 64, 1300), (129, 65, 1250), (256, 64, 640), (257, 129, 320),
          (300, 33, 1024), (511, 31, 1025), (640, 700, 64), (700, 641, 65), (1200, 24, 500),
          (40, 24, 20000), (300, 300, 4160)]
BOUND = {"slice4": 2.0 ** -26, "fp64_slice7": 2.0 ** -46.6 + 2.0 ** -42}


def _check(A, B, prec):
    import paper_2604_27451_gb300 as pkg

    ctx = pkg.Context(0)
    C = ctx.zgemm(A, B, prec)
    ctx.close()
    K = A.shape[1]
    top = lambda X, axis: np.maximum(np.abs(X.real), np.abs(X.imag)).max(axis)
    scale = np.outer(2 * top(A, 1), 2 * top(B, 0))
    D = C - A @ B
    assert (np.maximum(np.abs(D.real), np.abs(D.imag)) <= BOUND[prec] * K * scale).all()


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
@pytest.mark.parametrize("shape", SHAPES)
def test_tile_edges(shape, prec):
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((K, N)) + 1j * rng.standard_normal((K, N))
    # rows and columns of very different scales
    A *= 10.0 ** rng.integers(-6, 7, size=(M, 1))
    B *= 10.0 ** rng.integers(-6, 7, size=(1, N))
    _check(A, B, prec)


@pytest.mark.parametrize("prec,slices", [("slice4", 4), ("fp64_slice7", 7)])
def test_largest_digits(prec, slices):
    """Digits 128, -64, -64, ...: every product of a run has one sign and the
    largest modulus, so the accumulators reach the bound of an exact run."""
    t = 1.0 - sum(64.0 * 2.0 ** (-7 * (i + 1)) for i in range(1, slices))
    M, N, K = 260, 70, 1040
    A = np.full((M, K), t + 1j * t)
    B = np.full((K, N), t - 1j * t)
    _check(A, B, prec)
