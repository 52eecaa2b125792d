"""Small outputs with a long K in the slice precisions: either side of the rule
that takes them to the 8-slice products, rows and columns that cut their tiles
and a K that ends inside a block, through the public product.

Bound of a component, by the digits: each factor is off by 2^-57 of its line's
scale (at most twice the largest component) and the pairs of order 8 and more,
7.1 2^-58 of them, are left out, over 2 K real products; the FP64 kernels and
the K slices' sums round by at most 2^-53 of the sum of moduli for each of the
at most 128 + K / 128 additions of a chain, and so does the reference.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
@pytest.mark.parametrize("M, N, K", [(157, 6, 20011), (157, 12, 40009), (129, 31, 30000),
                                     (257, 15, 32769), (200, 18, 50003), (24, 157, 40001),
                                     (64, 64, 65601), (6, 6, 100003),
                                     (157, 12, 131072), (157, 12, 131073)])
def test_small_output_long_sum(M, N, K, prec):
    import paper_2604_27451_gb300 as pkg

    rng = np.random.default_rng(M + N + K)
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((K, N)) + 1j * rng.standard_normal((K, N))
    A *= 10.0 ** rng.integers(-6, 7, size=(M, 1))
    B *= 10.0 ** rng.integers(-6, 7, size=(1, N))
    ctx = pkg.Context(0)
    C = ctx.zgemm(A, B, prec)
    ctx.close()
    top = lambda X, axis: np.maximum(np.abs(X.real), np.abs(X.imag)).max(axis)
    scale = np.outer(2 * top(A, 1), 2 * top(B, 0))
    D = C - A @ B
    slices = (2 * 2.0 ** -57 + 7.1 * 2.0 ** -58) * 2 * K * scale
    chain = 2.0 ** -53 * (256 + 2 * K / 128) * (np.abs(A) @ np.abs(B))
    assert (np.maximum(np.abs(D.real), np.abs(D.imag)) <= slices + chain).all()
