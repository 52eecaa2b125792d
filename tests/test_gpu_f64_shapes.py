"""The FP64 GEMM over its tile shapes: sizes at and beside the tile edges,
single rows and columns, the core-sized sides 6 and 12 (whose tiles split k
between thread groups), short and long K with and without K slices.

Reference: complex128 matmul on the CPU.  Every computed element of either
side is within gamma = (K + 4) 2^-53 (first order) of the exact one relative
to the sum of |re|, |im| products, which is at most 2 |A||B|; the two sides
together stay within 4 (K + 4) 2^-53 |A||B|.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (1, 1, 5000), (6, 6, 17), (6, 6, 70001), (12, 12, 4097), (7, 5, 300),
          (61, 47, 83), (32, 16, 64), (33, 17, 65), (157, 6, 20000), (942, 1, 942),
          (1217, 4, 901), (5, 700, 64), (6, 300, 2000), (100, 36, 100), (65, 10, 128),
          (960, 240, 560), (64, 1, 15), (2, 3, 16), (31, 200, 33)]


@pytest.mark.parametrize("shape", SHAPES)
def test_f64_shapes(shape):
    import paper_2604_27451_gb300 as pkg

    M, N, K = shape
    rng = np.random.default_rng(M * 7 + N * 3 + K)
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((K, N)) + 1j * rng.standard_normal((K, N))
    ctx = pkg.Context(0)
    C = ctx.zgemm(A, B, "fp64")
    ctx.close()
    bound = 4.0 * (K + 4) * 2.0 ** -53 * (np.abs(A) @ np.abs(B))
    assert (np.abs(C - A @ B) <= bound).all()
