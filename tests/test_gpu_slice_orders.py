"""Every kept pair of slices of the exact-slice products, one by one, and full
exact runs.

Digits: a row (column) holds one element of half its power-of-two scale, which
meets a zero of the other operand, and otherwise numbers of a single digit, d
2^(-7 (i + 1)) of the scale with |d| <= 63: digit i alone is non-zero.  Rows
take i = m mod S and columns j = n mod S, so one product holds all S^2 pairs.
The sums of the pairs i + j < S are integers below 2^24 times a power of two and
come out exactly; the others are not kept and come out as zero.

Full runs: all digits at their largest, of one sign in the real part, over one
and two runs of 512 products.  The kept orders are summed in whole numbers.
The float-float sums take S orders a run, n in all: each rounds the low part,
of at most n 2^-25, by 2^-25 of it, together n^2 2^-50 of the sum, and the
order 6 of 7 may round once, 2^-55.  For S = 4 and 7 the last kept order is
6e-7 and 5e-13 of the sum.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SLICES = {"slice4": 4, "fp64_slice7": 7}


def _zgemm(A, B, prec):
    import paper_2604_27451_gb300 as pkg

    ctx = pkg.Context(0)
    C = ctx.zgemm(A, B, prec)
    ctx.close()
    return C


def _digits(rng, lines, K, S, fixed, zero):
    """[lines][K] whole digits and their values: line l of digit l mod S, the
    element `fixed` half the scale, `zero` zero (there the other operand is
    fixed)."""
    d = rng.integers(-63, 64, size=(lines, K)) + 1j * rng.integers(-63, 64, size=(lines, K))
    d[:, [fixed, zero]] = 0.0
    x = d * 2.0 ** (-7.0 * (np.arange(lines) % S + 1))[:, None]
    x[:, fixed] = 0.5
    scale = 2.0 ** rng.integers(-20, 21, size=(lines, 1))
    return d, x * scale, scale[:, 0]


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
@pytest.mark.parametrize("M, N, K", [(1040, 660, 64), (1040, 660, 300), (300, 290, 129),
                                     (257, 65, 1025), (130, 70, 20000)])
def test_single_digits(M, N, K, prec):
    S = SLICES[prec]
    rng = np.random.default_rng(M + K)
    da, A, sa = _digits(rng, M, K, S, 3, 7)
    db, Bt, sb = _digits(rng, N, K, S, 7, 3)
    # |sum| <= 2 K 63^2: in runs of 512 products below 2^24 each
    W = da @ db.T
    i, j = np.arange(M) % S, np.arange(N) % S
    order = i[:, None] + j[None, :]
    ref = np.where(order < S, W * 2.0 ** (-7.0 * (order + 2)), 0.0) * np.outer(sa, sb)
    assert np.array_equal(_zgemm(A, np.ascontiguousarray(Bt.T), prec), ref)


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
@pytest.mark.parametrize("M, N", [(300, 290), (1040, 660)])
@pytest.mark.parametrize("K", [256, 512])
def test_full_runs(M, N, K, prec):
    S = SLICES[prec]
    up = [127] + [63] * (S - 1)  # largest positive digits
    down = [-127] + [-64] * (S - 1)  # and negative ones
    val = lambda q: float(sum(d * 2.0 ** (-7 * (i + 1)) for i, d in enumerate(q)))
    A = np.full((M, K), complex(val(down), val(up)))
    B = np.full((K, N), complex(val(down), val(down)))

    def kept(a, b):  # in units of 2^(-7 (S + 1))
        return sum(a[i] * b[j] * 2 ** (7 * (S - 1 - i - j)) for i in range(S) for j in range(S - i))

    re = K * (kept(down, down) - kept(up, down))
    im = K * (kept(down, down) + kept(up, down))
    unit = 2.0 ** (-7 * (S + 1))
    n = S * (2 * K // 512)
    tol = (n * n * 2.0 ** -50 + 2.0 ** -52) * re * unit
    C = _zgemm(A, B, prec)
    assert np.abs(C.real - re * unit).max() <= tol
    assert np.abs(C.imag - im * unit).max() <= tol
