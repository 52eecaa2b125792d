"""The Ivv piece of M11 summed over pairs k < l, as the slice products do for
long sums, against the sum over all k and l of the plain FP64 build: an even
and an odd number of occupied spinors, and a sum just short of the rule.

With 7 slices a component of a product of K terms is off by at most 2 K 4
(2^-46.6 + 2^-42) of the largest components of its operands (scales of at
most twice those); the amplitude pieces enter M11 at most three times, twice
each, the two first-order ones with naux terms.
"""

import numpy as np
import pytest

from synth import make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc, nw, nv", [(2, 62, 66), (3, 60, 70), (2, 61, 65)])
def test_pair_sum(nc, nw, nv):
    import paper_2604_27451_gb300 as pkg

    naux, o = 30, nc + nw
    inst = make_instance(nc, nw, nv, naux, seed=10, scale=0.1)
    m11 = {}
    ctx = pkg.Context(0)
    for prec in ("fp64", "fp64_slice7"):
        ctx.prepare(inst.eps, inst.B, None, nc, nw, nv, precision=prec)
        m11[prec] = ctx.get_m11()
    t2 = ctx.get_t2()[0]
    ctx.close()
    t = max(np.abs(t2.real).max(), np.abs(t2.imag).max())
    g = t * 2 * (inst.eps[o:].max() - inst.eps[:o].min())
    b = max(np.abs(inst.B.real).max(), np.abs(inst.B.imag).max())
    per = 4 * (2.0 ** -46.6 + 2.0 ** -42)
    tol = per * (3 * 2 * 2 * nv * o * o * t * g + 2 * 2 * naux * b * b)
    assert np.abs(m11["fp64_slice7"] - m11["fp64"]).max() <= np.sqrt(2.0) * tol
    # and the amplitude part is far above that
    assert np.abs(m11["fp64"]).max() > 1e3 * tol
