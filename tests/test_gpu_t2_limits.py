"""The band transform at infinite and vanishing denominators: a virtual spinor
at infinity takes no part in E_MP2, and a vanishing denominator makes E_MP2
infinite, with the sign of the zero, not undefined.

E_MP2 sums o^2 v^2 / 4 terms of one sign, each a difference of sums of naux
products: within (2 naux + o^2 v^2) 2^-53 of itself on either side in FP64.
"""

import numpy as np
import pytest

from oracle import mp2
from synth import make_instance

pytestmark = pytest.mark.gpu


def _emp2(eps, B, nc, nw, nv):
    import paper_2604_27451_gb300 as pkg

    ctx = pkg.Context(0)
    e = ctx.prepare(eps, B, None, nc, nw, nv, precision="fp64")["emp2"]
    ctx.close()
    return e


@pytest.mark.parametrize("nc, nw, nv", [(2, 3, 6), (2, 34, 5)])
@pytest.mark.parametrize("which", [0, 3])
def test_virtual_at_infinity(nc, nw, nv, which):
    naux, o = 20, nc + nw
    inst = make_instance(nc, nw, nv, naux, seed=2, scale=0.1)
    eps = inst.eps.copy()
    eps[o + which] = np.inf
    rest = [p for p in range(o + nv) if p != o + which]
    ref = mp2.mp2_energy(inst.eps[rest], inst.B[:, rest][:, :, rest], nc, nw, nv - 1).real
    got = _emp2(eps, inst.B, nc, nw, nv)
    assert abs(got - ref) <= 4 * (2 * naux + (o * nv) ** 2) * 2.0 ** -53 * abs(ref)


def test_vanishing_denominator():
    nc, nw, nv, naux = 2, 3, 6, 20
    o = nc + nw
    inst = make_instance(nc, nw, nv, naux, seed=2, scale=0.1)
    eps = inst.eps.copy()
    eps[3], eps[4], eps[o], eps[o + 1] = 0.5, 0.75, 0.25, 1.0  # e_3 + e_4 = e_a + e_b
    assert _emp2(eps, inst.B, nc, nw, nv) == np.inf
