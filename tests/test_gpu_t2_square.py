"""Band transform of the amplitudes, of whose square only b > a is computed:
occupied counts around its 32-wide tiles (one tile, a ragged second one, an
even split), through E_MP2 and M11 against the oracle's explicit integrals.

An element of M11's second-order part sums nvirt o^2 products of an amplitude
and an integral, which are sums of naux themselves: in FP64 the part is off
by at most 2^-53 of its norm per term of the longest chain, 2 (naux + nvirt
o^2) of them on either side, and a few operations per amplitude.
"""

import numpy as np
import pytest

from oracle import adc2, mp2
from synth import make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc, nw, nv", [(2, 3, 2), (2, 29, 5), (2, 30, 6), (2, 31, 7), (3, 37, 4),
                                        (4, 60, 3), (2, 63, 5)])
def test_amplitude_square(nc, nw, nv):
    import paper_2604_27451_gb300 as pkg

    naux = 24
    inst = make_instance(nc, nw, nv, naux, seed=9, scale=0.1)
    ctx = pkg.Context(0)
    info = ctx.prepare(inst.eps, inst.B, None, nc, nw, nv, precision="fp64")
    got = ctx.get_m11()
    ctx.close()
    t2 = mp2.t2_amplitudes(inst.eps, inst.B, nc, nw, nv)
    first = adc2.m11(inst.eps, inst.B, nc, nw, nv, second_order=False)
    ref = adc2.m11(inst.eps, inst.B, nc, nw, nv, t2=t2)
    chain = 2.0 ** -53 * (4 * (naux + nv * (nc + nw) ** 2) + 32)
    tol = chain * np.linalg.norm(ref - first) + 2.0 ** -53 * 4 * naux * np.linalg.norm(ref)
    assert np.linalg.norm(got - ref) <= tol
    e = mp2.mp2_energy(inst.eps, inst.B, nc, nw, nv, t2=t2).real
    assert abs(info["emp2"] - e) <= chain * nv * abs(e)
