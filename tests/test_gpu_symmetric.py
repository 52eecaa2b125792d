"""Products of which only the tiles on and above the diagonal are computed:
(ai|bj) = (bj|ai) behind the MP2 amplitudes, at sizes where the diagonal cuts
tiles of either engine and (o v) is no multiple of them, against the oracle's
t2 from explicit integrals; and the rotation of B^P into natural spinors,
Hermitian by construction, through the MP2 energy of the truncated basis.

A component of (ai|bj) is a sum of 2 naux products of components of B, each
at most top^2: FP64 rounds it by (2 naux + 4) 2^-53 of their sum, the 7-slice
products by 2^-46.6 + 2^-42 (scales of at most twice the largest component).
<ab||ij> is a difference of two, the oracle's own FP64 sums double the
bound, and t2 divides by at least the smallest gap.
"""

import numpy as np
import pytest

from oracle import fns, mp2
from synth import make_instance

pytestmark = pytest.mark.gpu

SHAPES = [(2, 3, 5, 20), (2, 9, 60, 70), (3, 10, 41, 64), (2, 6, 97, 66)]


@pytest.mark.parametrize("prec", ["fp64", "fp64_slice7"])
@pytest.mark.parametrize("shape", SHAPES)
def test_amplitudes(shape, prec):
    import paper_2604_27451_gb300 as pkg

    nc, nw, nv, naux = shape
    inst = make_instance(nc, nw, nv, naux, seed=5, scale=0.1)
    ctx = pkg.Context(0)
    info = ctx.prepare(inst.eps, inst.B, None, nc, nw, nv, precision=prec)
    t2, emp2 = ctx.get_t2()
    ctx.close()
    ref = mp2.t2_amplitudes(inst.eps, inst.B, nc, nw, nv)
    o = nc + nw
    top = np.maximum(np.abs(inst.B.real), np.abs(inst.B.imag)).max()
    per = (2 * naux + 4) * 2.0 ** -53
    if prec != "fp64":
        per = max(per, 4 * (2.0 ** -46.6 + 2.0 ** -42))
    gap = 2 * (inst.eps[o:].min() - inst.eps[:o].max())
    tol = 2 * 2 * np.sqrt(2.0) * per * 2 * naux * top ** 2 / gap
    assert np.abs(t2 - ref).max() <= tol
    e = mp2.mp2_energy(inst.eps, inst.B, nc, nw, nv, t2=ref).real
    for got in (emp2, info["emp2"]):
        # E is quadratic in <ab||ij>: relative error twice the elements'
        assert abs(got - e) <= 4 * tol * gap * np.abs(ref).sum()


@pytest.mark.parametrize("nv", [9, 34, 70])
def test_natural_spinor_rotation(nv):
    import paper_2604_27451_gb300 as pkg

    nc, nw, naux = 2, 4, 40
    inst = make_instance(nc, nw, nv, naux, seed=6, scale=0.1)
    D = mp2.density_vv(inst.eps, inst.B, nc, nw, nv)
    occ = np.sort(np.linalg.eigvalsh(D))[::-1]
    k = (2 * nv) // 3
    tau = np.sqrt(occ[k] * occ[k - 1])  # in a gap of the occupations
    n, U, et = fns.natural_spinors(inst.eps, inst.B, nc, nw, nv, tau, D=D)
    e2, B2 = fns.rotate(inst.eps, inst.B, nc, nw, nv, U, et)
    ref = mp2.mp2_energy(e2, B2, nc, nw, U.shape[1]).real
    ctx = pkg.Context(0)
    info = ctx.prepare(inst.eps, inst.B, None, nc, nw, nv, precision="fp64", tau=tau)
    ctx.close()
    assert info["nvirt_kept"] == U.shape[1]
    # the energy does not depend on the eigenvectors' phases; the kept space
    # moves by the density's rounding over the gap between occupations
    sep = (occ[k - 1] - occ[k]) / occ[0]
    assert abs(info["emp2"] - ref) <= 1e-12 / sep * abs(ref)
