"""Rotation of B^P into natural spinors by the 8-slice products: sizes where
the rows (P, p) cut tiles, where more than one block of matrices is rotated,
and one that stays on the FP64 kernels.  The doubles part of M x for x in the
singles space, by the FP64 sigma, is linear in products of two rotated
vectors; the reference rotates B^P with the library's own spinors.

Four sums stand behind a component: two rotations over nvirt, the sum over
the Cholesky vectors and the one over the singles.  A sum of n complex
products rounds by at most 2 n 2^-53 of the norm (the 8-slice ones by less).
"""

import numpy as np
import pytest

from oracle import adc2, fns, mp2
from synth import make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
@pytest.mark.parametrize("nw, nv, naux, kept", [
    (4, 70, 64, 46), (5, 97, 66, 33), (3, 64, 80, 63), (2, 129, 35, 65), (3, 66, 60, 31)])
def test_rotated_couplings(nw, nv, naux, kept, prec):
    import paper_2604_27451_gb300 as pkg

    nc = 2
    inst = make_instance(nc, nw, nv, naux, seed=8, scale=0.1)
    occ = np.sort(np.linalg.eigvalsh(mp2.density_vv(inst.eps, inst.B, nc, nw, nv)))[::-1]
    tau = np.sqrt(occ[kept] * occ[kept - 1])
    ctx = pkg.Context(0)
    info = ctx.prepare(inst.eps, inst.B, None, nc, nw, nv, precision=prec, tau=tau)
    vk = info["nvirt_kept"]
    U = ctx.get_fns()[1]
    n1 = nc * vk
    n = n1 + nc * nw * vk * (vk - 1) // 2
    rng = np.random.default_rng(3)
    x = np.zeros((1, n), dtype=np.complex128)
    x[0, :n1] = rng.standard_normal(n1) + 1j * rng.standard_normal(n1)
    got = ctx.sigma(x, "fp64")[0, n1:]
    ctx.close()
    assert abs(vk - kept) <= 1  # a slice precision's density moves its lowest occupations
    e2, B2 = fns.rotate(inst.eps, inst.B, nc, nw, nv, U, np.zeros(vk))
    ref = adc2.m21(e2, B2, nc, nw, vk) @ x[0, :n1]
    tol = 2.0 ** -53 * 2 * (2 * nv + naux + n1)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
