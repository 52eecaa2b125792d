"""The eigensolver's two launches per step, from 400 indices on: sizes either
side of it, odd ones (a bye in every step) and one beyond a whole number of
tiles, through the natural occupations against numpy's eigenvalues of the
oracle's density, and the spinors' orthonormality.

An occupation moves by at most the norm of the density's error (Weyl): sums of
K = nvirt nocc^2 products on either side, each within (K + 8) 2^-53 of the sum
of the moduli, at most the trace for all elements together: 8 (K + 64) 2^-53
tr D covers both sides and the solvers.  U is a product of two unitaries of n
terms: 64 nvirt 2^-53.
"""

import numpy as np
import pytest

from oracle import mp2
from synth import make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [399, 400, 401, 450, 513])
def test_occupations_and_spinors(nv):
    import paper_2604_27451_gb300 as pkg

    nc, nw = 2, 3
    inst = make_instance(nc, nw, nv, 40, seed=nv, scale=0.1)
    D = mp2.density_vv(inst.eps, inst.B, nc, nw, nv)
    ref = np.linalg.eigvalsh(D)[::-1]
    ctx = pkg.Context(0)
    # half of the spinors, between two occupations
    tau = float(np.sqrt(ref[nv // 2 - 1] * ref[nv // 2]))
    vk = ctx.prepare(inst.eps, inst.B, None, nc, nw, nv, precision="fp64", tau=tau)["nvirt_kept"]
    occ, U = ctx.get_fns()
    ctx.close()
    tol = 8.0 * (nv * (nc + nw) ** 2 + 64) * 2.0 ** -53 * np.trace(D).real
    assert np.abs(occ - ref).max() <= tol
    eye = 64 * nv * 2.0 ** -53
    assert np.abs(U.conj().T @ U - np.eye(vk)).max() <= eye
    # the kept spinors carry their occupations: tr U^H D U is their sum
    assert abs(np.trace(U.conj().T @ D @ U).real - ref[:vk].sum()) <= vk * tol + eye * ref.sum()
