"""The Hermitian Jacobi eigensolver on both sides of the size where it moves
from one thread block to the whole grid, at even and odd sizes around its
tiles of 8 pairs, and on a spectrum of exact pairs: the natural occupations
of the MP2 density (Eqs. 15 and 17) against numpy's eigenvalues of the
oracle's density.

By Weyl's theorem an occupation moves by at most the norm of the density's
error: sums of K = nvirt nocc^2 products on either side, each within
(K + 8) 2^-53 of the sum of the moduli, which for all elements together is at
most the trace; 8 (K + 64) 2^-53 tr D covers both sides and the solvers.
"""

import numpy as np
import pytest

from oracle import fns, mp2
from synth import make_instance
from synth.generate import make_kramers_instance

pytestmark = pytest.mark.gpu


def _check(inst, nc, nw, nv):
    import paper_2604_27451_gb300 as pkg

    D = mp2.density_vv(inst.eps, inst.B, nc, nw, nv)
    tau = 1e-14
    ref = fns.natural_spinors(inst.eps, inst.B, nc, nw, nv, tau, D=D)[0]
    ctx = pkg.Context(0)
    ctx.prepare(inst.eps, inst.B, None, nc, nw, nv, precision="fp64", tau=tau)
    occ, U = ctx.get_fns()
    ctx.close()
    K = nv * (nc + nw) ** 2
    tol = 8.0 * (K + 64) * 2.0 ** -53 * np.trace(D).real
    assert np.abs(occ - ref).max() <= tol
    # U = V~ Z~ has orthonormal columns (products of two unitaries, n terms)
    assert np.abs(U.conj().T @ U - np.eye(U.shape[1])).max() <= 64 * nv * 2.0 ** -53


@pytest.mark.parametrize("nv", [2, 3, 23, 24, 25, 26, 31, 32, 33, 49])
def test_occupations(nv):
    _check(make_instance(2, 3, nv, 40, seed=nv, scale=0.1), 2, 3, nv)


def test_occupations_of_kramers_pairs():
    _check(make_kramers_instance(2, 4, 30, 40, seed=3, scale=0.1), 2, 4, 30)
