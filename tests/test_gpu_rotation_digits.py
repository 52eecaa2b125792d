"""The 8-slice rotation into natural spinors against extended precision, tight
enough to tell a missing slice pair: with a vanishing B^P the amplitudes are
below 2^-60 and the singles part of the transition moments is the rotated
dipole block, F[x][I a'] = sum_a conj(U[a][a']) d^x_aI, with the library's U.

Expected root mean square of a component's error, a sum of 2 v real products
of lines with power-of-two scales s_d and s_u: the digits cut off, evenly
spread below 2^-57 of the scale, 2^-57.8 sqrt(s_d^2 |u|^2 + s_u^2 |d|^2); the
28 pairs of order 8 and above, with digits of rms 37, 2^-58.2 sqrt(2 v) s_d
s_u; the result's rounding, below 2^-54 of it.  Twice the three together is
allowed.  One missing pair of order 7 is 2^-52.6 sqrt(2 v) s_d s_u.
"""

import numpy as np
import pytest

from synth import make_instance

pytestmark = pytest.mark.gpu


def _scale(x, axis):  # 2^e with every component below it
    return 2.0 ** (np.floor(np.log2(np.maximum(np.abs(x.real), np.abs(x.imag)).max(axis))) + 1)


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
def test_rotated_dipoles(prec):
    import paper_2604_27451_gb300 as pkg

    nc, nw, nv, naux, kept = 2, 8, 200, 40, 150
    o = nc + nw
    inst = make_instance(nc, nw, nv, naux, seed=5, scale=1e-10)
    ctx = pkg.Context(0)
    ctx.prepare(inst.eps, inst.B, inst.dip, nc, nw, nv, precision=prec, tau=1e-300)
    occ = ctx.get_fns()[0]
    tau = float(np.sqrt(occ[kept - 1] * occ[kept]))
    vk = ctx.prepare(inst.eps, inst.B, inst.dip, nc, nw, nv, precision=prec,
                     tau=tau)["nvirt_kept"]
    assert 3.0 * (o + nv) * nv * vk >= 1e7  # enough work for the slices
    U = ctx.get_fns()[1]
    F = ctx.get_moments()[:, :nc * vk].reshape(3, nc, vk)
    ctx.close()
    assert U.shape == (nv, vk)

    L = np.longdouble
    ur, ui = U.real.astype(L), U.imag.astype(L)
    su = _scale(U, 0)  # [vk]
    err = var = 0.0
    for x in range(3):
        for i in range(nc):
            d = inst.dip[x][o:, i]
            dr, di = d.real.astype(L)[:, None], d.imag.astype(L)[:, None]
            re, im = (ur * dr + ui * di).sum(0), (ur * di - ui * dr).sum(0)
            err += float(((F[x, i].real - re) ** 2 + (F[x, i].imag - im) ** 2).sum())
            sd, d2 = _scale(d, 0), float((np.abs(d) ** 2).sum())
            cut = 2.0 ** -115.6 * (sd ** 2 * (np.abs(U) ** 2).sum(0) + su ** 2 * d2)
            drop = 2.0 ** -116.4 * 2 * nv * (sd * su) ** 2
            res = 2.0 ** -108 * (re ** 2 + im ** 2).astype(float)
            var += float((2 * cut + 2 * drop + res).sum())
    assert np.sqrt(err) <= 2.0 * np.sqrt(var), (np.sqrt(err), np.sqrt(var))
