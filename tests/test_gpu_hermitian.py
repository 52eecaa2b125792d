"""The Hermiticity check of B^P at its limit, 1e-12 of the largest modulus:
deviations just inside and outside it, in one component and spread over both
(where a bound by components cannot tell), on and off the diagonal, at sizes
on both sides of the 32-wide tiles.  The largest entry is 1, and a deviation
of d is put there exactly, so the limit is crossed at d = 1e-12 up to the
rounding of one subtraction (2^-53)."""

import numpy as np
import pytest

from synth import make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [3, 27, 28, 60])
@pytest.mark.parametrize("where", ["upper", "lower", "diagonal"])
def test_limit(nv, where):
    import paper_2604_27451_gb300 as pkg

    nc, nw, naux = 2, 3, 4
    inst = make_instance(nc, nw, nv, naux, seed=nv)
    n = inst.n
    B0 = inst.B / (2 * np.abs(inst.B).max())
    B0[1, 0, 1] = B0[1, 1, 0] = 1.0
    ctx = pkg.Context(0)
    i, j = {"upper": (0, n - 1), "lower": (n - 1, 0), "diagonal": (n - 1, n - 1)}[where]
    for phase in (1j, (1 + 1j) / np.sqrt(2.0)):
        if where == "diagonal":
            phase = 0.5j  # a_ii - conj(a_ii) = twice the imaginary part
        for d, fails in ((0.0, False), (0.5e-12, False), (0.98e-12, False), (1.02e-12, True),
                         (1e-11, True)):
            B = B0.copy()
            B[2, i, j] = B[2, j, i] = 0.0
            B[2, i, j] = d * phase
            if fails:
                with pytest.raises(pkg.CvsadcError) as e:
                    ctx.prepare(inst.eps, B, None, nc, nw, nv)
                assert e.value.code == -2
            else:
                ctx.prepare(inst.eps, B, None, nc, nw, nv)
    ctx.close()
