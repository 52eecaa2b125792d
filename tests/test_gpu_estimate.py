"""The footprint estimate stays an upper bound of what a solve holds in the
precisions that keep 7-slice packs."""

import pytest

from synth import make_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64_slice7", "bf16x3", "slice4"])
@pytest.mark.parametrize("nc, nw, nv, L", [(6, 20, 100, 500), (6, 8, 41, 203)])
def test_estimate_bounds_held_bytes(nc, nw, nv, L, prec):
    import paper_2604_27451_gb300 as pkg
    from synth import physical_scale

    inst = make_instance(nc, nw, nv, L, seed=3, scale=physical_scale(nw, nv))
    ctx = pkg.Context(0)
    ctx.solve(inst.eps, inst.B, inst.dip, nc, nw, nv, 4, precision=prec, conv=1e-6, max_iter=60)
    held = ctx.device_bytes()
    ctx.close()
    assert held <= pkg.estimate_bytes(nc, nw, nv, L, nroots=4, precision=prec)
