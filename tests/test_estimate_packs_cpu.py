"""The footprint estimate prices the kept operand packs by what they hold:
every slice once, 8 ns bytes per element of a B operand (two real lines of 2 ns
bf16 segments), for the two B operands of the sigma.  Host arithmetic only."""

import pytest


@pytest.mark.parametrize("nc, nw, nv, L", [(6, 60, 300, 1500), (6, 40, 200, 1000),
                                           (6, 33, 157, 785)])
def test_seven_slice_packs(nc, nw, nv, L):
    import paper_2604_27451_gb300 as pkg

    est = lambda prec: pkg.estimate_bytes(nc, nw, nv, L, nroots=4, precision=prec)
    packs = 2 * 8 * 7 * nw * nv * L
    # beside the packs: workspaces of at most 3 GiB, and a margin of a tenth
    # and the padding to tiles of 64
    more = 1.1 * (1.15 * packs + 3 * 2**30)
    assert est("fp64_slice7") - est("fp64") <= more
    assert est("slice4") - est("fp64") <= more
    # and they are priced: B^P^T's packs of a mixed precision come on top
    assert est("slice4") - est("fp64") >= packs
