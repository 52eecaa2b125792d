"""The word that records an expired device wait: it belongs to one context, is
read and cleared by the call it happened in, and is clear in a new context."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_error_word_is_per_context_and_cleared():
    import paper_2604_27451_gb300 as pkg

    rng = np.random.default_rng(0)
    A = rng.standard_normal((70, 90)) + 1j * rng.standard_normal((70, 90))
    a, b = pkg.Context(0), pkg.Context(0)
    for _ in range(3):
        with pytest.raises(pkg.CvsadcError) as e:
            a.wait_probe(1_000_000)
        assert e.value.code == -5  # CVSADC_ETIMEOUT
        new = pkg.Context(0)
        want = A @ A.conj().T
        for ctx in (b, new, a):  # none of them sees it
            got = ctx.zgemm(A, A.conj().T.copy())
            assert np.allclose(got, want, rtol=0, atol=1e-12)
        new.close()
    a.close()
    b.close()
