"""The slice GEMMs on pairs of CTAs with fewer, as many and more K blocks than
their copy slots, by two contexts at the same time: a CTA of either launch
takes over the shared memory that one of the other has left, so anything that
still arrives there after its CTA has gone would change or stop a product.

The sums are deterministic, so every product equals the first one bit by bit.
The first is held against the CPU's within the bound of 4 slices (2^-26 of
2 K terms' scale, the power-of-two scales of row and column).
"""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M, N = 1040, 660  # more tiles of 128 x 64 than SMs: the pairs of CTAs in both precisions


@pytest.mark.parametrize("prec", ["slice4", "fp64_slice7"])
@pytest.mark.parametrize("K", [64, 65, 129, 200, 300, 520])
def test_slots_and_concurrent_launches(prec, K):
    import paper_2604_27451_gb300 as pkg

    rng = np.random.default_rng(K)
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((K, N)) + 1j * rng.standard_normal((K, N))
    ctx = pkg.Context(0)
    first = ctx.zgemm(A, B, prec)
    ctx.close()
    top = lambda X, axis: np.maximum(np.abs(X.real), np.abs(X.imag)).max(axis)
    scale = np.outer(2 * top(A, 1), 2 * top(B, 0))
    assert (np.abs(first - A @ B) <= 2.0 ** -26 * 2 * K * scale).all()

    bad = []

    def work():
        try:
            c = pkg.Context(0)
            for _ in range(12):
                if not np.array_equal(c.zgemm(A, B, prec), first):
                    bad.append("a product differs")
            c.close()
        except Exception as e:  # an expired wait, a CUDA error
            bad.append(repr(e))

    threads = [threading.Thread(target=work) for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
