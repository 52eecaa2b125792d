"""Creating a context while the default stream is busy: the error word of the
new context is cleared on the context's own stream, so a creation behind
queued work must not read what the memory held before."""

import pytest

pytestmark = pytest.mark.gpu


def test_create_while_the_default_stream_is_busy():
    import torch

    import paper_2604_27451_gb300 as pkg

    pkg.Context(0).close()
    x = torch.randn(4096, 4096, device="cuda")
    for _ in range(5):
        # non-zero bytes behind the next allocations, then queued work
        dirt = [torch.full((1 << 16,), 1, dtype=torch.int32, device="cuda") for _ in range(64)]
        torch.cuda.synchronize()
        del dirt
        torch.cuda.empty_cache()
        for _ in range(20):
            x @ x
        ctx = pkg.Context(0)
        assert ctx.device_bytes() > 0
        ctx.close()
    torch.cuda.synchronize()
