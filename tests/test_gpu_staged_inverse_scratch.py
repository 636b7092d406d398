"""The inverse shuffle of a length other than 2^k, asked for as staged on a
stream that has no staged buffers and, under capture, cannot get any: the
single pass serves it."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def test_captured_without_staged_buffers():
    import paper_2106_06161_gb300 as bs
    n = 100_003
    x = torch.arange(n, dtype=torch.int64, device="cuda")
    out = torch.zeros_like(x)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    bs.bshuffle_release_workspaces()
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_STAGED)
    try:
        with torch.cuda.stream(s):
            bs.permute(x[:1000], 1)  # the stream's workspace, without staged buffers
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                bs.inverse(x, 6, out=out)
    finally:
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), oracle.inverse(np.arange(n, dtype=np.int64), 6))
