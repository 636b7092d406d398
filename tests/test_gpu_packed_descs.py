"""Descriptors made by packed_descs serve any stream: the call returns when they
have arrived, also behind work that its own stream still has to do."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def test_descriptors_made_on_one_stream_and_launched_on_another():
    import paper_2106_06161_gb300 as bs
    sizes, seeds = [9_000, 1, 5_000], [7, 8, 9]
    x = torch.arange(sum(sizes), dtype=torch.int32, device="cuda")
    out = torch.zeros_like(x)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(b):
        bs.batched_packed(x, sizes, seeds)  # a stream's first call makes its workspace
    with torch.cuda.stream(a):
        bs.packed_descs(x, out, sizes, seeds)  # and the first descriptors their host buffer
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(200_000_000)
        descs = bs.packed_descs(x, out, sizes, seeds)
        # the copy is over: nothing is launched on words that are still on their way
        assert a.query()
    bs.bshuffle_batched(descs.data_ptr(), len(sizes), 4, 24, b.cuda_stream)
    b.synchronize()
    host, got, lo = x.cpu().numpy(), out.cpu().numpy(), 0
    for n, seed in zip(sizes, seeds):
        assert np.array_equal(got[lo:lo + n], oracle.permute(host[lo:lo + n], seed)), (n, seed)
        lo += n
