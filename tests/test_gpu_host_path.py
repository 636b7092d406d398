"""The tensor API's marshalling: seeds of every size and sign in a batch,
descriptors whose host copy is still in flight when the next call fills its
own, the current stream of each call, and what is refused."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    import paper_2106_06161_gb300
    paper_2106_06161_gb300.load()
    return paper_2106_06161_gb300


@pytest.mark.parametrize("seeds", [[0, 1, 2], [-1, -2**63, 5], [2**63, 2**64 - 1, 0], [-1, 2**64 - 1, 3],
                                   [2**70 + 9, -2**65 - 1, 1], [True, 0, 7]])
def test_batch_seeds(bs, seeds):
    x = np.arange(300, dtype=np.int32)
    y = bs.batched_packed(torch.from_numpy(x).cuda(), [100, 100, 100], seeds).cpu().numpy()
    for t, s in enumerate(seeds):
        assert np.array_equal(y[100 * t:100 * t + 100], oracle.permute(x[100 * t:100 * t + 100], s % 2**64)), s


def test_descriptors_in_flight(bs):
    # each batch waits behind a long kernel, while the host goes on to the next
    x = torch.arange(40_000, dtype=torch.int32, device="cuda")
    big = torch.zeros(2**27, dtype=torch.int64, device="cuda")
    outs = []
    for rep in range(60):
        if rep % 20 == 0:
            for _ in range(5):
                big.add_(1)
        sizes = [10_000 + rep, 30_000 - rep]
        outs.append((sizes, rep, bs.batched_packed(x, sizes, [rep, rep + 1000])))
    torch.cuda.synchronize()
    host = x.cpu().numpy()
    for (a, b), rep, y in outs:
        y = y.cpu().numpy()
        assert np.array_equal(y[:a], oracle.permute(host[:a], rep)), rep
        assert np.array_equal(y[a:], oracle.permute(host[a:], rep + 1000)), rep


def test_current_stream(bs):
    x = torch.arange(5000, dtype=torch.int64, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        bs.permute(x, 3)              # a stream's first call makes its workspace and waits for it
        torch.cuda._sleep(50_000_000)
        y = bs.permute(x, 3)
        assert not s.query()          # behind the sleep, not beside it on another stream
    s.synchronize()
    assert np.array_equal(y.cpu().numpy(), oracle.permute(np.arange(5000, dtype=np.int64), 3))


def test_refusals(bs):
    x = torch.arange(10, device="cuda")
    with pytest.raises(ValueError):
        bs.permute(torch.arange(10), 1)
    with pytest.raises(ValueError):
        bs.permute(torch.tensor(3, device="cuda"), 1)
    with pytest.raises(ValueError):
        bs.inverse([1, 2], 1)
    with pytest.raises(ValueError):
        bs.permute(x, 1, out=torch.empty(9, dtype=x.dtype, device="cuda"))
    with pytest.raises(ValueError):
        bs.permute(x, 1, out=torch.empty(20, dtype=x.dtype, device="cuda")[::2])
    with pytest.raises(bs.BShuffleError):
        bs.permute(x, 1, rounds=65)
    with pytest.raises(bs.BShuffleError):
        bs.permute(x, 1, out=x)
