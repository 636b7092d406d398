"""The staged inverse shuffle of lengths that are not powers of two: chunks of
the domain in order, each window of output slots filled exactly once.  Lengths
around the chunk, with nearly everything and nearly half of the domain kept,
for every width and round count path; a chunk that withholds its count; and
the default strategy at its size."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from tests.gpu_helpers import assert_no_device_error, to_device, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    import paper_2106_06161_gb300
    paper_2106_06161_gb300.load()
    return paper_2106_06161_gb300


@pytest.fixture
def staged(bs):
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_STAGED)
    yield bs
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)


@pytest.mark.parametrize("width", [4, 8, 16])
@pytest.mark.parametrize("n", [4097, 6000, 8191, 8193, 65_537, 131_071, 1_000_003, 2**21 + 1, 2**22 - 3])
def test_matches_oracle(staged, width, n):
    x = workloads.sweep_payload(n, width, 3)
    for seed, rounds in ((9, 24), (9, 23)):
        got = to_host(staged.inverse(to_device(x), seed, rounds), x)
        assert_no_device_error()
        assert np.array_equal(got, oracle.inverse(x, seed, rounds)), (seed, rounds)


def test_withheld_chunk_is_reported_and_the_next_call_exact(staged):
    from paper_2106_06161_gb300 import _lib as L
    n = 20_000                      # domain 2^15: 16 chunks of 2,048 indices
    x = np.arange(n, dtype=np.int64)
    d = to_device(x)
    staged.inverse(d, 3)
    staged.bshuffle_set_lookback_timeout_ns(50_000_000)
    staged.bshuffle_debug_skip_publish(4)
    try:
        staged.inverse(d, 3)
        torch.cuda.synchronize()
        assert staged.get_error() == L.BSHUFFLE_ERR_LOOKBACK_TIMEOUT
    finally:
        staged.bshuffle_debug_skip_publish(-1)
        staged.bshuffle_set_lookback_timeout_ns(2_000_000_000)
    got = to_host(staged.inverse(d, 3), x)
    assert staged.get_error() == 0
    assert np.array_equal(got, oracle.inverse(x, 3))


@pytest.mark.parametrize("n,width", [(2**24, 8), (2**25, 4), (2**24 - 5, 8), (2**25 + 1, 8), (2**26 + 12345, 4),
                                     (2**24 - 12345, 16), (2**24 + 1, 16), (2**28 + 12345, 8)])
def test_default_strategy_undoes_the_shuffle(bs, n, width):
    # at these sizes the default takes this path; the shuffle is checked
    # against the oracle elsewhere
    g = torch.Generator(device="cuda").manual_seed(n)
    shape = (n, 2) if width == 16 else (n,)
    x = torch.randint(-2**31, 2**31 - 1, shape, generator=g, device="cuda",
                      dtype=torch.int32 if width == 4 else torch.int64)
    y = bs.permute(x, 11)
    assert torch.equal(bs.inverse(y, 11), x)
    assert_no_device_error()
    # the single-pass kernel's output, slot by slot
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_SINGLE_PASS)
    try:
        want = bs.inverse(x, 5)
    finally:
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)
    assert torch.equal(bs.inverse(x, 5), want)
    assert_no_device_error()


def test_inside_a_graph(staged):
    n = 100_003
    x = torch.arange(n, dtype=torch.int64, device="cuda")
    want = oracle.inverse(np.arange(n, dtype=np.int64), 6)
    out = torch.empty_like(x)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        staged.inverse(x, 6, out=out)  # makes the stream's buffers
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            staged.inverse(x, 6, out=out)
    for _ in range(3):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
