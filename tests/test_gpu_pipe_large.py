"""The pipelined single pass of launches that do not take their tickets ahead
(96 MiB and more): 1- and 2-byte elements against the plain kernel, and a tile
that withholds its status, whose successors' waits run out."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def bs():
    import paper_2106_06161_gb300 as bs
    bs.load()
    yield bs
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)


def _random(n, dtype):
    info = torch.iinfo(dtype)
    gen = torch.Generator(device="cuda").manual_seed(n)
    return torch.randint(info.min, info.max, (n,), generator=gen, device="cuda", dtype=dtype)


@pytest.mark.parametrize("call", ["permute", "inverse"])
@pytest.mark.parametrize("n,dtype", [(96 * 2**20 - 1, torch.uint8), (96 * 2**20 + 1, torch.uint8),
                                     (48 * 2**20 - 1, torch.int16), (2**26 + 1, torch.int16)])
def test_narrow_elements(bs, call, n, dtype):
    x = _random(n, dtype)
    got = getattr(bs, call)(x, 5)
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_SINGLE_PASS)
    assert torch.equal(got, getattr(bs, call)(x, 5))
    assert bs.get_error() == 0


@pytest.mark.parametrize("call", ["permute", "inverse"])
def test_withheld_tile_is_reported_and_the_next_call_exact(bs, call):
    from paper_2106_06161_gb300 import _lib as L
    x = _random(2**24 - 5, torch.int64)
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_SINGLE_PASS)
    want = getattr(bs, call)(x, 3)
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_PIPELINED)
    assert bs.get_error() == 0
    bs.bshuffle_set_lookback_timeout_ns(50_000_000)
    bs.bshuffle_debug_skip_publish(100)
    try:
        getattr(bs, call)(x, 3)
        torch.cuda.synchronize()
        assert bs.get_error() == L.BSHUFFLE_ERR_LOOKBACK_TIMEOUT
    finally:
        bs.bshuffle_debug_skip_publish(-1)
        bs.bshuffle_set_lookback_timeout_ns(2_000_000_000)
    assert bs.get_error() == 0
    got = getattr(bs, call)(x, 3)
    assert bs.get_error() == 0
    assert torch.equal(got, want)
