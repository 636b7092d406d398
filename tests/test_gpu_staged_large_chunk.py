"""The staged passes on either side of the input size (1 GiB) from which pass 1
takes chunks of 4,096 elements in 512 threads, for both directions, lengths of
2^k and ragged ones, against the pipelined single pass and the input."""
import pytest
import torch

from tests.gpu_helpers import assert_no_device_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n", [(torch.int64, 2**27), (torch.int64, 2**27 - 1), (torch.int64, 2**27 + 4097),
                                     (torch.int64, 2**28 - 5), (torch.int32, 2**28), (torch.int32, 2**28 + 1)])
def test_large_chunk_matches_single_pass(dtype, n):
    import paper_2106_06161_gb300 as bs
    x = torch.arange(n, dtype=dtype, device="cuda")
    try:
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_PIPELINED)
        want = bs.permute(x, 21)
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_STAGED)
        got = bs.permute(x, 21)
        assert torch.equal(got, want)
        del got
        assert torch.equal(bs.inverse(want, 21), x)
    finally:
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)
    assert_no_device_error()
