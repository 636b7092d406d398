"""Gathers and scatters of 1- and 2-byte elements in the pipelined single pass
against the plain fused kernel and against the input: ragged tiles, element-
aligned slices, and lengths on either side of the line between tiles of two
and of four rounds (domains of 2^24 and 2^25)."""
import pytest
import torch

from tests.gpu_helpers import assert_no_device_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.uint8, torch.int16])
@pytest.mark.parametrize("n", [1, 3, 2047, 4097, 2**18 - 1, 2**18 + 1, 2**23 + 1, 2**24 + 7])
def test_narrow_elements_match_the_plain_kernel(dtype, n):
    import paper_2106_06161_gb300 as bs
    top = 256 if dtype == torch.uint8 else 2**15
    for offset in (0, 1):
        x = torch.randint(0, top, (n + offset,), dtype=dtype, device="cuda")[offset:]
        try:
            bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_SINGLE_PASS)
            want = bs.permute(x, 11)
            bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_PIPELINED)
            got = bs.permute(x, 11)
            back = bs.inverse(got, 11)
        finally:
            bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)
        assert torch.equal(bs.permute(x, 11), want)
        assert_no_device_error()
        assert torch.equal(got, want)
        assert torch.equal(back, x)
