"""Which lengths the inverse shuffle takes through the staged path by default:
both sides of every line, seen from the passes that it timed."""
import pytest
import torch

pytestmark = pytest.mark.gpu

MIB = 2**20


@pytest.mark.parametrize("n,width,staged", [
    # n = 2^k, nothing ranked
    (2**24, 8, True), (2**23, 8, False), (2**25, 4, True), (2**24, 4, False), (2**24, 16, True), (2**23, 16, False),
    # at least three quarters of the domain kept
    (126 * MIB // 8, 8, True), (126 * MIB // 8 - 1, 8, False), (224 * MIB // 16, 16, True),
    (224 * MIB // 16 - 1, 16, False), (3 * 2**24, 4, True),
    # less
    (2**24 + 1, 8, False), (2**25 + 1, 8, True), (2**25 + 1, 4, False), (2**24 + 1, 16, False),
])
def test_default_path(n, width, staged):
    import paper_2106_06161_gb300 as bs
    x = torch.zeros((n, width // 4), dtype=torch.int32, device="cuda")
    out = torch.empty_like(x)
    s = torch.cuda.current_stream().cuda_stream
    torch.cuda.synchronize()
    bs.bshuffle_release_workspaces()
    bs.bshuffle_set_pass_timing(True)
    try:
        bs.bshuffle_inverse(x.data_ptr(), out.data_ptr(), n, width, 3, 24, s)
        passes = bs.bshuffle_last_pass_ms(s)
    finally:
        bs.bshuffle_set_pass_timing(False)
    assert len(passes) == (2 if staged else 0)
    assert bs.get_error() == 0
