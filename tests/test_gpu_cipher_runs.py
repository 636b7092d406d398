"""Runs of consecutive indices that share the cipher's first round, on either
side of the left half's width from which they do (domains of 2^13 to 2^16 for
runs of 128 and 256 indices, 2^22 and 2^24 for the wide strides), against the
oracle."""
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


@pytest.mark.parametrize("k", [4, 9, 12, 13, 14, 15, 16, 17, 22])
@pytest.mark.parametrize("rounds", [23, 24])
def test_pipelined_indices_and_scatter(bs, k, rounds):
    n = (1 << k) - 3
    want = oracle.indices(n, 3, rounds)
    x = torch.arange(n, device="cuda")
    try:
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_PIPELINED)
        got = bs.indices(n, 3, rounds=rounds, dtype=torch.int32)
        back = bs.inverse(bs.permute(x, 3, rounds=rounds), 3, rounds=rounds)
    finally:
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)
    assert np.array_equal(got.cpu().numpy().astype(np.uint64), want)
    assert torch.equal(back, x)


@pytest.mark.parametrize("k", [4, 11, 14, 21, 22, 24])
def test_power_of_two_indices(bs, k):
    got = bs.indices(1 << k, 3, dtype=torch.int32)
    assert np.array_equal(got.cpu().numpy().astype(np.uint64), oracle.indices(1 << k, 3))


@pytest.mark.parametrize("k", [12, 13, 14, 15, 16, 17])
def test_fused_consumers(bs, k):
    n = (1 << k) - 3
    rng = np.random.default_rng(k)
    x = rng.integers(-100, 100, size=n).astype(np.float32)  # exact sums
    got = bs.mc_group_diff(torch.from_numpy(x).cuda(), n // 3, 9, 10).cpu().numpy()
    # whole-number sums; two quotients and their difference, each rounded once
    assert np.allclose(got, oracle.mc_statistics(x, n // 3, 9, 10), rtol=0, atol=4 * 100 * 2.0**-52)
    w = rng.integers(0, 1000, size=n, dtype=np.uint32)
    quota = int(w.sum()) // 2
    got = bs.shapley_voting(torch.from_numpy(w.view(np.int32)).cuda(), quota, 5, 10).cpu().numpy()
    assert bs.get_error() == 0
    assert np.array_equal(got.astype(np.uint64), np.asarray(oracle.shapley_voting(w, quota, 5, 10)).astype(np.uint64))
