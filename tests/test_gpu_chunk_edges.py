"""The fused consumers at the edges of their 256-index chunks: first groups
shorter than a chunk, exactly a chunk and one off it, domains smaller than a
chunk, pivots in the first and the last chunk, and weights whose chunk sums
pass 32 bits."""
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


@pytest.mark.parametrize("n,n1", [(2, 1), (100, 99), (300, 255), (300, 256), (300, 257), (5000, 512), (5000, 4999),
                                  (70_001, 1), (70_001, 65_536)])
def test_mc_first_group_sizes(bs, n, n1):
    x = np.random.default_rng(n + n1).standard_normal(n).astype(np.float32)
    got = bs.mc_group_diff(torch.from_numpy(x).cuda(), n1, 9, 20).cpu().numpy()
    want = oracle.mc_statistics(x, n1, 9, 20)
    # two orders of summing n doubles of size about 1: n ulps at most
    assert np.allclose(got, want, rtol=0, atol=n * 2.0**-52)


@pytest.mark.parametrize("n,top", [(3, 10), (200, 10), (5000, 10), (5000, 2**32 - 1), (300_000, 2**32 - 1)])
@pytest.mark.parametrize("share", [0.0, 0.5, 1.0])
def test_shapley_pivot_chunks(bs, n, top, share):
    w = np.random.default_rng(n).integers(0, top, size=n, endpoint=True, dtype=np.uint32)
    total = int(w.astype(np.uint64).sum())
    quota = max(1, int(share * total) if share < 1.0 else total)
    got = bs.shapley_voting(torch.from_numpy(w.view(np.int32)).cuda(), quota, 5, 40).cpu().numpy()
    assert bs.get_error() == 0
    assert np.array_equal(got.astype(np.uint64), np.asarray(oracle.shapley_voting(w, quota, 5, 40)).astype(np.uint64))
