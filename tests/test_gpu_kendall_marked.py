"""Pairs of rows that are no permutations (ties) share the GPU as the others do:
each has a CTA of its own, however they follow one another."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def st():
    import paper_2106_06161_gb300
    paper_2106_06161_gb300.load()
    from paper_2106_06161_gb300 import stats
    return stats


def _tied(n, pairs, seed):
    rng = np.random.default_rng(seed)
    rows = np.argsort(rng.random((2 * pairs, n)), axis=1).astype(np.int32)
    rows[:, 0] = rows[:, 1]
    return rows


@pytest.mark.parametrize("n,pairs", [(2, 3000), (33, 2500), (40, 257)])
def test_counts_of_marked_pairs_in_a_row(st, n, pairs):
    # more than the CTAs of a launch, and not a multiple of them
    rows = _tied(n, pairs, n)
    rows[-1] = np.arange(n)  # one row without ties
    i, j = np.triu_indices(n, 1)
    s, t = rows[0::2], rows[1::2]
    want = np.sum((s[:, i] < s[:, j]) != (t[:, i] < t[:, j]), axis=1)
    assert np.array_equal(st.kendall_pairs(torch.from_numpy(rows).cuda()).cpu().numpy(), want)


def _ms(fn):
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_marked_pairs_run_side_by_side(st):
    # 256 pairs fit on the GPU at once: a few times one pair's time at most
    # (one after another they would take 256 times)
    rows = torch.from_numpy(_tied(1000, 256, 1)).cuda()
    one, many = _ms(lambda: st.kendall_pairs(rows[:2])), _ms(lambda: st.kendall_pairs(rows))
    assert many < 8 * one, (one, many)
