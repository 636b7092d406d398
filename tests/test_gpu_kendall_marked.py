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


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 100, 511, 512, 513])
def test_few_pairs_and_many_are_counted_alike(st, n):
    # few short rows compare every pair, many take the inversion count (and its
    # marked pairs: a tie, values past the length)
    pairs, few = 1300, 70
    rng = np.random.default_rng(n)
    rows = np.argsort(rng.random((2 * pairs, n)), axis=1).astype(np.int64)
    if n > 1:
        rows[3, 0] = rows[3, 1]
        rows[8, n - 1] = n
        rows[11, 0] = 2**32 - 1
        rows[2 * pairs - 1] = 0
    dev = torch.from_numpy(rows.astype(np.uint32).view(np.int32)).cuda()
    got = st.kendall_pairs(dev).cpu().numpy()
    assert np.array_equal(got[:few], st.kendall_pairs(dev[:2 * few]).cpu().numpy())
    i, j = np.triu_indices(n, 1)
    for p in (*range(8), 500, pairs - 2, pairs - 1):
        s, t = rows[2 * p], rows[2 * p + 1]
        assert got[p] == np.sum((s[i] < s[j]) != (t[i] < t[j])), p


def test_few_short_rows_take_one_pass(st):
    # 100 pairs of length 100 take about as long as one by the all-pairs kernel
    # alone; the inversion count and its check, two launches, twice as long
    rows = np.argsort(np.random.default_rng(4).random((2 * 1300, 100)), axis=1).astype(np.int32)
    dev = torch.from_numpy(rows).cuda()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def graph(pairs):
        with torch.cuda.stream(s):
            st.kendall_pairs(dev[:2 * pairs])
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                for _ in range(50):
                    st.kendall_pairs(dev[:2 * pairs])
        return g

    def us(g):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) * 20.0

    few, many = graph(100), graph(1300)
    best = [min(us(g) for _ in range(20)) for g in (few, many)]
    # 3.2 and 7.1 us; 6.2 and 7.1 with two launches for both
    assert best[0] < 0.7 * best[1], best
