"""The rank statistics at the edges of their 32-element steps and 32-word
bitmap rows, and the Kendall counts of rows that are no permutations (ties,
values past the length), which take the all-pairs kernel."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def st():
    import paper_2106_06161_gb300
    paper_2106_06161_gb300.load()
    from paper_2106_06161_gb300 import stats
    return stats


def _discordant(s, t):
    """#{i < j : (s_i < s_j) != (t_i < t_j)} from the definition."""
    i, j = np.triu_indices(len(s), 1)
    return int(np.sum((s[i] < s[j]) != (t[i] < t[j])))


def _counts(st, rows):
    return st.kendall_pairs(torch.from_numpy(rows.astype(np.uint32).view(np.int32)).cuda()).cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 100, 1023, 1024, 1025, 2048, 4095, 4096])
def test_inversion_counts(st, n):
    rng = np.random.default_rng(n)
    rows = [np.arange(n), np.arange(n)[::-1], np.arange(n), np.arange(n)]
    rows += [rng.permutation(n) for _ in range(36)]
    rows = np.stack(rows).astype(np.uint32)
    got = _counts(st, rows)
    assert got[0] == n * (n - 1) // 2 and got[1] == 0
    assert np.array_equal(got.astype(np.uint64), oracle.kendall_pairs(rows))


@pytest.mark.parametrize("n", [2, 33, 300])
def test_rows_that_are_no_permutations(st, n):
    rng = np.random.default_rng(n)
    perm = [rng.permutation(n) for _ in range(4)]
    tie_s, tie_t = perm[0].copy(), perm[1].copy()
    tie_s[0] = tie_s[1]
    tie_t[n - 1] = tie_t[0]
    big = perm[2].astype(np.int64)
    big[0] = n
    top = perm[3].astype(np.int64)
    top[n - 1] = 2**32 - 1
    rows = [perm[0], perm[1], tie_s, perm[1], perm[0], tie_t, big, perm[1], perm[2], top,
            np.zeros(n), np.zeros(n), perm[2], perm[3]]
    rows = np.stack([np.asarray(r, dtype=np.int64) for r in rows])
    want = [_discordant(rows[2 * p], rows[2 * p + 1]) for p in range(len(rows) // 2)]
    assert _counts(st, rows).tolist() == want


def test_marked_pairs_among_many(st):
    n, pairs = 50, 1500
    rng = np.random.default_rng(1)
    rows = np.stack([rng.permutation(n) for _ in range(2 * pairs)])
    for p in (0, 255, 256, 700, 1499):
        rows[2 * p, 3] = rows[2 * p, 4]
    want = [_discordant(rows[2 * p], rows[2 * p + 1]) for p in range(pairs)]
    assert _counts(st, rows).tolist() == want


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 255, 256, 257, 1025, 4096, 4097])
def test_sampled_ranks(st, n):
    # 4,096 is the longest row of the one-kernel form
    for seed0, rounds in ((3, 24), (2**64 - 2, 24), (3, 5)):
        got = st.sample_ranks(n, 6, seed0, rounds).cpu().numpy()
        assert got.dtype == np.int32 and got.shape == (6, n)
        for r in range(6):
            idx = oracle.indices(n, (seed0 + r) % 2**64, rounds)
            assert np.array_equal(got[r][idx], np.arange(n)), (seed0, rounds, r)


def test_sampled_ranks_of_nothing(st):
    assert st.sample_ranks(7, 0).shape == (0, 7)
    with pytest.raises(Exception):
        st.sample_ranks(0, 3)
    with pytest.raises(Exception):
        st.sample_ranks(10, 3, rounds=65)
