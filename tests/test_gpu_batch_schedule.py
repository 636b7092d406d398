"""The batched kernel's schedule at its edges: instances on both sides of a
tile and of a warp's part of one, fewer tiles than CTAs and many more (the
look-back ring wraps), counts around the planner's runs of 32, and launches
whose ring tags follow one another."""
import numpy as np
import pytest
import torch

import oracle
from tests.gpu_helpers import to_device, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    import paper_2106_06161_gb300
    paper_2106_06161_gb300.load()
    return paper_2106_06161_gb300


def _check(bs, sizes, width, which, seed0=7):
    rng = np.random.default_rng(width)
    host = rng.integers(0, 256, size=(int(sum(sizes)), width), dtype=np.uint8)
    seeds = [seed0 + t for t in range(len(sizes))]
    got = to_host(bs.batched_packed(to_device(host), sizes, seeds), host)
    assert bs.get_error() == 0
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    for t in which:
        a, b = offs[t], offs[t + 1]
        if b > a:
            want = host[a:b][oracle.indices(int(b - a), seeds[t]).astype(np.int64)]
            assert np.array_equal(got[a:b], want), (t, b - a)


@pytest.mark.parametrize("width", [2, 4, 8, 16])
@pytest.mark.parametrize("size", [1, 127, 128, 129, 1024, 3071, 3072, 3073, 4095, 4096, 4097, 8193, 20_000])
def test_tile_edges(bs, width, size):
    _check(bs, [size, 1, size, 0, 3], width, range(5))


@pytest.mark.parametrize("count", [1, 31, 32, 33, 1023, 1025, 33_000])
def test_planner_runs(bs, count):
    sizes = np.random.default_rng(count).integers(0, 70, size=count)
    _check(bs, sizes, 4, list(range(0, count, max(1, count // 200))) + [count - 1])


def test_ring_wraps_and_tags_follow(bs):
    # 90,000 one-tile instances (two passes over the 65,536-word ring), between
    # launches of multi-tile instances that read the words left behind
    big = [70_000, 30_000, 9_000, 100_001]
    many = np.full(90_000, 17)
    for rep in range(3):
        _check(bs, big, 4, range(4), seed0=rep)
        _check(bs, many, 4, range(0, 90_000, 4999), seed0=rep)
    _check(bs, [300_000] * 40 + [5_000_000], 8, [0, 39, 40])


def test_three_streams(bs):
    sizes = [50_000, 3_000, 120_000]
    host = np.arange(sum(sizes), dtype=np.int32)
    x = torch.from_numpy(host).cuda()
    torch.cuda.synchronize()
    outs = []
    streams = [torch.cuda.Stream() for _ in range(3)]
    for rep in range(4):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                outs.append((rep * 3 + i, bs.batched_packed(x, sizes, [rep * 3 + i] * 3)))
    torch.cuda.synchronize()
    for seed, y in outs:
        y, off = y.cpu().numpy(), 0
        for n in sizes:
            assert np.array_equal(y[off:off + n], oracle.permute(host[off:off + n], seed))
            off += n
