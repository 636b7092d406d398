"""On domains where a launch is all latency the default is the plain single
pass, whatever the element and the round count."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _graph(fn, stream, calls=40):
    fn()
    stream.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for _ in range(calls):
            fn()
    return g


def _ms(g):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    g.replay()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b)


@pytest.mark.parametrize("dtype,n,rounds", [(torch.int16, 2**17 + 1, 24), (torch.int16, 700_001, 24),
                                            (torch.uint8, 2**18 - 3, 10), (torch.int32, 2**17 + 1, 10)])
def test_default_is_no_slower_than_the_plain_kernel(dtype, n, rounds):
    import paper_2106_06161_gb300 as bs
    x = torch.zeros(n, dtype=dtype, device="cuda")
    out = torch.empty_like(x)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    best = [float("inf")] * 2
    # several captures of each: the time of one graph of launches that short
    # settles at one of two values
    for _ in range(5):
        for i, strategy in enumerate((bs.BSHUFFLE_STRATEGY_AUTO, bs.BSHUFFLE_STRATEGY_SINGLE_PASS)):
            bs.bshuffle_set_strategy(strategy)
            try:
                with torch.cuda.stream(s):
                    g = _graph(lambda: bs.permute(x, 3, rounds, out=out), s)
            finally:
                bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)
            best[i] = min(best[i], *(_ms(g) for _ in range(10)))
    # the same kernel; the pipelined one takes 1.1 to 1.3 times as long here
    assert best[0] < 1.07 * best[1], best
