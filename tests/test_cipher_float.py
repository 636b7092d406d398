"""The rounds of domains up to 2^25 run in single precision (from 2^22 with one
integer multiply-add).

On the CPU: the three fused multiply-adds, in exact integer arithmetic, give
the words of the 64-bit product for every left half of every width they serve.
On the GPU: the index output on both sides of the switch, for every domain
exponent from the smallest, equals the oracle's.
"""
import numpy as np
import pytest

import oracle

M0 = 0xD2B74407B1CE6E93
LO, HI = M0 & 0xFFFFFFFF, M0 >> 32
MAX_L = 10
TWO23 = 1 << 23


def _pattern(numerator, shift):
    """Low bits of the float floor(numerator / 2^shift), which must lie in [2^23, 2^24)."""
    v = numerator >> shift
    assert (v >= TWO23).all() and (v < 2 * TWO23).all()
    return v - TWO23


@pytest.mark.parametrize("L", range(2, MAX_L + 1))
def test_products_exact(L):
    left = np.arange(1 << L, dtype=np.int64)
    mask = (1 << L) - 1
    wide = [int(v) * M0 for v in left]
    x = left + TWO23
    # high word: a 24-bit multiplier with 21 fraction bits and its addend
    mul = (7 << 21) + (LO >> 11)
    assert mul < 1 << 24 and HI & 1023 == 7
    hi = _pattern(x * mul + TWO23 * ((1 << 21) - mul), 21)
    assert np.array_equal(hi & mask, [(w >> 32) & mask for w in wide])
    # low word, plain and shifted up one bit (odd k)
    for up in (0, 1):
        m = (LO & 1023) << up
        lo = _pattern(x * m + TWO23 * (1 - m), 0)
        assert np.array_equal(lo & ((2 << L) - 1 if up else mask), [(w & mask) << up if up else w & mask for w in wide])
    # the odd bit: bit L - 1 of the low word
    m = LO & mask
    odd = _pattern(x * m + TWO23 * ((1 << (L - 1)) - m), L - 1)
    assert np.array_equal(odd & 1, [(w >> (L - 1)) & 1 for w in wide])


@pytest.mark.parametrize("L", [11, 12])
def test_mixed_products_exact(L):
    left = np.arange(1 << L, dtype=np.int64)
    mask = (1 << L) - 1
    wide = [int(v) * M0 for v in left]
    x = left + TWO23
    # high word: the pattern of floor(x * 1.694... - its low bits at left = 0), plus left * 1030
    mul = TWO23 + (LO >> 9)
    frac = _pattern(x * mul - ((mul & mask) << 23), 23)
    hi = frac + left * ((HI & 4095) - 1)
    assert np.array_equal(hi & mask, [(w >> 32) & mask for w in wide])
    for up in (0, 1):
        m = -365 << up
        lo = _pattern(x * m + TWO23 * (1 - m) + (1 << 22), 0)
        assert np.array_equal(lo & ((2 << L) - 1 if up else mask), [(w & mask) << up if up else w & mask for w in wide])
    m = LO & mask
    odd = _pattern(x * m + TWO23 * ((1 << (L - 1)) - m), L - 1)
    assert np.array_equal(odd & 1, [(w >> (L - 1)) & 1 for w in wide])


@pytest.mark.parametrize("L", range(2, 17))
def test_split_high_word_exact(L):
    # the inverse round's high word: 1.694... as 217/128 and a negative rest,
    # both multiply-adds rounded down, the first one to 24 significant bits
    left = np.arange(1 << L, dtype=np.int64)
    mask = (1 << L) - 1
    rest = LO - 0xB2000000
    assert -(1 << 22) < rest < 0 and float(np.float32(rest)) == rest
    exact = -left * rest                                   # in units of 2^-32, non-negative
    drop = np.maximum(np.array([int(v).bit_length() for v in exact]) - 24, 0)
    y = -(((exact + (1 << drop) - 1) >> drop) << drop)      # towards minus infinity
    frac = _pattern((left + TWO23) * 217 * (1 << 25) + y, 32)
    hi = frac + left * (HI - 1)
    assert np.array_equal(hi & mask, [((int(v) * M0) >> 32) & mask for v in left])


@pytest.mark.gpu
@pytest.mark.parametrize("k", range(13, 27))
def test_staged_shuffle_uses_the_inverse_cipher(k):
    import torch

    import paper_2106_06161_gb300 as bs
    bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_STAGED)
    try:
        for width, dtype in ((4, torch.int32), (8, torch.int64)):
            x = torch.arange(1 << k, dtype=dtype, device="cuda")
            got = bs.permute(x, 77)
            assert bs.get_error() == 0
            assert torch.equal(got, bs.indices(1 << k, 77, dtype=dtype))   # the forward cipher
    finally:
        bs.bshuffle_set_strategy(bs.BSHUFFLE_STRATEGY_AUTO)


@pytest.mark.gpu
@pytest.mark.parametrize("k", range(4, 27))
def test_indices_match_oracle(k):
    import torch

    import paper_2106_06161_gb300 as bs
    for n in sorted({1 << k, (1 << k) - 3, (1 << (k - 1)) + 1 if k > 4 else 9}):
        for seed in (0, 2**63 + 12345):
            got = bs.indices(n, seed, dtype=torch.int64).cpu().numpy()
            assert bs.get_error() == 0
            assert np.array_equal(got.astype(np.uint64), np.asarray(oracle.indices(n, seed)).astype(np.uint64)), (n, seed)
