"""What a user has this library do, as cases that can be timed and compared.

A case is a dict of plain values; "kind" names the entry point:

  permute / inverse   one shuffle (or its undoing) of n elements of 1 to 16 bytes
  indices             the source index of every output slot
  batched             independent shuffles of uneven segments in one call
  rows                the differentiable row shuffle, forward and backward
  mc                  the permutation-test statistic, `count` shuffles of n values
  shapley             pivot counts of a weighted voting game over sampled orders
  ranks               sampled permutations and the Kendall counts of their pairs
                      (the two GPU steps of the Mallows-kernel MMD test)

The sizes are those of workloads.py and bench.py (the paper's worst-case lengths
2^w + 1, the sweep of widths, the 4096 uneven instances, the [65536 x 1024]
rows, the 50,000 + 50,000 samples, the 10,000 players, 100,000 permutations).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2106_06161_gb300 as bs
from paper_2106_06161_gb300 import stats

ROUNDS = 24
_INT = {1: torch.uint8, 2: torch.int16, 4: torch.int32, 8: torch.int64}
_FLOAT = {"float32": torch.float32, "bfloat16": torch.bfloat16}


def listed() -> list[dict]:
    return [
        # the smallest call: a handful of keys, all latency (first column of the paper's Table 1)
        {"name": "keys_257", "kind": "permute", "n": 257, "bytes": 8},
        # the ordinary call: a million 4-byte values, resident in L2
        {"name": "values_1000003", "kind": "permute", "n": 1_000_003, "bytes": 4},
        # the benchmark: 2 GiB of 64-bit keys, nothing dropped
        {"name": "keys_2p28", "kind": "permute", "n": 2**28, "bytes": 8},
        # the same with the worst padding: the domain is nearly twice the length
        {"name": "keys_2p28_12345", "kind": "permute", "n": 2**28 + 12345, "bytes": 8},
        # a corpus of 16-bit token ids
        {"name": "tokens_2p26_1", "kind": "permute", "n": 2**26 + 1, "bytes": 2},
        # {key, value} records put back in their first order
        {"name": "inverse_records_2p24_1", "kind": "inverse", "n": 2**24 + 1, "bytes": 16},
        # the epoch order of a data loader: indices alone
        {"name": "indices_2p23_1", "kind": "indices", "n": 2**23 + 1, "bytes": 8},
        # many uneven segments at once (per-group or per-shard shuffles)
        {"name": "batched_4096", "kind": "batched", "count": 4096, "lo": 100, "hi": 2_000_000, "bytes": 4},
        # a training step's row shuffle: activations forward, gradients backward
        {"name": "rows_65537", "kind": "rows", "rows": 65537, "cols": 1024, "dtype": "bfloat16"},
        # a permutation test of two groups of 50,000
        {"name": "mc_100000", "kind": "mc", "n": 100_000, "n1": 50_000, "count": 10_000},
        # Shapley values of 10,000 players by sampling, simple majority
        {"name": "shapley_10000", "kind": "shapley", "n": 10_000, "count": 100_000},
        # the statistical test of Sec. 5 at its largest length
        {"name": "ranks_1000", "kind": "ranks", "n": 1000, "count": 100_000},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["permute", "permute", "permute", "inverse", "inverse", "indices", "indices",
                       "batched", "batched", "rows", "rows", "mc", "shapley", "ranks"])
    if kind in ("permute", "inverse", "indices"):
        width = rng.choice([4, 8] if kind == "indices" else [1, 2, 4, 4, 8, 8, 8, 16])
        n = _log_int(rng, 200, (2**28 + 12345) * 8 // max(width, 8))
        shape = rng.random()
        if shape < 0.2:  # nothing dropped
            n = 1 << (n.bit_length() - 1)
        elif shape < 0.4:  # the worst padding
            n = (1 << (n.bit_length() - 1)) + 1
        return {"kind": kind, "n": n, "bytes": width}
    if kind == "batched":
        return {"kind": kind, "count": _log_int(rng, 16, 2048), "lo": 100, "hi": _log_int(rng, 1000, 2_000_000),
                "bytes": rng.choice([1, 2, 4, 4, 8])}
    if kind == "rows":
        dtype = rng.choice(sorted(_FLOAT))
        cols = 8 * _log_int(rng, 4, 512)
        most = 2**26 // cols
        rows = _log_int(rng, 256, most)
        if rng.random() < 0.3:
            rows = 1 << (rows.bit_length() - 1)
        return {"kind": kind, "rows": rows, "cols": cols, "dtype": dtype}
    if kind == "mc":
        n = _log_int(rng, 100, 100_000)
        return {"kind": kind, "n": n, "n1": max(1, int(n * rng.uniform(0.05, 0.95))), "count": _log_int(rng, 100, 10_000)}
    if kind == "shapley":
        return {"kind": kind, "n": _log_int(rng, 8, 10_000), "count": _log_int(rng, 1000, 100_000)}
    return {"kind": kind, "n": _log_int(rng, 5, 1000), "count": 2 * _log_int(rng, 500, 50_000)}


# ------------------------------------------------------------------ inputs


def _values(n: int, width: int, seed: int) -> torch.Tensor:
    """n uniform random elements of `width` bytes; 16 bytes are {key, number} records."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if width == 16:
        rec = torch.empty(n, 2, dtype=torch.int64, device="cuda")
        rec[:, 0] = torch.randint(-2**63, 2**63 - 1, (n,), generator=gen, device="cuda")
        rec[:, 1] = torch.arange(n, device="cuda")
        return rec
    info = torch.iinfo(_INT[width])
    return torch.randint(info.min, info.max, (n,), generator=gen, device="cuda", dtype=_INT[width])


def _samples(case: dict, seed: int) -> torch.Tensor:
    """Two groups, N(0, 1) and N(0.05, 1)."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(case["n"])
    x[case["n1"]:] += 0.05
    return torch.from_numpy(x.astype(np.float32)).cuda()


def _segments(case: dict) -> np.ndarray:
    """Log-uniform segment lengths: the case's own, whatever the data's seed."""
    u = np.random.default_rng(2024).uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["count"])
    return np.floor(np.exp(u)).astype(np.int64)


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    state = {"case": case, "seed": seed * 7919 + 1}  # the shuffle's seed
    if kind in ("permute", "inverse"):
        state["x"] = _values(case["n"], case["bytes"], seed)
    elif kind == "batched":
        state["sizes"] = _segments(case)
        state["seeds"] = [state["seed"] + t for t in range(case["count"])]
        state["x"] = _values(int(state["sizes"].sum()), case["bytes"], seed)
    elif kind == "rows":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        shape = (case["rows"], case["cols"])
        state["x"] = torch.randn(shape, generator=gen, device="cuda").to(_FLOAT[case["dtype"]]).requires_grad_()
        state["grad"] = torch.randn(shape, generator=gen, device="cuda").to(_FLOAT[case["dtype"]])
    elif kind == "mc":
        state["x"] = _samples(case, seed)
    elif kind == "shapley":
        w = (1 + np.floor(np.random.default_rng(seed).lognormal(2.0, 1.0, size=case["n"]))).astype(np.int32)
        state["quota"] = int(w.sum()) // 2 + 1
        state["weights"] = torch.from_numpy(w).cuda()
    return state


# ------------------------------------------------------------------ one pass


def run(state: dict):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "permute":
        return bs.permute(state["x"], seed=seed)
    if kind == "inverse":
        return bs.inverse(state["x"], seed=seed)
    if kind == "indices":
        return bs.indices(case["n"], seed=seed, dtype=_INT[case["bytes"]])
    if kind == "batched":
        return bs.batched_packed(state["x"], state["sizes"], state["seeds"])
    if kind == "rows":
        y = bs.shuffle_rows(state["x"], seed)
        grad, = torch.autograd.grad(y, state["x"], state["grad"])
        return {"y": y.detach(), "grad": grad}
    if kind == "mc":
        return bs.mc_group_diff(state["x"], case["n1"], seed, case["count"])
    if kind == "shapley":
        return bs.shapley_voting(state["weights"], state["quota"], seed, case["count"])
    ranks = stats.sample_ranks(case["n"], case["count"], seed)
    return {"ranks": ranks, "discordant": stats.kendall_pairs(ranks)}


# ------------------------------------------------------------------ what it takes


def work(case: dict) -> dict:
    """Bytes: every input read once, every output written once.  Operations: one
    evaluation of the bijection per element placed, a round of it being three
    32-bit multiplies, their additions and two logic operations."""
    kind = case["kind"]
    per_eval = 8.0 * ROUNDS
    if kind in ("permute", "inverse"):
        return {"bytes": 2.0 * case["n"] * case["bytes"], "flops": per_eval * case["n"]}
    if kind == "indices":
        return {"bytes": 1.0 * case["n"] * case["bytes"], "flops": per_eval * case["n"]}
    if kind == "batched":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        n = case["count"] * mean
        return {"bytes": 2.0 * n * case["bytes"] + 16.0 * case["count"], "flops": per_eval * n}
    if kind == "rows":
        one = 2.0 * case["rows"] * case["cols"] * torch.empty(0, dtype=_FLOAT[case["dtype"]]).element_size()
        return {"bytes": 2.0 * one, "flops": 2.0 * per_eval * case["rows"]}
    if kind == "mc":
        placed = min(case["n1"], case["n"] - case["n1"])  # the other group's sum is the rest
        return {"bytes": 4.0 * case["n"] + 8.0 * case["count"], "flops": (per_eval + 1.0) * placed * case["count"]}
    if kind == "shapley":  # an order is followed to its pivot, about half of the players
        return {"bytes": 12.0 * case["n"], "flops": (per_eval + 1.0) * case["n"] / 2 * case["count"]}
    n, count = case["n"], case["count"]
    return {"bytes": 8.0 * n * count + 4.0 * count, "flops": (per_eval + math.log2(n)) * n * count}


# ------------------------------------------------------------------ computed numbers in 64 bits


def _round_keys(seed: int) -> list[int]:
    """SplitMix64's outputs, low 32 bits."""
    mask, keys = 2**64 - 1, []
    for r in range(ROUNDS):
        z = (seed + 0x9E3779B97F4A7C15 * (r + 1)) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        keys.append((z ^ (z >> 31)) & 0xFFFFFFFF)
    return keys


def _images(k: int, seeds: list[int]) -> torch.Tensor:
    """f(0), f(1), ... f(2^k - 1) for every seed, as a (len(seeds), 2^k) int64 tensor."""
    lbits = k // 2
    rbits = k - lbits
    keys = torch.tensor([_round_keys(s) for s in seeds], device="cuda")
    i = torch.arange(1 << k, device="cuda").expand(len(seeds), -1)
    left, right = i >> rbits, i & ((1 << rbits) - 1)
    m0 = 0xD2B74407B1CE6E93 - 2**64
    for r in range(ROUNDS):
        prod = left * m0  # modulo 2^64
        hi, lo = (prod >> 32) & 0xFFFFFFFF, prod & 0xFFFFFFFF
        new_left = (hi ^ keys[:, r:r + 1] ^ right) & ((1 << lbits) - 1)
        if rbits > lbits:  # the old right half's top bit comes in underneath
            lo = (lo << 1) | (right >> lbits)
        left, right = new_left, lo & ((1 << rbits) - 1)
    return (left << rbits) | right


def exact(case: dict, seed: int):
    """The statistic of the permutation test; everything else is moved or counted."""
    if case["kind"] != "mc":
        return None
    n, n1, first = case["n"], case["n1"], seed * 7919 + 1
    k = max(4, (n - 1).bit_length())
    x = torch.zeros(1 << k, dtype=torch.float64, device="cuda")
    x[:n] = _samples(case, seed).double()
    total = x.sum()
    out = []
    step = max(1, 2**23 >> k)
    for b in range(0, case["count"], step):
        f = _images(k, [first + t for t in range(b, min(b + step, case["count"]))])
        kept = f < n
        head = kept & (kept.cumsum(1) <= n1)
        s1 = (x[f] * head).sum(1)
        out.append(s1 / n1 - (total - s1) / (n - n1))
    return torch.cat(out)
