"""The sort of keys alone (cpma_sort_batch without tags) at the sizes and key
shapes where its form changes: 256 buckets up to 1.25M keys, the top 16
varying bits and windows above, the passes over all digits when a window does
not hold its buckets or when at most 24 bits vary; bins in a block, and digit
passes where a bin is deep."""
import numpy as np
import pytest
import torch

from paper_2305_05055_gb300 import cpma as cp
from paper_2305_05055_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = np.uint64
EDGE = 1280 * 1024  # the largest batch that goes by 256 buckets


def shaped(kind, k, seed):
    x = W.full_range_keys(seed, k)
    if isinstance(kind, int):                    # that many random low bits
        return x >> U(64 - kind)
    if kind == "top":                            # only high bits vary
        return (x >> U(40)) << U(40)
    if kind == "edges":                          # skewed high part, random low part
        return ((x & U(1023)) * ((x >> U(10)) & U(1023)) << U(32)) | (x >> U(44))
    if kind == "repeats":                        # 1000 copies of every key
        return np.arange(k, dtype=U) // U(1000) * U(7919)
    if kind == "one":
        return np.full(k, 77, U)
    if kind == "reversed":
        return np.arange(k, 0, -1, dtype=U) * U(1000)
    if kind == "run":                            # one value fills whole windows
        x = x >> U(14)
        x[: min(k, 13_000)] = U(123456789)
        return x
    assert kind == "clusters"                    # a few deep bins in every block
    return ((x >> U(50)) << U(44)) | (x & U(15))


@pytest.mark.parametrize("k", [4_097, 6_145, 100_001, EDGE, EDGE + 1, 1_400_000])
@pytest.mark.parametrize("kind", [5, 24, 25, 34, 40, 64, "top", "edges", "repeats", "one", "reversed",
                                  "run", "clusters"])
def test_sort_forms(kind, k):
    keys = shaped(kind, k, 100 + k % 97)
    g = cp.CPMA(torch.arange(1, 100, dtype=torch.int64, device="cuda"))
    dk = torch.from_numpy(keys.view(np.int64)).cuda()
    for _ in range(2):                           # the second on used scratch
        out, _ = cp.cpma_sort_batch(g.handle, dk)
    assert np.array_equal(out.cpu().numpy().view(U), np.sort(keys))


def test_large_insert_after_a_full_window():
    # an update whose batch is large enough for windows and skewed enough that
    # they give up: the set is the plain one
    import oracle
    base = W.uniform_keys(5, 100_000, bits=40)
    batch = np.concatenate([W.uniform_keys(6, 1_000_000, bits=30) + U(1 << 39),
                            W.uniform_keys(7, 400_000, bits=40)])
    p = oracle.PlainSet(base)
    g = cp.CPMA(torch.from_numpy(base.view(np.int64)).cuda())
    added = g.insert_batch(torch.from_numpy(batch.view(np.int64)).cuda())
    assert int(added.item()) == p.insert_batch(batch) and g.size() == len(p)
    s, c = g.sum()
    assert int(cp.to_u64(s)[0]) == p.sum() and int(c.item()) == len(p)
