"""The constructor over keys with many repeats, byte for byte against the oracle:
more than one in eight (the distinct keys are compacted first) and fewer in one
long run (a leaf's warp searches for the run's end), at either side of that line,
the runs at the ends of the set and inside it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_05055_gb300 import cpma as cp
from paper_2305_05055_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = np.uint64


def same(keys, **cfg):
    g = cp.CPMA(torch.from_numpy(np.ascontiguousarray(keys).view(np.int64)).cuda(), **cfg)
    o = oracle.SeqCPMA(keys, **cfg)
    data, used, heads = g.layout()
    od, ou, oh = o.layout()
    assert g.leaves() == o.leaves() and g.size() == o.size()
    assert np.array_equal(used.cpu().numpy().view(np.uint32), ou)
    assert np.array_equal(cp.to_u64(heads), oh)
    assert np.array_equal(data.cpu().numpy(), od)
    more = W.uniform_keys(99, 500, bits=40)
    assert int(g.insert_batch(torch.from_numpy(more.view(np.int64)).cuda()).item()) == \
        o.insert_batch(more)


@pytest.mark.parametrize("codec", [0, 1])
@pytest.mark.parametrize("where", ["first", "inside", "last", "two"])
@pytest.mark.parametrize("run", [63, 64, 65, 127, 128, 129, 4000, 24_999, 25_001, 40_000])
def test_one_long_run(run, where, codec):
    n = 200_000                                   # 25,000 is one in eight
    rest = np.unique(W.uniform_keys(run, n, bits=40))[1:n - run]
    key = {"first": U(0), "last": U(2**64 - 1)}.get(where, rest[rest.size // 3])
    runs = np.full(run, key, U)
    if where == "two":                            # side by side, one above the other
        runs[run // 2:] = key + U(1)
    same(np.concatenate([rest, runs]), leaf_bytes=512, codec=codec)


@pytest.mark.parametrize("LB", [256, 2048])
@pytest.mark.parametrize("each", [1, 2, 7, 8, 9, 40, 1000])
def test_every_key_repeated(each, LB):
    keys = np.repeat(np.unique(W.uniform_keys(each, 100_000 // each + 2, bits=40)), each)
    same(keys, leaf_bytes=LB)


@pytest.mark.parametrize("n", [2, 4096, 4097, 5000, 300_000, 1_400_000])
def test_all_equal(n):
    same(np.full(n, 12345, U), leaf_bytes=512)


def test_rebuilds_of_a_set_of_repeats():
    base = np.repeat(W.uniform_keys(5, 30_000, bits=40), 5)
    cfg = dict(leaf_bytes=512, rebuild_pm=1)
    g, o = cp.CPMA(torch.from_numpy(base.view(np.int64)).cuda(), **cfg), oracle.SeqCPMA(base, **cfg)
    batch = np.repeat(W.uniform_keys(6, 20_000, bits=40), 3)
    assert int(g.insert_batch(torch.from_numpy(batch.view(np.int64)).cuda()).item()) == \
        o.insert_batch(batch)
    for a, b in zip(g.layout(), o.layout()):
        assert a.cpu().numpy().tobytes() == b.tobytes()
