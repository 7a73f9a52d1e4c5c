"""The constructor's layout, byte for byte against the oracle, where its passes
over the sorted keys can go wrong: repeats across tiles and leaves, sizes at
the edges of a tile (2048 keys) and of a block's run of tiles, codes of every
length, more keys than the two-pass sort's smallest batch, both codecs."""
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
    assert g.leaves() == o.leaves() and g.size() == o.size() and g.bytes() == o.bytes()
    assert np.array_equal(data.cpu().numpy(), od)
    assert np.array_equal(used.cpu().numpy().view(np.uint32), ou)
    assert np.array_equal(cp.to_u64(heads), oh)
    s, c = g.sum()
    assert int(c.item()) == o.size()
    more = W.uniform_keys(99, 500, bits=40)          # the count and byte total it left
    assert int(g.insert_batch(torch.from_numpy(more.view(np.int64)).cuda()).item()) == \
        o.insert_batch(more)


@pytest.mark.parametrize("codec", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 2047, 2048, 2049, 4095, 4096, 4097, 20_481, 1_310_721])
def test_build_sizes(n, codec):
    same(W.uniform_keys(n, n, bits=40), codec=codec, leaf_bytes=256)


@pytest.mark.parametrize("LB", [256, 512, 2048])
@pytest.mark.parametrize("kind", ["repeats", "runs", "long", "edges", "extremes"])
def test_build_shapes(kind, LB):
    n = 120_000
    if kind == "repeats":
        keys = W.uniform_keys(1, n, bits=14)
    elif kind == "runs":                              # one key fills several tiles
        keys = W.uniform_keys(2, n, bits=40)
        keys[: n // 2] = keys[7]
    elif kind == "long":
        keys = W.full_range_keys(3, n)
    elif kind == "edges":
        src, dst = W.rmat_edges(4, 11, n)
        keys = (src << U(32)) | dst
    else:
        keys = np.concatenate([W.full_range_keys(5, 5_000), np.arange(60_000, dtype=U),
                               np.array([0, 2**64 - 1, 2**63, 2**64 - 1], U)])
    same(keys, leaf_bytes=LB)


@pytest.mark.parametrize("kind", ["uniform", "mixed", "long", "runs"])
def test_build_of_many_leaves(kind):
    # a thread writes each leaf from 256 leaves per SM on; one of more keys
    # than bytes (a run of repeats) is written by a warp
    if kind == "uniform":
        keys = W.uniform_keys(11, 2_600_001, bits=40)
    elif kind == "mixed":   # codes of 1 to 10 bytes, every shift of the 8-byte words
        keys = np.concatenate([W.uniform_keys(12, 1_500_000, bits=24), W.full_range_keys(13, 700_001),
                               W.uniform_keys(14, 600_000, bits=46)])
    elif kind == "long":
        keys = W.full_range_keys(15, 1_000_003)
    else:
        keys = W.uniform_keys(16, 2_700_000, bits=40)
        keys[100_000:103_000] = keys[5]
        keys[200_000:200_200] = keys[6]
    g = cp.CPMA(torch.from_numpy(np.ascontiguousarray(keys).view(np.int64)).cuda(), leaf_bytes=256)
    assert g.leaves() > 256 * torch.cuda.get_device_properties(0).multi_processor_count
    del g
    same(keys, leaf_bytes=256)
