"""Updates of large leaves with codes of more than 4 bytes, byte for byte against
the oracle, where they change from a warp per leaf to a thread per leaf and back:
few leaves, many leaves with few keys each, more than four keys a leaf; with and
without graphs, and tagged."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_05055_gb300 import cpma as cp
from paper_2305_05055_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def T(a):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, np.uint64)).view(np.int64)).cuda()


def same_layout(g, o, what):
    data, used, heads = g.layout()
    od, ou, oh = o.layout()
    assert np.array_equal(used.cpu().numpy().view(np.uint32), ou), what
    assert np.array_equal(cp.to_u64(heads), oh), what
    assert np.array_equal(data.cpu().numpy(), od), what


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("LB,n,ks", [(2048, 60_000, (9_000, 12_000)),          # few leaves
                                     (528, 900_000, (20_000, 60_000, 200_000))])  # around the lines
def test_layouts(LB, n, ks, graphs):
    base = W.full_range_keys(81, n)
    g, o = cp.CPMA(T(base), leaf_bytes=LB), oracle.SeqCPMA(base, leaf_bytes=LB)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if LB == 528:
        assert ks[0] > 128 * sms and o.leaves() > 128 * sms and ks[-1] > 4 * o.leaves()
    if graphs:
        g.use_graphs(1 << 20)
    for i, k in enumerate(ks):
        keys = np.concatenate([W.full_range_keys(90 + i, k - k // 4),
                               W.sample_present(oracle.PlainSet(base).S, 91, k // 4)])
        assert int(g.insert_batch(T(keys)).item()) == o.insert_batch(keys)
        same_layout(g, o, ("insert", k))
        assert int(g.delete_batch(T(keys)).item()) == o.delete_batch(keys)
        same_layout(g, o, ("delete", k))
    if not graphs:
        more = W.full_range_keys(99, ks[1])
        counts = torch.zeros(3, dtype=torch.int64, device="cuda")
        tags = torch.arange(more.size, dtype=torch.int32, device="cuda") % 3
        cp.cpma_insert_batch_tagged(g.handle, T(more), tags, 3, counts)
        assert int(counts.sum().item()) == o.insert_batch(more)
        same_layout(g, o, "tagged")


@pytest.mark.parametrize("graphs", [False, True])
def test_some_keys_in_each_leaf(graphs):
    """Leaves of up to four keys, of five and more, and of none, beside each other."""
    test_layouts(1024, 400_000, (9_000, 16_000), graphs)
