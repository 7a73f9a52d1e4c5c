"""The sort of large batches where its form is chosen by a sample of the keys: one
key repeated about as often as a window holds, often enough for the sample to
tell, and for half of the batch; tags, which must move stably, at the edges of the
blocks' equal shares; more keys than windows are used for."""
import numpy as np
import pytest
import torch

from paper_2305_05055_gb300 import cpma as cp
from paper_2305_05055_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = np.uint64
EDGE = 1280 * 1024


def handle():
    return cp.CPMA(torch.arange(1, 100, dtype=torch.int64, device="cuda"))


@pytest.mark.parametrize("k", [EDGE + 1, 1_400_000, 3_000_001])
@pytest.mark.parametrize("times", [1_900, 2_047, 2_048, 2_049, 2_600, 3_500, 20_000, 600_000])
def test_one_key_repeated(times, k):
    keys = W.uniform_keys(times, k, bits=40)
    keys[W.splitmix64(3, times) % U(k)] = keys[7]      # scattered (a few fall together)
    g, dk = handle(), torch.from_numpy(keys.view(np.int64)).cuda()
    for _ in range(2):
        out, _ = cp.cpma_sort_batch(g.handle, dk)
    assert np.array_equal(out.cpu().numpy().view(U), np.sort(keys))
    c = cp.CPMA(dk)                                     # the constructor's form of the same sort
    s, n = c.sum()
    want = np.unique(keys)
    assert int(n.item()) == want.size and int(cp.to_u64(s)[0]) == int(want.sum(dtype=U))


@pytest.mark.parametrize("k", [4_097, 4_098, 100_003, EDGE, EDGE + 1, 2_000_003])
@pytest.mark.parametrize("kind", ["uniform", "few", "one", "sorted"])
def test_tags_stay_in_order(kind, k):
    keys = W.uniform_keys(11, k, bits=40)
    if kind == "few":
        keys = keys % U(5) * U(1 << 30)
    elif kind == "one":
        keys[:] = U(9)
    elif kind == "sorted":
        keys = np.sort(keys >> U(12))
    g = handle()
    tags = np.arange(k, dtype=np.int32)
    out, t = cp.cpma_sort_batch(g.handle, torch.from_numpy(keys.view(np.int64)).cuda(),
                                torch.from_numpy(tags).cuda())
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(out.cpu().numpy().view(U), keys[order])
    assert np.array_equal(t.cpu().numpy(), tags[order])


@pytest.mark.parametrize("k", [1700 << 16, (1700 << 16) + 1])
def test_more_keys_than_windows_take(k):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(k)
    x = torch.randint(0, 1 << 40, (k,), dtype=torch.int64, device="cuda", generator=gen)
    g = handle()
    out, _ = cp.cpma_sort_batch(g.handle, x)
    assert torch.equal(out, torch.sort(x).values)
