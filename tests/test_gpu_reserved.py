"""A reservation covers every smaller batch too: the sort's counts per block take
the most room at some key count below the reserved one (as many blocks as run at
once, then fewer with more tiles each), and a reservation for tagged batches
serves untagged ones."""
import numpy as np
import pytest
import torch

from paper_2305_05055_gb300 import cpma as cp
from paper_2305_05055_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def T(a):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, np.uint64)).view(np.int64)).cuda()


@pytest.mark.parametrize("tagged", [False, True])
def test_smaller_batches_take_no_memory(tagged):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = cp.CPMA(T(W.uniform_keys(61, 2_000_000, bits=40)), leaf_bytes=512)
    # one tile of 4096 keys more than 2, 3 or 4 blocks per SM take at once
    for per_sm in (2, 3, 4):
        most = (per_sm * sms + 1) * 4096
        g.reserve(most, tagged=tagged)
        held = g.mem_held()
        for k in (most, most - 4096, most - 4097, most // 2, most // 3, 5000):
            keys = W.uniform_keys(62, k, bits=40)
            cp.cpma_sort_batch(g.handle, T(keys))
            if tagged:
                cp.cpma_sort_batch(g.handle, T(keys), torch.zeros(k, dtype=torch.int32, device="cuda"))
            assert g.mem_held() == held, (per_sm, k)
