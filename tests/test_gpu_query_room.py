"""The memory that range queries hold for their own speed (the prefix over the
leaves, the marks inside them) makes room for every other call on the handle:
under a budget in which a call fits on a fresh handle, it fits after a range_map
that took that memory, with the same result."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_05055_gb300 import cpma as cp
from paper_2305_05055_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = np.uint64
N = 60_000


def T(a):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, np.uint64)).view(np.int64)).cuda()


def query_scratch(q):
    """What q range queries hold besides the prefix or the marks (rounded up)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 3 * (8 * (q + 1) + 256) + 8 * (2 * sms + 2) + 256


def merge(g, keys):
    return cp.to_u64(g.insert_batch(T(keys)))


def reserve(g, keys):
    g.reserve(200_000)
    return None


def sort_batch(g, keys):
    return cp.to_u64(cp.cpma_sort_batch(g.handle, T(np.tile(keys, 20)))[0])


def point(g, keys):
    out = cp.to_u64(g.insert_batch(T(keys[:3000])))
    assert g.point_stats() == dict(calls=1, batch=0)
    return out


def profile(g, keys):
    g.profile(True)
    return None


CALLS = dict(merge=(merge, {}, 0), rebuild=(merge, dict(rebuild_pm=1), 0), reserve=(reserve, {}, 0),
             sort_batch=(sort_batch, {}, 0), point=(point, {}, 16384), profile=(profile, {}, 0))


@pytest.mark.parametrize("name", CALLS)
def test_the_queries_memory_makes_room(name):
    call, cfg, point_max = CALLS[name]
    base = W.uniform_keys(41, N, bits=40)
    keys = W.uniform_keys(42, 20_000, bits=40)
    S = oracle.PlainSet(base).S

    def fresh():
        g = cp.CPMA(T(base), leaf_bytes=512, **cfg)
        g.set_point_max(point_max)
        return g

    f = fresh()
    want = call(f, keys)
    g = fresh()
    alone = g.mem_held()
    q = 2 * g.leaves()
    lo, hi, _ = W.range_queries_by_rank(S, 43, q, 1, 50)
    s0 = g.range_map(T(lo), T(hi))
    budget = f.mem_peak() + query_scratch(q)
    assert g.mem_held() - alone > query_scratch(q) + 4096            # it holds the marks
    assert g.mem_held() + f.mem_peak() - alone > budget              # and the call not beside them
    if name == "profile":
        budget = g.mem_held() + 64                                   # 96 bytes are wanted
    g.set_mem_budget(budget)
    got = call(g, keys)
    assert g.mem_peak() <= budget
    assert (got is None) == (want is None)
    if want is not None:
        assert np.array_equal(got, want)
    for a, b in zip(f.layout(), g.layout()):
        assert torch.equal(a, b)
    if name in ("reserve", "sort_batch", "profile"):                 # the set is as it was
        for a, b in zip(g.range_map(T(lo), T(hi)), s0):
            assert torch.equal(a, b)


def test_clone_of_a_set_that_holds_marks():
    # an allocator with room for one more copy of the leaves, and no marks
    base = W.uniform_keys(44, N, bits=40)
    held, room = {}, [1 << 60]

    def alloc(n, stream, ctx):
        if sum(held.values()) + n > room[0]:
            return None
        p = torch.cuda.caching_allocator_alloc(int(n))
        held[p] = int(n)
        return p

    def free(p, stream, ctx):
        held.pop(p)
        torch.cuda.caching_allocator_delete(p)

    a, f = cp.ALLOC_FN(alloc), cp.FREE_FN(free)
    g = cp.CPMA(T(base), leaf_bytes=512, alloc=a, free=f)
    q = 2 * g.leaves()
    lo, hi, _ = W.range_queries_by_rank(oracle.PlainSet(base).S, 45, q, 1, 50)
    want = g.range_map(T(lo), T(hi))
    room[0] = sum(held.values()) + g.bytes() // 2
    c = g.clone()
    for x, y in zip(c.layout(), g.layout()):
        assert torch.equal(x, y)
    for x, y in zip(g.range_map(T(lo), T(hi)), want):
        assert torch.equal(x, y)
    del c, g
    assert not held


def test_a_lower_budget_gives_the_queries_memory_back():
    base = W.uniform_keys(46, N, bits=40)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=512)
    q = 2 * g.leaves()
    lo, hi, _ = W.range_queries_by_rank(p.S, 47, q, 1, 50)
    alone = g.mem_held()
    want = p.range_map(lo, hi)
    for rnd in range(2):
        for got, w in zip(g.range_map(T(lo), T(hi)), want):
            assert np.array_equal(cp.to_u64(got), w)
        held = g.mem_held()
        assert held - alone > query_scratch(q) + 4096
        g.set_mem_budget(held)                   # not below: kept
        assert g.mem_held() == held
        g.set_mem_budget(1)
        assert g.mem_held() - alone <= query_scratch(q)
        g.set_mem_budget(0)


def test_a_query_leaves_half_of_the_free_memory():
    # all but a few MB of the device taken: the marks (some 300 MB) are not
    base = W.uniform_keys(48, 40_000_000, bits=40)
    g = cp.CPMA(T(base), leaf_bytes=512)
    L = g.leaves()
    lo = torch.arange(L + 1, dtype=torch.int64, device="cuda") << 18
    hi = lo + (1 << 20)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    marks = L * 512
    free = torch.cuda.mem_get_info()[0]
    taken = torch.empty(free - marks - marks // 2, dtype=torch.uint8, device="cuda")
    before = g.mem_held()
    want = g.range_map(lo, hi)
    assert g.mem_held() - before < marks // 2
    del taken
    torch.cuda.empty_cache()
    got = g.range_map(lo, hi)
    assert g.mem_held() - before > marks
    for a, b in zip(got, want):
        assert torch.equal(a, b)
