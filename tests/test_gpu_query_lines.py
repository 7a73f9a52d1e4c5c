"""Queries at the counts where their form changes -- a warp, eight lanes or a
thread per leaf, a block of 64 or 256 threads, the offsets' scan in the ends'
kernel or on its own, warps or threads for extraction, marks or not -- bit for bit
against the plain sorted set, with queries that end in their first leaf, in the
next one and far away.  Full sums and the prefix over the leaves by eight lanes and
by one."""
import ctypes as C

import numpy as np
import pytest
import torch

import oracle
from paper_2305_05055_gb300 import cpma as cp
from paper_2305_05055_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = np.uint64


def T(a):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, np.uint64)).view(np.int64)).cuda()


def keys_of(kind, n, seed):
    if kind == "edges":
        src, dst = W.rmat_edges(seed, 12, n)
        return (src << U(32)) | dst
    if kind == "dense":
        return W.uniform_keys(seed, n, bits=18)
    if kind == "mixed":  # clusters of one-byte gaps, 64 bits apart
        return (W.full_range_keys(seed, n // 64 + 1)[:, None] + np.arange(64, dtype=U) * U(3)).ravel()
    return W.uniform_keys(seed, n, bits=kind)


def counts(LB):
    """Just below and above the lines, per SM, and the fixed ones."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per = [64, 96, 160, 256] if LB <= 512 else [24, 64, 160, 256]
    return [1, 2, 1024, 1025] + [sms * p + d for p in per for d in (0, 1)]


def queries(S, q):
    lo, hi, _ = W.range_queries_by_rank(S, 31 + q, q, 1, 40)
    wide = slice(None, None, 97)
    lo[wide], hi[wide], _ = W.range_queries_by_rank(S, 37 + q, lo[wide].size, 100, 3_000)
    if q > 8:
        lo[1], hi[1] = 0, 0xFFFFFFFFFFFFFFFF   # everything but the largest key
        hi[2] = lo[2]                           # empty
        lo[3], hi[3] = hi[3], lo[3]             # reversed
        lo[4], hi[4] = S[-1], 0xFFFFFFFFFFFFFFFF
        lo[5], hi[5] = 0, S[0]                  # nothing below the first key
        lo[6::17] += U(1)
    return lo, hi


def same(got, want, what):
    for a, b in zip(got, want):
        assert np.array_equal(cp.to_u64(a), np.asarray(b, np.uint64)), what


@pytest.mark.parametrize("LB", [256, 512, 1024, 2048])
@pytest.mark.parametrize("kind", [40, 64, "edges", "mixed"])
def test_at_the_lines(kind, LB):
    base = keys_of(kind, 60_000, 5)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=LB)
    for q in counts(LB):
        lo, hi = queries(p.S, q)
        tl, th = T(lo), T(hi)
        want = p.range_map(lo, hi)
        same(g.range_map(tl, th), want, ("range_map", q))
        s, c = torch.empty_like(tl), torch.empty_like(tl)
        cp.cpma_range_map_noalloc(g.handle, tl, th, s, c)   # neither prefix nor marks
        same((s, c), want, ("noalloc", q))
        for op, mask, value in (("sum", 1, 1), ("min", 7, 5), ("max", 3, 2), ("xor", 15, 9)):
            same(g.range_reduce(tl, th, op, mask, value), p.range_reduce(lo, hi, op, mask, value),
                 (op, q))
        ln = (W.splitmix64(q, q) % U(60)).astype(U)
        ln[::7] = 0
        ln[1::101] = U(5000)
        ln[-1] = U(0xFFFFFFFFFFFFFFFF)
        same(g.range_map_length(tl, T(ln)), p.range_map_length(lo, ln), ("length", q))


@pytest.mark.parametrize("LB", [256, 512, 1024, 2048])
@pytest.mark.parametrize("kind", [40, "edges", "mixed"])
def test_extraction_at_its_line(kind, LB):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    base = keys_of(kind, 60_000, 6)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=LB)
    for q in (1, 3, sms * LB // 128, sms * LB // 128 + 1):
        lo, hi = queries(p.S, q)
        lo[1::97], hi[1::97] = lo[0], hi[0]      # not everything, many times
        woff, wout = p.range_extract(lo, hi)
        off, out = g.range_extract(T(lo), T(hi))
        assert np.array_equal(cp.to_u64(off), woff) and np.array_equal(cp.to_u64(out), wout)
        for cap in {1, int(woff[-1]) // 2, int(woff[-1])} - {0}:
            off = torch.empty(q + 1, dtype=torch.int64, device="cuda")
            out = torch.full((wout.size + 8,), 77, dtype=torch.int64, device="cuda")
            tl, th = T(lo), T(hi)
            assert 0 == cp.lib().cpma_range_extract(
                g.handle, C.c_void_p(tl.data_ptr()), C.c_void_p(th.data_ptr()), q,
                C.c_void_p(off.data_ptr()), C.c_void_p(out.data_ptr()), C.c_uint64(cap),
                C.c_void_p(torch.cuda.current_stream().cuda_stream))
            got, n = cp.to_u64(out), min(cap, wout.size)
            assert np.array_equal(cp.to_u64(off), woff)
            assert np.array_equal(got[:n], wout[:n]) and (got[n:] == 77).all()


@pytest.mark.parametrize("LB", [256, 272, 512, 528, 1024, 2048])
@pytest.mark.parametrize("kind", [40, 64, "edges", "dense", "mixed"])
def test_sums_and_prefix_of_few_leaves(kind, LB):
    base = keys_of(kind, 90_000, 7)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=LB, rho_leaf=0, rho_root=1)
    for _ in range(2):                           # the second time with empty leaves
        s, c = g.sum()
        assert int(cp.to_u64(s)[0]) == p.sum() and int(c.item()) == len(p)
        lo, hi, _ = W.range_queries_by_rank(p.S, 8, 200, 1000, 60_000)   # more than the set's leaves
        tl, th = T(lo), T(hi)
        same(g.range_map(tl, th), p.range_map(lo, hi), "range_map")
        for op, mask, value in (("sum", 1, 0), ("min", 31, 5), ("max", 31, 2), ("xor", 3, 1)):
            same(g.range_reduce(tl, th, op, mask, value), p.range_reduce(lo, hi, op, mask, value), op)
        gone = p.S[p.S.size // 4:p.S.size // 2].copy()
        assert int(g.delete_batch(T(gone)).item()) == p.delete_batch(gone)


@pytest.mark.parametrize("LB,n", [(256, 1_500_000), (512, 2_400_000), (2048, 24_000_000)])
def test_sums_around_the_line_of_many_leaves(LB, n):
    # leaves of 40-bit keys at either side of what takes eight lanes each
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    line = sms * 256 * (2 if LB > 512 else 1)
    seen = set()
    for m in (n, n * 2 if LB < 2048 else n):
        base = W.uniform_keys(9, m, bits=40)
        g = cp.CPMA(T(base), leaf_bytes=LB)
        seen.add(g.leaves() <= line)
        s, c = g.sum()
        want = np.unique(base)
        assert int(c.item()) == want.size and int(cp.to_u64(s)[0]) == int(want.sum(dtype=U))
    assert LB == 2048 or seen == {True, False}, seen
