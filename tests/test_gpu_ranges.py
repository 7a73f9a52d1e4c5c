"""Range queries over byte-code leaves, bit for bit against the plain sorted
set: queries that together cover more leaves than the set has (the leaves are
then reduced once and differenced) and fewer (walked), around that line, over
codes of one to ten bytes, and with leaves that deletions left empty; few
queries (eight lanes per leaf), at least one per leaf (marks inside the leaves)."""
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


def same(got, want, what):
    for a, b in zip(got, want):
        assert np.array_equal(cp.to_u64(a), np.asarray(b, np.uint64)), what


def check(g, p, lo, hi, seed):
    tl, th = T(lo), T(hi)
    same(g.range_map(tl, th), p.range_map(lo, hi), "range_map")
    for op, mask, value in (("sum", 1, 1), ("min", 0, 0), ("min", 7, 5), ("max", 0, 0),
                            ("max", 3, 2), ("xor", 0, 0), ("xor", 15, 9), ("max", 1, 2)):
        same(g.range_reduce(tl, th, op, mask, value), p.range_reduce(lo, hi, op, mask, value),
             (op, mask, value))
    off, out = g.range_extract(tl[:300], th[:300])
    woff, wout = p.range_extract(lo[:300], hi[:300])
    assert np.array_equal(cp.to_u64(off), woff) and np.array_equal(cp.to_u64(out), wout)
    ln = (W.splitmix64(seed, lo.size) % U(3000)).astype(U)
    ln[::7] = 0
    ln[1::11] = U(0xFFFFFFFFFFFFFFFF)
    same(g.range_map_length(tl, T(ln)), p.range_map_length(lo, ln), "length")


@pytest.mark.parametrize("LB", [256, 512, 2048])
@pytest.mark.parametrize("kind", [40, 64, "edges", "dense", "mixed"])
def test_ranges_both_forms(kind, LB):
    base = keys_of(kind, 60_000, 5)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=LB)
    S = p.S
    for q, most in ((1, 60_000), (2, 60_000), (65, 300), (700, 20_000), (2_000, 3), (9_000, 40)):
        lo, hi, _ = W.range_queries_by_rank(S, 31 + q, q, 1, most)
        if q > 4:
            lo[0], hi[0] = 0, 0xFFFFFFFFFFFFFFFF   # everything but the largest key
            hi[1] = lo[1]                           # empty
            lo[2], hi[2] = hi[2], lo[2]             # reversed
            lo[3], hi[3] = S[-1], 0xFFFFFFFFFFFFFFFF
            lo[4], hi[4] = 0, S[0]                  # nothing below the first key
            lo[5::17] += U(1)
        check(g, p, lo, hi, q)


def test_total_at_the_line():
    # q copies of one range: the inner leaves number just below, at and just
    # above the set's leaves
    base = W.uniform_keys(3, 50_000, bits=40)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=256)
    L, S = g.leaves(), p.S
    _, _, heads = g.layout()
    heads = cp.to_u64(heads)
    for inner in (1, 3, L // 2, L - 2):
        lo, hi = heads[0], heads[inner + 1] + U(1)
        for q in {max(2, L // inner - 1), max(2, L // inner), L // inner + 1, L // inner + 2}:
            check(g, p, np.full(q, lo, U), np.full(q, hi, U), q)


@pytest.mark.parametrize("LB", [256, 272, 2048])
@pytest.mark.parametrize("kind", [40, 64, "edges", "mixed"])
def test_a_query_per_leaf_and_more(kind, LB):
    # the leaves are marked from L queries on; some leaves hold nothing
    base = keys_of(kind, 30_000, 8)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=LB, rho_leaf=0, rho_root=1)
    gone = p.S[p.S.size // 4:p.S.size // 2].copy()
    assert int(g.delete_batch(T(gone)).item()) == p.delete_batch(gone)
    L, S = g.leaves(), p.S
    for q in (L - 1, L, 3 * L + 1):
        lo, hi, _ = W.range_queries_by_rank(S, 5 + q, q, 1, 60)
        lo[::5] += U(1)
        hi[::7] -= U(1)
        lo[0], hi[0] = 0, 0xFFFFFFFFFFFFFFFF
        lo[-1], hi[-1] = gone[0], gone[-1]
        tl, th = T(lo), T(hi)
        want = p.range_map(lo, hi)
        same(g.range_map(tl, th), want, (L, q))
        g.set_mem_budget(g.mem_held())               # the memory it holds is enough
        same(g.range_map(tl, th), want, (L, q, "again"))
        g.set_mem_budget(0)
    h = cp.CPMA(T(S), leaf_bytes=LB)
    h.set_mem_budget(h.mem_held() + 64 * q)          # room for the queries, not for the marks
    lo, hi, _ = W.range_queries_by_rank(S, 4, 4 * q, 1, 60)
    same(h.range_map(T(lo[:q]), T(hi[:q])), p.range_map(lo[:q], hi[:q]), "within the budget")
    h.set_mem_budget(0)
    h.reserve(1, 4 * q)
    held = h.mem_held()
    same(h.range_map(T(lo), T(hi)), p.range_map(lo, hi), "reserved")
    assert h.mem_held() == held


def test_empty_leaves_inside():
    base = np.arange(40_000, dtype=U) * U(1000)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=256, rho_leaf=0, rho_root=1)
    gone = base[5_000:35_000]
    assert int(g.delete_batch(T(gone)).item()) == p.delete_batch(gone)
    lo, hi, _ = W.range_queries_by_rank(base, 8, 500, 1, 30_000)
    check(g, p, lo, hi, 1)
    lo, hi, _ = W.range_queries_by_rank(base, 9, 500, 1, 20)
    check(g, p, lo, hi, 2)


@pytest.mark.parametrize("LB,a,b", [(2048, 2, 3), (2048, 1, 7), (256, 1, 7)])
def test_leaves_emptied_by_slices_of_many_keys(LB, a, b):
    # (slices of more keys than one work item holds: the leaf is left pending
    # and rewritten, empty, by the redistribution; no lower density bound)
    base = keys_of("edges", 30_000, 8)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=LB, rho_leaf=0, rho_root=1)
    gone = p.S[p.S.size * a // 8:p.S.size * b // 8].copy()
    assert int(g.delete_batch(T(gone)).item()) == p.delete_batch(gone)
    _, used, heads = g.layout()
    heads, used = cp.to_u64(heads)[:used.numel()], used.cpu().numpy()
    assert (used == 0).sum() > 1
    want = [U(0xFFFFFFFFFFFFFFFF)]           # an empty leaf's head: the next one's
    for h, u in zip(heads[::-1], used[::-1]):
        want.append(h if u else want[-1])
    assert np.array_equal(heads, np.array(want[:0:-1], U))
    assert bool(g.has_batch(T(p.S)).all()) and not bool(g.has_batch(T(gone)).any())
    lo, hi, _ = W.range_queries_by_rank(p.S, 9, 500, 1, 60)
    check(g, p, lo, hi, 2)


def test_without_room_for_the_prefix_and_in_a_capture():
    base = W.uniform_keys(13, 200_000, bits=40)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base))
    lo, hi, _ = W.range_queries_by_rank(p.S, 4, 300, 1, 100_000)
    want = p.range_map(lo, hi)
    tl, th = T(lo), T(hi)
    g.range_map(tl[:1], th[:1])                      # one query: no prefix
    held = g.mem_held()
    g.reserve(1, 300)
    s, c = torch.empty_like(tl), torch.empty_like(tl)
    h = cp.CPMA(T(base))
    h.set_mem_budget(h.mem_held() + 16_000)          # room for the queries, not for the prefix
    same(h.range_map(tl, th), want, "within the budget")
    h.set_mem_budget(0)
    same(h.range_map(tl, th), want, "without one")
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        cp.cpma_range_map(g.handle, tl, th, s, c, stream=st)
    s.zero_()
    c.fill_(7)
    graph.replay()
    torch.cuda.synchronize()
    same((s, c), want, "captured")
    assert g.mem_held() > held


def test_extract_cap():
    base = W.uniform_keys(17, 30_000, bits=40)
    p, g = oracle.PlainSet(base), cp.CPMA(T(base), leaf_bytes=256)
    lo, hi, _ = W.range_queries_by_rank(p.S, 4, 50, 1, 2_000)
    woff, wout = p.range_extract(lo, hi)
    tl, th = T(lo), T(hi)
    total = int(woff[-1])
    for cap in (1, 2, int(woff[7]), int(woff[7]) + 1, total - 1, total, total + 5, (1 << 64) - 1):
        off = torch.empty(51, dtype=torch.int64, device="cuda")
        out = torch.full((total + 8,), 77, dtype=torch.int64, device="cuda")
        rc = cp.lib().cpma_range_extract(g.handle, C.c_void_p(tl.data_ptr()), C.c_void_p(th.data_ptr()),
                                         50, C.c_void_p(off.data_ptr()), C.c_void_p(out.data_ptr()),
                                         C.c_uint64(cap),
                                         C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        n = min(cap, total)
        got = cp.to_u64(out)
        assert np.array_equal(cp.to_u64(off), woff) and np.array_equal(got[:n], wout[:n])
        assert (got[n:] == 77).all()
