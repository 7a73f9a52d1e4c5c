"""Leaves that a redistribution leaves empty when the lower density bound is a
few bytes a leaf: the heads of a window's source leaves become codes of a byte or
two, so a destination leaf can fall inside one long code.  Deletes of at most
four keys a leaf, none of which empties its leaf or leaves it pending, until the
oracle's layout has such a leaf; layout, lookups and ranges after each batch."""
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


def clustered(rng, n, p):
    long = rng.random(n) < p                    # gaps of 6 to 8 bytes among short ones
    d = np.where(long, 2.0 ** rng.uniform(36, 52, n), rng.integers(1, 100, n))
    return np.cumsum(d.astype(U))


def thin_out(rng, o):
    """Up to four keys of half the leaves, leaving each at least one."""
    _, used, heads = o.layout()
    E, full = o.elements(), used > 0
    leaf = np.nonzero(full)[0][np.searchsorted(heads[full], E, side="right") - 1]
    gone = []
    for j in np.unique(leaf):
        m = E[leaf == j]
        if rng.random() < .5 or m.size < 3:
            continue
        gone.append(rng.choice(m, min(4, m.size - 1), replace=False))
    return np.concatenate(gone)


def same_layout(g, o, what):
    data, used, heads = g.layout()
    od, ou, oh = o.layout()
    assert np.array_equal(used.cpu().numpy().view(np.uint32), ou), what
    assert np.array_equal(cp.to_u64(heads), oh), what
    assert np.array_equal(data.cpu().numpy(), od), what


@pytest.mark.parametrize("then", ["delete", "insert"])
@pytest.mark.parametrize("rho,p,seed", [(34, .05, 15), (36, .05, 25), (38, .05, 33), (40, .05, 23),
                                        (36, .1, 27)])
def test_leaf_emptied_by_a_sparse_window(rho, p, seed, then):
    rng = np.random.default_rng(seed)
    base = clustered(rng, 3000, p)
    cfg = dict(leaf_bytes=256, rho_leaf=rho, rho_root=rho)
    o, g = oracle.SeqCPMA(base, **cfg), cp.CPMA(T(base), **cfg)
    s = oracle.PlainSet(base)
    empty = 0
    for rnd in range(60):
        gone = thin_out(rng, o)
        assert int(g.delete_batch(T(gone)).item()) == o.delete_batch(gone) == s.delete_batch(gone)
        same_layout(g, o, rnd)
        empty = int((o.layout()[1] == 0).sum())
        if empty:
            break
    assert empty, "no leaf was emptied: the case no longer reaches the rule"
    assert bool(g.has_batch(T(s.S)).all()) and not bool(g.has_batch(T(gone)).any())
    lo, hi, _ = W.range_queries_by_rank(s.S, 9, 200, 1, 200)
    for got, want in zip(g.range_map(T(lo), T(hi)), s.range_map(lo, hi)):
        assert np.array_equal(cp.to_u64(got), want)
    # the next batch starts from the structure with the empty leaf
    if then == "delete":
        more = thin_out(rng, o)
        assert int(g.delete_batch(T(more)).item()) == o.delete_batch(more) == s.delete_batch(more)
    else:
        more = rng.integers(0, int(s.S[-1]), 400).astype(U)
        assert int(g.insert_batch(T(more)).item()) == o.insert_batch(more) == s.insert_batch(more)
    same_layout(g, o, then)
    assert bool(g.has_batch(T(s.S)).all())
