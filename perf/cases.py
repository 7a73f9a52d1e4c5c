"""What a user of this library has it do, as measurable cases.

A case names a set (how its keys are distributed, how many, leaf size) and one
call or a few on it, through the public binding ``paper_2305_05055_gb300.cpma``.
Key distributions are those of the benchmark: keys uniform in [0, 2^bits)
(40-bit keys of the headline, 34-bit ones of the skewed rounds, 64-bit hashes),
batches of zipfian keys, and the edges ``u << 32 | v`` of an R-MAT graph.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_2305_05055_gb300 import cpma as cp

DEV = "cuda"
TOP = -(1 << 63)  # flips the sign bit: unsigned order of keys <-> int64 order
RMAT = (0.57, 0.19, 0.19)  # Graph500 quadrant probabilities
ZIPF_THETA = 0.99


def listed():
    return [
        # a lookup of one page of ids in a small set: latency of one call
        dict(name="has_small", kind="has", dist="uniform", bits=40, n=100_000, q=100, leaf=512),
        # the headline set answering a large membership batch (a join, a filter)
        dict(name="has_large", kind="has", dist="uniform", bits=40, n=100_000_000, q=1_000_000, leaf=512),
        # one pass over everything: App. A sum()
        dict(name="scan", kind="sum", dist="uniform", bits=40, n=100_000_000, leaf=512),
        # the headline range workload: 1e5 ranges of 10 to 1e6 elements each
        dict(name="ranges", kind="range", dist="uniform", bits=40, n=100_000_000, q=100_000, wmin=10,
             wmax=1_000_000, leaf=512),
        # out-degree of every vertex of a graph: many short adjacent ranges
        dict(name="degrees", kind="degrees", dist="graph", scale=20, n=16 << 20, q=1 << 20, leaf=512),
        # neighbour lists of a search frontier, packed
        dict(name="neighbours", kind="neighbours", dist="graph", scale=20, n=16 << 20, q=100_000, leaf=512),
        # ordered scans of a key-value index (hashed 64-bit keys, up to 100 records)
        dict(name="scans_by_length", kind="length", dist="uniform", bits=64, n=10_000_000, q=100_000, wmin=1,
             wmax=100, leaf=512),
        # an aggregate with a predicate over wide ranges (the odd keys, as in the benchmark)
        dict(name="filtered_sums", kind="reduce", dist="uniform", bits=40, n=50_000_000, q=3_001, wmin=10,
             wmax=1_000_000, op="sum", mask=1, value=1, leaf=512),
        # a small sliding-window update of an index: new keys in, expired keys out
        dict(name="window_1e3", kind="window", dist="uniform", bits=40, n=10_000_000, k=1_000, tags=0, leaf=512),
        # the headline update: 1e6 keys into 1e8, and as many expired ones out
        dict(name="window_1e6", kind="window", dist="uniform", bits=40, n=100_000_000, k=1_000_000, tags=0,
             leaf=512),
        # a stream of edges over a graph: power-law batches, keys with long gaps
        dict(name="edge_window", kind="window", dist="graph", scale=20, n=16 << 20, k=100_003, tags=0, leaf=512),
        # bulk load of unsorted keys
        dict(name="build", kind="build", dist="uniform", bits=40, n=30_000_000, leaf=512),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["has", "has", "sum", "range", "range", "degrees", "neighbours", "length", "reduce",
                       "window", "window", "window", "window", "build"])
    leaf = rng.choice([256, 512, 512, 512, 1024, 2048])
    if kind in ("degrees", "neighbours"):
        scale = rng.randint(14, 20)
        return dict(kind=kind, dist="graph", scale=scale, n=16 << scale,
                    q=_log_int(rng, 100, 1 << scale), leaf=leaf)
    bits = rng.choice([34, 40, 40, 64])
    c = dict(kind=kind, dist="uniform", bits=bits, n=_log_int(rng, 100_000, 50_000_000), leaf=leaf)
    if kind == "has":
        c["q"] = _log_int(rng, 1, 1_000_000)
    elif kind in ("range", "length", "reduce"):
        c["q"] = _log_int(rng, 1, 100_000)
        c["wmin"] = _log_int(rng, 1, 100)
        c["wmax"] = c["wmin"] * _log_int(rng, 1, 10_000)
        if kind == "reduce":
            c["op"] = rng.choice(["sum", "min", "max", "xor"])
            c["mask"] = rng.choice([0, 1, 7, 255])
            c["value"] = c["mask"] & rng.randint(0, 255)
    elif kind == "window":
        c["dist"] = rng.choice(["uniform", "uniform", "zipf", "graph"])
        if c["dist"] == "zipf":
            c["bits"] = 34
        elif c["dist"] == "graph":
            del c["bits"]
            c["scale"] = rng.randint(14, 20)
            c["n"] = 16 << c["scale"]
        c["k"] = _log_int(rng, 1, max(1, min(1_000_000, c["n"] // 50)))
        c["tags"] = rng.choice([0, 0, 1, _log_int(rng, 2, 500)])
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, bits):
    if bits == 64:
        return torch.randint(-(1 << 63), (1 << 63) - 1, (n,), dtype=torch.int64, device=DEV, generator=g)
    return torch.randint(0, 1 << bits, (n,), dtype=torch.int64, device=DEV, generator=g)


def _mix34(x):
    """A bijection on [0, 2^34) that scatters the zipfian ranks."""
    m = (1 << 34) - 1
    x = (x * 0x2545F4915) & m
    x = x ^ (x >> 17)
    x = (x * 0x1D8AF0A6B) & m
    return x ^ (x >> 17)


def _zipf(g, n):
    """Zipfian keys (theta 0.99 over 2^34 items): the continuous inverse of the rank distribution."""
    u = torch.rand(n, dtype=torch.float64, device=DEV, generator=g)
    e = 1.0 - ZIPF_THETA
    top = float(1 << 34) ** e
    r = torch.pow(1.0 + u * (top - 1.0), 1.0 / e)
    return _mix34(torch.clamp(r.to(torch.int64) - 1, 0, (1 << 34) - 1))


def _rmat(g, n, scale, perm):
    a, b, c = RMAT
    src = torch.zeros(n, dtype=torch.int64, device=DEV)
    dst = torch.zeros(n, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        u = torch.rand(n, device=DEV, generator=g)
        right = ((u >= a) & (u < a + b)) | (u >= a + b + c)
        src = (src << 1) | (u >= a + b)
        dst = (dst << 1) | right
    return (perm[src] << 32) | perm[dst]


def _keys(case, g, n, batch, perm):
    if case["dist"] == "graph":
        return _rmat(g, n, case["scale"], perm)
    if case["dist"] == "zipf" and batch:
        return _zipf(g, n)
    return _uniform(g, n, case["bits"])


def _perm(case, g):
    return torch.randperm(1 << case["scale"], device=DEV, generator=g) if case["dist"] == "graph" else None


def _sorted_set(keys):
    """The distinct keys in unsigned order, sign bit flipped (so int64 order is theirs)."""
    return torch.unique(keys ^ TOP)


def _neighbours_most(case):
    """Room for the frontier's neighbour lists (four times the mean; keys past it are not written)."""
    return 64 * case["q"] + 65536


def _widths(case, g):
    u = torch.rand(case["q"], dtype=torch.float64, device=DEV, generator=g)
    a, b = math.log(case["wmin"]), math.log(case["wmax"] + 1)
    return torch.clamp(torch.exp(a + (b - a) * u).to(torch.int64), case["wmin"], case["wmax"])


def _inputs(case, seed):
    """The set's keys and the call's arguments."""
    g = _gen(seed)
    perm = _perm(case, g)
    base = _keys(case, g, case["n"], False, perm)
    kind, a = case["kind"], {}
    if kind == "has":  # half of them present
        q = _keys(case, g, case["q"], False, perm)
        at = torch.randint(0, case["n"], (case["q"],), device=DEV, generator=g)
        hit = torch.rand(case["q"], device=DEV, generator=g) < 0.5
        a["keys"] = torch.where(hit, base[at], q)
    elif kind in ("range", "reduce"):
        s = _sorted_set(base)
        r = torch.randint(0, s.numel(), (case["q"],), device=DEV, generator=g)
        w = r + _widths(case, g)
        a["lo"] = s[r] ^ TOP
        a["hi"] = torch.where(w < s.numel(), s[torch.clamp(w, max=s.numel() - 1)] ^ TOP, -1)
    elif kind == "length":
        a["start"] = _keys(case, g, case["q"], False, perm)
        a["length"] = _widths(case, g)
    elif kind in ("degrees", "neighbours"):
        v = torch.randperm(1 << case["scale"], device=DEV, generator=g)[: case["q"]]
        if kind == "degrees":
            v = torch.sort(v).values
        a["lo"], a["hi"] = v << 32, (v + 1) << 32
    elif kind == "window":
        a["batches"] = [_keys(case, g, case["k"], True, perm) for _ in range(2)]
        if case["tags"]:
            a["request"] = torch.randint(0, case["tags"], (case["k"],), dtype=torch.int32, device=DEV, generator=g)
    return base, a


def _leaves_most(case):
    """More leaves than the case's set takes (half full after a build, at least 8 bytes of head each)."""
    kb = 3.5 if case["dist"] == "graph" else _key_bytes(case)
    return int(1.25 * case["n"] * kb / (0.5 * case["leaf"] - 8)) + 64


def _layout_buffers(case):
    """Where a program keeps its copy of the structure (a checkpoint): leaf bytes, used counts, head index."""
    m = _leaves_most(case)
    return dict(data=torch.zeros(m * case["leaf"], dtype=torch.uint8, device=DEV),
                used=torch.zeros(m, dtype=torch.int32, device=DEV),
                heads=torch.zeros(m, dtype=torch.int64, device=DEV))


def _call(name, *args):
    """A function of the C ABI: for callers that keep their own output buffers."""
    args = [C.c_void_p(x.data_ptr()) if torch.is_tensor(x) else x for x in args]
    rc = getattr(cp.lib(), name)(*args, C.c_void_p(torch.cuda.current_stream().cuda_stream))
    if rc != cp.CPMA_OK:
        raise cp.CPMAError(rc, name)


def _export(c, to):
    if c.leaves() > to["used"].numel():
        raise RuntimeError("the layout buffers are too small")
    _call("cpma_export_layout", c.handle, to["data"], to["used"], to["heads"])
    return to


def prepare(case, seed):
    base, a = _inputs(case, seed)
    if case["kind"] in ("build", "window"):
        a["layout"] = _layout_buffers(case)
    if case["kind"] == "build":
        return dict(case=case, keys=base, **a)
    if case["kind"] == "neighbours":
        a["offsets"] = torch.zeros(case["q"] + 1, dtype=torch.int64, device=DEV)
        a["out"] = torch.zeros(_neighbours_most(case), dtype=torch.int64, device=DEV)
    c = cp.CPMA(base, leaf_bytes=case["leaf"])
    if case["kind"] == "window":
        c.reserve(case["k"], tagged=bool(case["tags"]))
        c.use_graphs(1 << 21)
        c.insert_batch(a["batches"][0])
    elif "q" in case:
        c.reserve(1, case["q"])
    return dict(case=case, set=c, at=0, **a)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "build":
        c = cp.CPMA(state["keys"], leaf_bytes=case["leaf"])
        return dict(leaves=c.leaves(), layout=_export(c, state["layout"]))
    c = state["set"]
    if kind == "has":
        return c.has_batch(state["keys"])
    if kind == "sum":
        return c.sum()
    if kind in ("range", "degrees"):
        return c.range_map(state["lo"], state["hi"])
    if kind == "neighbours":
        out = state["out"]
        _call("cpma_range_extract", c.handle, state["lo"], state["hi"], case["q"], state["offsets"], out, out.numel())
        return state["offsets"], out
    if kind == "length":
        return c.range_map_length(state["start"], state["length"])
    if kind == "reduce":
        return c.range_reduce(state["lo"], state["hi"], case["op"], case["mask"], case["value"])
    # the window slides: one batch in, the one before it out, and the set as it is then
    new, old = state["batches"][1 - state["at"]], state["batches"][state["at"]]
    state["at"] = 1 - state["at"]
    if case["tags"]:
        added = cp.cpma_insert_batch_tagged(c.handle, new, state["request"], case["tags"])
        removed = cp.cpma_delete_batch_tagged(c.handle, old, state["request"], case["tags"])
    else:
        added, removed = c.insert_batch(new), c.delete_batch(old)
    return dict(added=added, removed=removed, layout=_export(c, state["layout"]))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _gap(case):
    if case["dist"] == "graph":
        return float(1 << case["scale"]) / 16
    return 2.0 ** case["bits"] / case["n"]


def _key_bytes(case):
    """Mean bytes of a key's code when the gaps are exponential."""
    g = _gap(case)
    return 1.0 + sum(math.exp(-(128.0 ** t) / g) for t in range(1, 10))


def work(case):
    n, kind = case["n"], case["kind"]
    size = n * _key_bytes(case)              # the codes of all keys
    leaves = size / (0.5 * case["leaf"]) + 1  # half full after a build
    array = leaves * (case["leaf"] + 12)      # leaf bytes, used counts and head index
    touched = lambda items: leaves * -math.expm1(-items / leaves)  # noqa: E731
    leaf = size / leaves
    if kind == "has":
        return dict(bytes=9 * case["q"] + touched(case["q"]) * leaf, flops=0)
    if kind == "sum":
        return dict(bytes=size + 4 * leaves + 16, flops=0)
    if kind in ("degrees", "neighbours"):
        share = case["q"] / float(1 << case["scale"])
        out = 16 * case["q"] if kind == "degrees" else 8 * case["q"] + 8 * n * share
        return dict(bytes=16 * case["q"] + size * share + out, flops=0)
    if kind in ("range", "length", "reduce"):
        a, b = case["wmin"], case["wmax"] + 1
        mean = (b - a) / math.log(b / a)
        covered = -math.expm1(-case["q"] * (mean + n / leaves) / n)
        return dict(bytes=32 * case["q"] + size * covered, flops=0)
    if kind == "window":
        k = case["k"]
        tags = 4 * k + 8 * case["tags"] if case["tags"] else 0
        return dict(bytes=2 * (8 * k + tags + 2 * touched(k) * leaf) + 2 * array, flops=0)
    return dict(bytes=8 * n + 3 * array, flops=0)  # keys in, array built, then copied out


# ---------------------------------------------------------------------------
# the same results from sorted arrays
# ---------------------------------------------------------------------------

def _prefix(x):
    return torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(x, 0)])


def exact(case, seed):
    base, a = _inputs(case, seed)
    kind = case["kind"]
    if kind == "build":
        return None  # a layout, not numbers
    s = _sorted_set(base)
    del base
    at = lambda x, of=s: torch.searchsorted(of, x ^ TOP)  # noqa: E731
    below = lambda lo, hi: (lo ^ TOP) < (hi ^ TOP)  # noqa: E731
    if kind == "has":
        i = at(a["keys"])
        return (s[torch.clamp(i, max=s.numel() - 1)] == (a["keys"] ^ TOP)).to(torch.uint8)
    if kind == "sum":
        return (s ^ TOP).sum().reshape(1), torch.tensor([s.numel()], device=DEV)
    if kind in ("range", "degrees", "length", "reduce", "neighbours"):
        if kind == "reduce":
            v = s ^ TOP
            s = s[(v & case["mask"]) == case["value"]]
            del v
        if kind == "length":
            i = at(a["start"])
            j = torch.minimum(i + a["length"], torch.tensor(s.numel(), device=DEV))
        else:
            i, j = at(a["lo"], s), at(a["hi"], s)
            j = torch.where(below(a["lo"], a["hi"]), j, i)
        v = s ^ TOP
        if kind == "neighbours":
            off = _prefix(j - i)
            t = torch.arange(int(off[-1]), device=DEV)
            q = torch.searchsorted(off, t, right=True) - 1
            out = torch.zeros(_neighbours_most(case), dtype=torch.int64, device=DEV)
            out[: t.numel()] = v[i[q] + t - off[q]][: out.numel()]
            return off, out
        op = case.get("op", "sum")
        if op == "sum":
            p = _prefix(v)
            r = p[j] - p[i]
        elif op == "xor":
            p = np.concatenate([[0], np.bitwise_xor.accumulate(v.cpu().numpy())]).astype(np.int64)
            p = torch.from_numpy(p).to(DEV)
            r = p[j] ^ p[i]
        else:
            k = i if op == "min" else j - 1
            r = v[torch.clamp(k, 0, max(v.numel() - 1, 0))] if v.numel() else torch.zeros_like(i)
            r = torch.where(j > i, r, -1 if op == "min" else 0)
        return r, j - i
    # window: S with the first batch in it, then the second in and the first out
    b0, b1 = (torch.unique(b ^ TOP) for b in a["batches"])
    if case["tags"]:
        return None  # the counts are the first occurrences', request by request
    have = torch.unique(torch.cat([s, b0]))
    added = (~torch.isin(b1, have)).sum().reshape(1)
    return dict(added=added, removed=torch.tensor([b0.numel()], device=DEV), layout=None)
