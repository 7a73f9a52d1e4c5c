"""Host build of a thread's walk over a byte-code leaf (leaf_walk.cuh: the leaf
sums, the partial sums at the ends of ranges, the ranks of range bounds)
against the keys that the oracle's encoder put there: codes of every length
from 1 to 10 bytes, alone and mixed in one leaf, bounds at and beside every
kind of element, every remainder of the used bytes."""
import bisect
import ctypes as C
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

import oracle

HERE = os.path.dirname(os.path.abspath(__file__))
M64 = (1 << 64) - 1


@pytest.fixture(scope="module")
def lw(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("lw") / "liblw.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-o", out,
                    os.path.join(HERE, "leaf_walk_host.cu")], check=True)
    lib = C.CDLL(out)
    u8, u32, u64, p64 = C.c_void_p, C.c_uint32, C.c_uint64, C.POINTER(C.c_uint64)
    lib.lw_sum.restype, lib.lw_sum.argtypes = u64, [u8, u32, u32, C.c_int, u64]
    lib.lw_visit.restype, lib.lw_visit.argtypes = u32, [u8, u32, p64]
    lib.lw_range.argtypes = [u8, u32, u64, u64, p64]
    lib.lw_take.argtypes = [u8, u32, u64, u64, p64]
    lib.lw_below.restype, lib.lw_below.argtypes = u32, [u8, u32, u64]
    lib.lw_has.argtypes = [u8, u32, u64]
    lib.lw_masked.argtypes = [u8, u32, u32, u32, p64]
    lib.lw_team.restype, lib.lw_team.argtypes = u32, [u8, u32, p64]
    lib.lw_between.restype, lib.lw_between.argtypes = u32, [u8, u32, u64, u64, p64]
    lib.lw_from.restype, lib.lw_from.argtypes = u32, [u8, u32, u64, p64]
    lib.lw_marked.argtypes = [u8, u32, u64, p64]
    return lib


def leaves(seed, count, LB):
    """Sorted key lists whose codes have chosen lengths, one byte short of a
    length, exactly at it, or mixed."""
    rng = random.Random(seed)
    for i in range(count):
        kind = i % 6
        v = rng.randrange(1 << rng.choice([8, 40, 63]))
        keys = [v]
        want = rng.randint(1, 300)
        for _ in range(want):
            if kind == 0:
                ln = rng.choice([1, 2, 3])
            elif kind == 1:
                ln = rng.choice([4, 5])
            elif kind == 2:
                ln = 5 if rng.random() < 0.1 else rng.choice([1, 2, 3, 4])
            elif kind == 3:
                ln = rng.choice([6, 7])
            elif kind == 4:
                ln = rng.randint(1, 9)
            else:
                ln = 4
            lo, hi = (1 << (7 * (ln - 1))) if ln > 1 else 1, (1 << (7 * ln)) - 1
            d = rng.choice([lo, hi, rng.randint(lo, hi), rng.randint(lo, hi)])
            if keys[-1] + d > M64:
                break
            keys.append(keys[-1] + d)
        if kind == 4 and keys[0] > 0 and len(keys) > 1 and rng.random() < 0.5:
            keys = [0, (1 << 63) + rng.randrange(1 << 62)]  # a 10-byte code
        while oracle.leaf_bytes(np.array(keys, dtype=np.uint64)) > LB:
            keys = keys[:-1]
        buf, used = oracle.leaf_encode(np.array(keys, dtype=np.uint64), LB)
        leaf = np.zeros(LB + 64, dtype=np.uint8)
        at = -leaf.ctypes.data % 16
        leaf[at:at + LB] = buf[:LB]
        yield keys, leaf[at:], used


def sums(lw, p, u, keys):
    """Every form of the leaf sum that takes this leaf gives the keys' sum; the
    two in 32 bits say so when a code is too long for them."""
    want, m = sum(keys) & M64, len(keys)
    short = all(b - a < 1 << 28 for a, b in zip(keys, keys[1:]))
    few = lw.lw_sum(p, u, m, 2, M64) if m <= 256 else want
    span = keys[-1] - keys[0]   # the least: 2^64 - 1 in this leaf, the next one empty
    return (lw.lw_sum(p, u, m, 0, M64) == lw.lw_sum(p, u, m, 0, span) ==
            lw.lw_sum(p, u, m, 0, span + 1) == want and
            lw.lw_sum(p, u, m, 1, 0) == want and
            (few if short else want) == want and
            lw.lw_sum(p, u, m, 3, 0) == (want if short else M64))


@pytest.mark.parametrize("m", [1, 2, 3, 60, 127, 128, 129, 130, 254, 255, 256, 257, 258, 400, 2040])
def test_leaf_sum_by_number_of_codes(lw, m):
    rng = random.Random(m)
    for ln in (1, 2, 3, 4, 0, -1, -2):
        keys = [rng.randrange(1 << 40)]
        top = {-1: 1 << 14, -2: 1 << 21}.get(ln)   # spans at the edge of two and three planes
        if top and m > 1:
            keys += sorted(keys[0] + d for d in rng.sample(range(1, top - 1), min(m - 2, 250)))
            keys.append(keys[0] + top - 1)
        while len(keys) < m and not top:
            n = ln or rng.choice([1, 1, 1, 2, 3, 4])
            keys.append(keys[-1] + rng.choice([(1 << (7 * n)) - 1, max(1, 1 << (7 * (n - 1)))]))
        while oracle.leaf_bytes(np.array(keys, dtype=np.uint64)) > 2048:
            keys.pop()
        buf, u = oracle.leaf_encode(np.array(keys, dtype=np.uint64), 2048)
        leaf = np.zeros(2048 + 64, dtype=np.uint8)
        at = -leaf.ctypes.data % 16
        leaf[at:at + 2048] = buf[:2048]
        assert sums(lw, leaf[at:].ctypes.data, u, keys)


@pytest.mark.parametrize("d", [1 << 7, 1 << 14, 1 << 21, 1 << 28])
def test_leaf_sum_of_two_elements_a_span_apart(lw, d):
    # the second is 2^64 - 1 and the next leaf empty: its head says d as well
    for gap in (d - 1, d):
        keys = [M64 - gap, M64]
        buf, u = oracle.leaf_encode(np.array(keys, dtype=np.uint64), 256)
        leaf = np.zeros(256 + 64, dtype=np.uint8)
        at = -leaf.ctypes.data % 16
        leaf[at:at + 256] = buf[:256]
        assert lw.lw_sum(leaf[at:].ctypes.data, u, 2, 0, gap) == sum(keys) & M64


@pytest.mark.parametrize("LB", [256, 512, 2048])
def test_walk_against_keys(lw, LB):
    rng = random.Random(LB)
    lengths = set()
    for keys, leaf, u in leaves(LB + 1, 400, LB):
        lengths |= {oracle.leb_len(b - a) for a, b in zip(keys, keys[1:])}
        p = leaf.ctypes.data
        assert sums(lw, p, u, keys)
        out = (C.c_uint64 * (len(keys) + 8))()
        assert lw.lw_visit(p, u, out) == len(keys) and list(out[:len(keys)]) == keys
        assert lw.lw_team(p, u, out) == len(keys) and list(out[:len(keys)]) == keys
        if all(b - a < 1 << 28 for a, b in zip(keys, keys[1:])):
            for mask in (0, 1, 255, 0xFFFFFFFF):
                value = rng.choice(keys) & mask
                got = [x for x in keys if x & mask == value]
                lw.lw_masked(p, u, mask, value, out)
                assert list(out[:2]) == [sum(got) & M64, len(got)]
        marks = [0, M64, keys[0], keys[-1], (keys[-1] + 1) & M64]
        for _ in range(6):
            x = rng.choice(keys)
            marks += [x, (x + 1) & M64, max(x - 1, 0), rng.randrange(keys[0], keys[-1] + 1)]
        res = (C.c_uint64 * 4)()
        for lo in marks:
            a = bisect.bisect_left(keys, lo)
            lw.lw_marked(p, u, lo, res)
            assert list(res) == [sum(keys[:a]) & M64, a, sum(keys) & M64, len(keys)]
            assert lw.lw_below(p, u, lo) == bisect.bisect_left(keys, lo)
            assert lw.lw_has(p, u, lo) == (lo in keys)
            for hi in rng.sample(marks, 6):
                if lo >= hi:
                    continue
                a, b = bisect.bisect_left(keys, lo), bisect.bisect_left(keys, hi)
                lw.lw_range(p, u, lo, hi, res)
                assert (res[0], res[1]) == (sum(keys[a:b]) & M64, b - a)
                n = lw.lw_between(p, u, lo, hi, out)
                assert list(out[:n]) == keys[a:b]
            a = bisect.bisect_left(keys, lo)
            n = lw.lw_from(p, u, lo, out)
            assert list(out[:n]) == (keys[a:] if 0 < a else [])
            for most in (0, 1, 2, rng.randint(0, len(keys)), len(keys) - a, 1 << 40, M64):
                got = keys[a:a + most]
                lw.lw_take(p, u, lo, most, res)
                # the elements below lo matter only where some are taken
                assert (res[1], res[2]) == (len(got), sum(got) & M64)
                assert res[0] == a
    assert lengths >= set(range(1, 8))
