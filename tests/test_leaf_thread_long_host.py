"""Host build of the thread-granular leaf insert and delete for leaves with codes
of any length (k_insert_thread_long runs it per leaf) against the oracle's
leaf encoder: the bytes of the union or difference from scratch, the count,
head and changed-key mask; the leaf untouched when the result does not fit."""
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
UNCHANGED, WRITTEN, TOO_BIG = range(3)


@pytest.fixture(scope="module")
def lt(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("ltl") / "libltl.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-o", out,
                    os.path.join(HERE, "leaf_thread_long_host.cu")], check=True)
    return C.CDLL(out)


def enc(keys, LB):
    buf, used = oracle.leaf_encode(np.array(keys, dtype=np.uint64), LB)
    return bytes(buf[:used])


@pytest.mark.parametrize("LB", [256, 512, 2048])
@pytest.mark.parametrize("delete", [False, True])
def test_long_codes(lt, LB, delete):
    rng = random.Random(LB + delete)
    seen = set()
    for it in range(1500):
        mix = rng.choice([[1, 5], [2, 3, 5], [6, 7], [8, 9], [1, 2, 3, 4, 5, 6, 7, 8, 9], [5], [4, 5]])
        keys = [rng.randrange(1 << rng.choice([10, 40, 62]))]
        for _ in range(rng.randint(0, 250)):
            n = rng.choice(mix)
            lo, hi = (1 << (7 * (n - 1))) if n > 1 else 1, (1 << (7 * n)) - 1
            d = rng.choice([lo, hi, rng.randint(lo, hi)])
            if keys[-1] + d > M64:
                break
            keys.append(keys[-1] + d)
        if it % 50 == 0:
            keys = [rng.randrange(9), (1 << 63) + rng.randrange(1 << 62)]  # a 10-byte code
        while oracle.leaf_bytes(np.array(keys, dtype=np.uint64)) > LB - rng.choice([0, 0, 40]):
            keys.pop()
        sl = []
        for _ in range(rng.randint(1, 4)):
            x = rng.choice(keys) + rng.choice([0, 0, 1, -1, rng.randrange(1 << 30)] if delete else
                                              [0, 1, -1, rng.randrange(1 << 30), -rng.randrange(1 << 40)])
            sl.append(min(max(x, 0), M64))
            if rng.random() < 0.2:
                sl[-1] = rng.choice([0, M64, keys[0], keys[-1]])
        if rng.random() < 0.3 and len(keys) > 4:
            i = rng.randrange(len(keys) - 3)
            sl = keys[i:i + len(sl)] if delete else [keys[i] + q for q in range(1, len(sl) + 1)]
        sl = sorted(min(x, M64) for x in sl)
        e = enc(keys, LB)
        leaf = bytearray(LB + 32)
        leaf[:len(e)] = e
        buf = (C.c_uint8 * len(leaf)).from_buffer(leaf)
        out = (C.c_uint32 * 8)()
        st = lt.lt_long(buf, LB, len(e), len(keys), (C.c_uint64 * 4)(*sl), len(sl), out, int(delete))
        old = set(keys)
        new = sorted(old - set(sl)) if delete else sorted(old | set(sl))
        hit = 0
        for q, x in enumerate(sl):
            if (x in old) == delete and (q == 0 or sl[q - 1] != x):
                hit |= 1 << q
        if hit == 0:
            assert st == UNCHANGED and bytes(leaf[:len(e)]) == e
            continue
        nb = oracle.leaf_bytes(np.array(new, dtype=np.uint64)) if new else 0
        assert (out[0], out[1], out[2]) == (nb, len(new), hit)
        if nb > LB:
            assert st == TOO_BIG and bytes(leaf[:len(e)]) == e
            continue
        assert st == WRITTEN
        assert bytes(leaf[:nb]) == (enc(new, LB) if new else b"") and not any(leaf[nb:])
        assert out[3] | (out[4] << 32) == (new[0] if new else M64)
        seen.add((len(sl), nb > len(e)))
    assert len(seen) >= 4
