"""Host build of a leaf's walk by a team of lanes, against the keys that the
oracle's encoder put there: leaves of 8 used bytes to 2048, every remainder of the
16-byte chunks, codes of 1 to 10 bytes (a lane's run starts inside one)."""
import ctypes as C
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

import oracle

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lt(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("lt") / "liblt.so")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-o", out,
                    os.path.join(HERE, "leaf_team_host.cu")], check=True)
    lib = C.CDLL(out)
    lib.lt_team.restype = C.c_uint32
    lib.lt_team.argtypes = [C.c_void_p, C.c_uint32, C.c_int, C.c_int, C.POINTER(C.c_uint64)]
    return lib


@pytest.mark.parametrize("lanes", [8, 16, 32])
@pytest.mark.parametrize("LB", [256, 272, 512, 1024, 2048])
def test_runs_of_a_team(lt, LB, lanes):
    rng = random.Random(LB * 100 + lanes)
    for i in range(300):
        lens = [[1], [1, 2, 3], [4, 5], [6, 7, 8], [9, 10], list(range(1, 11))][i % 6]
        keys, used = [rng.randrange(1 << 20)], 8
        most = rng.choice([8, 9, 24, 25, LB // 2, LB])
        while True:
            n = rng.choice(lens)
            d = rng.randrange(1 << (7 * (n - 1)) if n > 1 else 1, min(1 << (7 * n), 1 << 64))
            if used + n > most or keys[-1] + d >= 1 << 64:
                break
            keys.append(keys[-1] + d)
            used += n
        leaf, u = oracle.leaf_encode(np.array(keys, np.uint64), LB)
        buf = (C.c_uint8 * (LB + 16)).from_buffer_copy(bytes(leaf) + bytes(16))
        out = (C.c_uint64 * (len(keys) + 64))()
        for s in (0, 1):
            assert lt.lt_team(buf, u, lanes, s, out) == len(keys), (u, s)
            assert list(out[:len(keys)]) == keys
