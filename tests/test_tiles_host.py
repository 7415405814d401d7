"""The host arithmetic that splits a mesh into the tiles of a persistent launch,
compiled for the CPU: every element in exactly one tile, no tile empty or larger
than a full one, and half of the blocks only where the caller's limit allows it."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1211_0582_gb300", "csrc")
FULLS = (2, 6, 8, 18, 20, 36, 64)
SOURCE = '#include "tiles.cuh"\nusing namespace dgmx;\nextern "C" {\n' + "".join(f"""
int ntiles_{f}(long long K, int grid) {{ return make_tiles<{f}>(K, grid).ntiles; }}
long long start_{f}(long long K, int grid, int t) {{ return make_tiles<{f}>(K, grid).start(t); }}
int size_{f}(long long K, int grid, int t) {{ return make_tiles<{f}>(K, grid).size(t, K); }}
int blocks_{f}(long long K, int cap, int most) {{ return small_mesh_blocks<{f}>(K, cap, most); }}
""" for f in FULLS) + "}\n"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-D__host__=", "-D__device__=", f"-I{CSRC}",
                    str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    lib = ctypes.CDLL(str(d / "t.so"))
    for f in FULLS:
        getattr(lib, f"start_{f}").restype = ctypes.c_longlong
        for name, args in (("ntiles", 0), ("start", 1), ("size", 1), ("blocks", 1)):
            getattr(lib, f"{name}_{f}").argtypes = [ctypes.c_longlong, ctypes.c_int] + [ctypes.c_int] * args
    return lib


@pytest.mark.parametrize("full", FULLS)
@pytest.mark.parametrize("grid", [1, 7, 76, 152, 304])
def test_tiles_partition_the_mesh(lib, full, grid):
    ntiles, start, size = (getattr(lib, f"{n}_{full}") for n in ("ntiles", "start", "size"))
    around = {r * full * grid + d for r in (0, 1, 2) for d in (-1, 0, 1, grid - 1, grid, grid + 1, full * grid // 2)}
    for K in sorted(k for k in around | {1, 2, full, full + 1, grid, 5 * full * grid + 3} if k > 0):
        n = ntiles(K, grid)
        at = 0
        for t in range(n):
            assert start(K, grid, t) == at
            assert 1 <= size(K, grid, t) <= full
            at += size(K, grid, t)
        assert at == K
        # the remainder takes at most one more round of tiles than the full ones
        assert n <= (K // (full * grid) + 1) * grid


@pytest.mark.parametrize("full,cap,most", [(20, 152, 20), (20, 152, 12), (18, 304, 18), (8, 608, 8), (64, 608, 20)])
def test_half_of_the_blocks_up_to_the_limit(lib, full, cap, most):
    blocks = getattr(lib, f"blocks_{full}")
    half = cap // 2
    assert blocks(1, cap, most) == half
    assert blocks(most * half, cap, most) == half
    assert blocks(most * half + 1, cap, most) == cap
    assert blocks(1, 1, most) == 1 and blocks(full, 1, most) == 1
