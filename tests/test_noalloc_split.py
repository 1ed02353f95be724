"""The tile height and z-chunk that seg_otsu_threshold_noalloc picks (host-side
check of the function itself; no GPU): the fullest block of the split never
smooths more, in 32-row planes with the four halo planes of a tile, than with
tiles of 32 rows x 64 planes or of 64 rows in at most 64 chunks, and its tile
indices stay in 32 bits."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "seg_internal.h"
extern "C" void split(unsigned x, unsigned y, unsigned z, unsigned blocks, unsigned *o) {
    const seg::HistSplit s = seg::hist_split(x, y, z, blocks);
    o[0] = s.ty; o[1] = s.tz;
}
"""
MAX_YZ = 2147483583


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "split.cpp").write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1407_2089_gb300", "csrc"), "-I", os.path.join(cuda, "include"),
                    str(d / "split.cpp"), "-o", str(d / "split.so")], check=True)
    lib = ctypes.CDLL(str(d / "split.so"))
    o = (ctypes.c_uint * 2)()

    def f(x, y, z, blocks):
        lib.split(x, y, z, blocks, o)
        return o[0], o[1]
    return f


def up(a, b):
    return -(-a // b)


def cost(x, y, z, blocks, ty, tz):
    tiles = up(x, 64) * up(y, ty) * up(z, tz)
    return up(tiles, blocks) * (tz + 4) * (7 if ty == 64 else 5)


def check(split, x, y, z, blocks):
    ty, tz = split(x, y, z, blocks)
    assert ty in (32, 64) and 1 <= tz <= z
    assert up(x, 64) * up(y, ty) * up(z, tz) < 2 ** 32 and up(z, tz) * tz < 2 ** 32
    c = cost(x, y, z, blocks, ty, tz)
    assert c <= cost(x, y, z, blocks, 32, 64 if z > 64 else z), (x, y, z)
    for n in range(1, min(z, 64) + 1):
        assert c <= cost(x, y, z, blocks, 64, up(z, n)), (x, y, z, n)


@pytest.mark.parametrize("dims", [(64, 64, 20000), (64, 64, 1 << 20), (1, 1, 100000), (1024, 32, 2000), (1024, 65, 512),
                                  (701, 512, 64), (24, 24, 8), (1, 1, 1), (65536, 65535, 1), (1, 1, MAX_YZ),
                                  (1, MAX_YZ, 1), (64, 64, 1048575), (3000, 3000, 400)])
@pytest.mark.parametrize("blocks", [1, 148, 152])
def test_listed(split, dims, blocks):
    check(split, *dims, blocks)


def test_drawn(split):
    rng = random.Random(4)
    for _ in range(300):
        x, y = (int(2 ** rng.uniform(0, 13)) for _ in range(2))
        z = int(2 ** rng.uniform(0, 17))
        if x * y * z < 2 ** 32:
            check(split, x, y, z, 152)
