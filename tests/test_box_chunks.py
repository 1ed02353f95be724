"""How the denoise front end's box passes cut a line along y or z into chunks (host-side
check of the functions the kernels use; no GPU): every position is output
once, with 3 r positions or the line's start before it, and no position that a
chunk names leaves a signed 32-bit integer, for lines up to the longest."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1407_2089_gb300", "csrc")
MAX_YZ = 2147483583

SRC = """
#include "seg_internal.h"
extern "C" unsigned chunks(unsigned n, unsigned len) { return seg::box_chunks(n, len); }
extern "C" void chunk(unsigned n, unsigned len, unsigned k, unsigned r, long long *o) {
    const seg::BoxChunk c = seg::box_chunk(n, len, k, r);
    o[0] = c.first; o[1] = c.n; o[2] = c.c0; o[3] = c.c1; o[4] = c.start;
}
extern "C" unsigned length() { return seg::DN_CHUNK; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("box")
    (d / "box.cpp").write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I",
                    os.path.join(cuda, "include"), str(d / "box.cpp"), "-o", str(d / "box.so")], check=True)
    return ctypes.CDLL(str(d / "box.so"))


@pytest.mark.parametrize("r", [1, 8, 16])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256, 257, 300, 511, 513, 1000, 65535, 65536,
                               MAX_YZ - 300, MAX_YZ - 256, MAX_YZ - 200, MAX_YZ - 1, MAX_YZ])
def test_chunks(lib, n, r):
    length = lib.length()
    nc = lib.chunks(n, length)
    assert nc == -(-n // length)
    o = (ctypes.c_longlong * 5)()
    ks = range(nc) if nc < 2000 else list(range(40)) + list(range(nc - 40, nc))
    at = None  # end of the previous chunk's outputs
    for k in ks:
        lib.chunk(n, length, k, r, o)
        first, left, c0, c1, start = list(o)
        if c0 >= c1:  # equal chunks may end the line before the last one
            assert at == n
            continue
        begin, end = first + c0, first + c1
        if k == 0 or k - 1 in ks:
            assert begin == (at or 0)
        at = end
        assert c1 - c0 <= length and end <= n and first + left == n
        assert c0 == min(begin, 3 * r) and bool(start) == (first == 0)
        assert 0 <= c0 and c1 + 6 * r + 64 < 2 ** 31 and 0 < left < 2 ** 31
    assert at == n


def test_total_outputs(lib):
    o = (ctypes.c_longlong * 5)()
    for n in (1, 100, 256, 257, 767, 5530):
        seen = []
        for k in range(lib.chunks(n, 256)):
            lib.chunk(n, 256, k, 5, o)
            seen += list(range(o[0] + o[2], o[0] + o[3]))
        assert seen == list(range(n))
