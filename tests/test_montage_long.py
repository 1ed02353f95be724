"""Registration of tiles whose extent nears the limits of 32-bit positions."""
import ctypes

import numpy as np
import pytest


def test_extent_limit_without_cuda():
    # refused by the argument checks, before any CUDA call
    import paper_1407_2089_gb300 as seg
    for dims in [(seg.SEG_MAX_YZ + 1, 1, 1), (1, 2 ** 31 - 1, 1), (1, 1, 2 ** 31)]:
        ptrs = (ctypes.c_void_p * 2)(4096, 4096)
        st = (seg.seg_offset * 2)()
        delta = (seg.seg_offset * 2)()
        edges = np.zeros(1, dtype=seg.MONTAGE_EDGE_DTYPE)
        n = ctypes.c_uint32()
        rc = seg._lib.seg_register_montage(0, ptrs, 1, 2, seg.seg_dims(*dims), st, seg.seg_offset(1, 0, 0), 0, delta,
                                           ctypes.c_void_p(edges.ctypes.data), 1, ctypes.byref(n))
        assert rc == seg.SEG_ETOOBIG, dims


@pytest.mark.gpu
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("sign", [1, -1])
def test_offset_beyond_half_of_the_range(axis, sign):
    # two lines of 2^30 + 3000 voxels that share their ends: tile position
    # plus extent is past 2^31; scored as the shared ends alone
    import torch

    import paper_1407_2089_gb300 as seg
    D, share, pad, r, true = 2 ** 30 + 3000, 900, 40, 3, 2
    rng = np.random.default_rng(axis)
    line = rng.integers(0, 3000, size=share + 2 * pad).astype(np.int16)
    lo = torch.full((D,), 7, dtype=torch.int16, device="cuda")  # its end lies in the shared part
    hi = torch.full((D,), 7, dtype=torch.int16, device="cuda")  # its start does
    n = share + pad
    lo[-n:] = torch.from_numpy(line[:n]).cuda()
    hi[:n] = torch.from_numpy(line[pad + true:pad + true + n].copy() if pad + true + n <= len(line) else
                              np.concatenate([line[pad + true:], np.full(pad + true + n - len(line), 7, np.int16)])).cuda()
    shape = [1, 1, 1]
    shape[2 - axis] = D
    tiles = [lo.view(shape), hi.view(shape)]
    stage = np.zeros((2, 3), np.int64)
    stage[1, axis] = D - n + pad
    if sign < 0:
        tiles.reverse()
        stage[:, axis] = stage[::-1, axis].copy()
    radius = [0, 0, 0]
    radius[axis] = r
    torch.cuda.synchronize()
    delta, edges = seg.seg_register_montage(tiles, stage, radius)
    # the same with short tiles that hold the shared ends
    m = n + r + 5
    short = [lo[-m:].cpu().numpy().view(np.uint16), hi[:m].cpu().numpy().view(np.uint16)]
    shape[2 - axis] = m
    short = [np.ascontiguousarray(t.reshape(shape)) for t in short]
    st = np.zeros((2, 3), np.int64)
    st[1, axis] = m - n + pad
    if sign < 0:
        short.reverse()
        st[:, axis] = st[::-1, axis].copy()
    import oracle
    wd, we = oracle.register(short, st, radius)
    assert we["score"][0] > 0.9 and abs(int(we["shift"][0][axis])) == true
    for k in ("shift", "score", "in_tree"):
        assert np.array_equal(edges[k], we[k]), (k, edges[k], we[k])
    assert np.array_equal(delta, wd)
