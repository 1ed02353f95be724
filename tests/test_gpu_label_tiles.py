"""GPU parity of labels and cells where the label kernel's tiles meet their
limits: more runs in a tile than it stages at once, coordinate sums of a tile
beyond 32 bits, and label rows at every alignment."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def seg():
    import torch
    assert torch.cuda.is_available()
    import paper_1407_2089_gb300 as seg
    return seg


def stripes(dims, period, keep):
    """Bright stripes along y, `keep` of `period` voxels wide; every third one ends early."""
    X, Y, Z = dims
    v = np.full((Z, Y, X), 100, np.uint16)
    on = np.arange(X) % period < keep
    v[:, :, on] = 30000
    v[:, Y // 2:, on & (np.arange(X) // period % 3 == 0)] = 100
    return v


def bright(dims, cut):
    X, Y, Z = dims
    v = np.full((Z, Y, X), 100, np.uint16)
    v[:, cut:, :] = 30000
    return v


@pytest.mark.parametrize("make,dims,min_volume", [
    (lambda d: stripes(d, 8, 4), (65536, 3, 2), 20),      # 8192 runs in a row
    (lambda d: stripes(d, 8, 4), (9001, 5, 3), 40),       # the same with rows at odd alignments
    (lambda d: bright(d, 7), (65533, 20, 3), 30),         # x sums
    (lambda d: bright(d, 1000), (8, 3_000_000, 1), 30),   # y sums of a tile beyond 2^32
    (lambda d: stripes(d, 40, 21), (130, 67, 5), 30),     # runs across 128-voxel segments
    (lambda d: stripes(d, 300, 200), (701, 31, 4), 30),
])
def test_tiles(seg, make, dims, min_volume):
    vol = make(dims)
    ctx = seg.seg_create(device=0)
    try:
        (lab, cells, thr), = seg.segment(ctx, vol, min_volume=min_volume)
    finally:
        seg.seg_destroy(ctx)
    ref = oracle.segment(vol, min_volume=min_volume)
    assert ref.n_cells
    assert_matches_oracle(vol, lab, cells, thr, ref=ref, what=str(dims))
