"""GPU parity of the registration sums where their arithmetic or their launches
change: products that fill 32 bits, that leave room for a few rows of a
sub-box and for all, windows wider than the overlap, more pairs than one
group holds, and tiles that barely or no longer touch at some shifts."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def seg():
    import torch
    assert torch.cuda.is_available()
    import paper_1407_2089_gb300 as seg
    return seg


def check(seg, tiles, stage, radius):
    delta, edges = seg.seg_register_montage(tiles, stage, radius)
    wd, we = oracle.register(tiles, stage, radius)
    assert len(edges) == len(we) and len(we)
    for k in ("a", "b", "shift", "in_tree", "score"):
        assert np.array_equal(edges[k], we[k]), (k, edges[k], we[k])
    assert np.array_equal(delta, wd)


@pytest.mark.parametrize("lo,hi", [(65000, 65536), (0, 65536), (0, 9000), (0, 4096), (0, 256), (0, 1)])
def test_value_ranges(seg, lo, hi):
    rng = np.random.default_rng(hi + lo)
    G = rng.integers(lo, hi, size=(20, 70, 100)).astype(np.uint16)
    tiles = [np.ascontiguousarray(G[1:17, 2:60, 0:60]), np.ascontiguousarray(G[0:16, 3:61, 38:98])]
    check(seg, tiles, np.array([[0, 0, 0], [39, 0, 0]]), (3, 2, 2))


@pytest.mark.parametrize("dims,offset,radius", [
    ((40, 30, 12), (37, 0, 0), (5, 2, 1)),     # 3 voxels of overlap, shifts that part the tiles
    ((40, 30, 12), (-38, 27, 11), (6, 6, 3)),
    ((20, 18, 9), (3, -2, 1), (12, 12, 6)),    # the widest window
    ((9, 7, 3), (1, 1, 0), (12, 12, 6)),       # the window wider than the tiles
    ((300, 5, 2), (20, 0, 0), (4, 4, 1)),
    ((5, 300, 3), (0, -280, 1), (1, 7, 2)),
])
def test_overlaps(seg, dims, offset, radius):
    rng = np.random.default_rng(sum(dims))
    tiles = [rng.integers(0, 3000, size=dims[::-1]).astype(np.uint16) for _ in range(2)]
    check(seg, tiles, np.array([[0, 0, 0], offset]), radius)


def test_two_groups(seg):
    # 13 tiles that all overlap: 78 pairs
    rng = np.random.default_rng(5)
    G = rng.integers(0, 3000, size=(12, 60, 60)).astype(np.uint16)
    pos = [np.array([rng.integers(0, 20), rng.integers(0, 20), rng.integers(0, 3)]) for _ in range(13)]
    tiles = [np.ascontiguousarray(G[p[2]:p[2] + 9, p[1]:p[1] + 36, p[0]:p[0] + 36]) for p in pos]
    check(seg, tiles, np.array(pos), (2, 1, 1))
