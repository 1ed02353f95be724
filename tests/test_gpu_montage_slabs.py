"""GPU parity of the registration on flat tiles, whose planes are summed in
slabs of rows (the rows every shift shares start or end in any of them), on
deep ones, whose planes are added up by several blocks, and on sub-boxes that
the tile's depth cuts short."""
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


@pytest.mark.parametrize("dims,offset,radius", [
    ((250, 700, 1), (50, 0, 0), (2, 2, 0)),       # four slabs, the shared rows nearly all of them
    ((250, 701, 1), (-40, 350, 0), (3, 6, 0)),    # the shared rows start in a tile's middle
    ((240, 900, 2), (10, -450, 1), (2, 12, 1)),
    ((4000, 70, 1), (270, 3, 0), (4, 12, 1)),     # two slabs
    ((600, 2100, 1), (-5, 0, 0), (1, 1, 0)),      # 32 slabs
    ((40, 130, 1), (30, 125, 0), (4, 8, 0)),      # no row shared by every shift
    ((12, 9, 700), (5, 0, 40), (3, 2, 2)),      # planes in many blocks
    ((4, 5, 14000), (1, 1, 3), (12, 12, 0)),      # more planes than their sums are kept for at once
    ((9, 200, 130), (2, 100, -3), (2, 3, 6)),
    ((50, 40, 17), (30, 3, 0), (3, 2, 2)),      # one plane in the last sub-box
])
def test_shapes(seg, dims, offset, radius):
    rng = np.random.default_rng(sum(dims) + radius[1])
    G = rng.integers(0, 3000, size=[d + abs(o) + 20 for d, o in zip(dims[::-1], offset[::-1])]).astype(np.uint16)
    at = [np.array([max(0, -o) + r for o, r in zip(offset, radius)]), None]
    move = np.array([(r + 1) // 2 for r in radius])  # the second tile's true position, off the stage's
    at[1] = at[0] + np.array(offset) + move
    tiles = [np.ascontiguousarray(G[p[2]:p[2] + dims[2], p[1]:p[1] + dims[1], p[0]:p[0] + dims[0]]) for p in at]
    assert tiles[0].shape == tiles[1].shape == dims[::-1]
    stage = np.array([[0, 0, 0], offset])
    delta, edges = seg.seg_register_montage(tiles, stage, radius)
    wd, we = oracle.register(tiles, stage, radius)
    assert len(edges) == len(we) == 1
    for k in ("a", "b", "shift", "in_tree", "score"):
        assert np.array_equal(edges[k], we[k]), (k, edges[k], we[k])
    assert np.array_equal(delta, wd)
