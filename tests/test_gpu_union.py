"""GPU parity of the component labels where the union kernels' shapes change:
bricks of every height (narrow to wide rows), bricks with more runs than they
stage, several threads per row pair, and components across many brick faces."""
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


def boxes(dims, seed, p):
    """3 x 3 x 3 bright boxes at a fraction p of the voxels: they merge into larger shapes as p grows."""
    X, Y, Z = dims
    hit = np.random.default_rng(seed).random((Z, Y, X)) < p
    on = hit.copy()
    for a in range(3):
        s = on.copy()
        for k in (1, 2):
            moved = np.zeros_like(on)
            src = [slice(None)] * 3
            dst = [slice(None)] * 3
            src[a], dst[a] = slice(None, -k), slice(k, None)
            moved[tuple(dst)] = on[tuple(src)]
            s |= moved
        on = s
    return np.where(on, 40000, 300).astype(np.uint16)


@pytest.mark.parametrize("dims,p", [
    ((66, 100, 40), 0.004),     # 32 x 8-row bricks
    ((300, 70, 20), 0.01),      # 16 x 8
    ((900, 40, 18), 0.01),      # fewer planes, two threads a row pair
    ((2100, 37, 9), 0.01),
    ((9000, 19, 7), 0.004),     # 4 x 2 rows
    ((65536, 9, 4), 0.002),
    ((2000, 33, 17), 0.03),     # bricks past their capacity
    ((128, 65, 30), 0.05),      # one large component
    ((40, 1, 50), 0.02),        # one row a plane
    ((40, 50, 1), 0.02),        # one plane
])
def test_components(seg, dims, p):
    vol = boxes(dims, sum(dims), p)
    ctx = seg.seg_create(device=0)
    try:
        (lab, cells, thr), = seg.segment(ctx, vol, min_volume=10)
    finally:
        seg.seg_destroy(ctx)
    assert_matches_oracle(vol, lab, cells, thr, min_volume=10, what=str(dims))
