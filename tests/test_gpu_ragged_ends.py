"""GPU parity of ragged x-tiled rows (X > 512, X % 8 != 0) behind a bright
volume of the same batch, whose values the staging ring still holds past the
rows' ends, with values that need the 32-bit y pass nowhere, and in one column
of the last octet only."""
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


@pytest.mark.parametrize("X", [514, 516, 518, 1026, 1030])
def test_last_octet(seg, X):
    rng = np.random.default_rng(X)
    shape = (7, 19, X)
    bright = rng.integers(5000, 65536, size=(9, 40, (X + 7) // 8 * 8)).astype(np.uint16)
    vols = [bright] + [rng.integers(100, 3000, size=shape).astype(np.uint16)]
    for x in range(X // 8 * 8, X):
        v = rng.integers(100, 3000, size=shape).astype(np.uint16)
        v[:, :, x] = rng.integers(60000, 65536, size=shape[:2])
        vols.append(v)
    ctx = seg.seg_create(device=0, batch_window_us=30_000_000)
    try:
        reqs = [seg.seg_submit_volume(ctx, v, min_volume=1) for v in vols]
        seg.seg_flush(ctx)
        for i, (v, req) in enumerate(zip(vols, reqs)):
            assert seg.seg_wait(ctx, req) == seg.SEG_DONE
            lab = np.empty(v.shape, np.uint32)
            seg.seg_read_labels(ctx, req, 0, lab)
            cells, thr = seg.seg_read_features(ctx, req, 0)
            assert_matches_oracle(v, lab, cells, thr, min_volume=1, what="%d of %s" % (i, v.shape))
            seg.seg_release(ctx, req)
        assert seg.seg_get_stats(ctx)["batches"] == 1
    finally:
        seg.seg_destroy(ctx)
