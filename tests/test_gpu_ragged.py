"""GPU parity of volumes whose rows are not whole octets, one batch of many
widths (smoothed rows padded to octets in the label image, or not where that
does not fit), and the same with the smoothed images kept."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_matches_oracle

pytestmark = pytest.mark.gpu

WIDTHS = [1, 2, 3, 4, 5, 6, 7, 9, 10, 11, 13, 14, 18, 22, 33, 66, 250, 509, 514, 701, 1382, 2051, 8190, 8194, 9002]


@pytest.fixture(scope="module")
def seg():
    import torch
    assert torch.cuda.is_available()
    import paper_1407_2089_gb300 as seg
    return seg


def volume(X, seed, top):
    Y, Z = 13, 6
    rng = np.random.default_rng(seed)
    v = rng.normal(200, 20, size=(Z, Y, X))
    for _ in range(3 + X // 60):
        z, y, x = rng.integers(0, [Z, Y, X])
        v[max(0, z - 2):z + 3, max(0, y - 3):y + 4, max(0, x - 3):x + 4] += top
    v[:, : Y // 3, -1:] += top  # reaches the row's end
    return np.rint(v).clip(0, 65535).astype(np.uint16)


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("top", [1500, 30000])
def test_widths(seg, keep, top):
    ctx = seg.seg_create(device=0, batch_window_us=30_000_000, flags=seg.SEG_KEEP_SMOOTHED if keep else 0)
    try:
        vols = [volume(X, 7 * X + top, top) for X in WIDTHS]
        reqs = [seg.seg_submit_volume(ctx, v, min_volume=4) for v in vols]
        seg.seg_flush(ctx)
        for v, req in zip(vols, reqs):
            assert seg.seg_wait(ctx, req) == seg.SEG_DONE
            lab = np.empty(v.shape, np.uint32)
            seg.seg_read_labels(ctx, req, 0, lab)
            cells, thr = seg.seg_read_features(ctx, req, 0)
            assert_matches_oracle(v, lab, cells, thr, min_volume=4, what="X=%d" % v.shape[2])
            if keep:
                got = np.empty(v.shape, np.uint16)
                seg.seg_read_smoothed(ctx, req, 0, got)
                assert np.array_equal(got, oracle.smooth(v)), v.shape
            seg.seg_release(ctx, req)
        assert seg.seg_get_stats(ctx)["batches"] == 1
    finally:
        seg.seg_destroy(ctx)
