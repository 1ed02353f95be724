"""GPU parity of the label runs where the way they are read changes: every run
labelled (the records are copied), some dropped (the records are compacted,
more than one block scan per row tile), and a cell table with no room for the
records (two passes over the label image)."""
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


def speckled(dims, seed, p, box):
    """Bright 3 x 3 x 3 boxes at a fraction p of the voxels, and one large box."""
    X, Y, Z = dims
    v = np.full((Z, Y, X), 100, np.uint16)
    for z, y, x in np.argwhere(np.random.default_rng(seed).random((Z, Y, X)) < p):
        v[z:z + 3, y:y + 3, x:x + 3] = 60000
    v[: box[2], : box[1], : box[0]] = 60000
    return v


@pytest.mark.parametrize("dims,p,box,min_volume", [
    ((64, 40, 12), 0.0, (20, 20, 8), 30),       # every run labelled
    ((64, 40, 12), 0.001, (20, 20, 8), 60),     # some dropped
    ((2048, 96, 9), 0.0015, (60, 60, 5), 60),   # several block scans a row tile
    ((41, 300, 7), 0.002, (20, 20, 5), 90),     # several row tiles, odd rows
    ((64, 40, 12), 0.001, (40, 30, 10), 5000),  # no room for the records
    ((33, 40, 12), 0.002, (30, 30, 10), 5000),
])
def test_runs(seg, dims, p, box, min_volume):
    import torch
    vol = speckled(dims, sum(dims), p, box)
    ref = oracle.segment(vol, min_volume=min_volume)
    want = oracle.label_runs(ref.labels)
    assert len(want)
    ctx = seg.seg_create(device=0)
    try:
        req = seg.seg_submit_volume(ctx, vol, min_volume=min_volume)
        seg.seg_flush(ctx)
        assert seg.seg_wait(ctx, req) == seg.SEG_DONE
        cells, _ = seg.seg_read_features(ctx, req, 0)
        assert np.array_equal(cells, ref.cells)
        got = [seg.seg_read_label_runs(ctx, req, 0)]
        for t in (torch.zeros(12 * len(want) + 24, dtype=torch.uint8),
                  torch.zeros(12 * len(want) + 24, dtype=torch.uint8).pin_memory(),
                  torch.zeros(12 * len(want) + 24, dtype=torch.uint8, device="cuda:0")):
            got.append(seg.seg_read_label_runs(ctx, req, 0, t).cpu().numpy().view(seg.LABEL_RUN_DTYPE))
            assert not t[12 * len(want):].any()
        seg.seg_release(ctx, req)
    finally:
        seg.seg_destroy(ctx)
    for g in got:
        assert len(g) == len(want)
        for f in ("label", "row", "x_begin", "x_end"):
            assert np.array_equal(g[f], want[f]), f
