"""GPU parity of the denoise front end's box passes at every radius, for lines
shorter than the window, lines of one and of several chunks, chunks near a
line's start and end, and a batch of mixed radii."""
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


def noise(dims, seed, top=4000):
    X, Y, Z = dims
    return np.random.default_rng(seed).integers(0, top, size=(Z, Y, X)).astype(np.uint16)


def check(seg, vols, radii):
    ctx = seg.seg_create(device=0, batch_window_us=30_000_000)
    try:
        reqs = [seg.seg_submit_volume(ctx, v, denoise_radius=r) for v, r in zip(vols, radii)]
        seg.seg_flush(ctx)
        for v, r, req in zip(vols, radii, reqs):
            assert seg.seg_wait(ctx, req) == seg.SEG_DONE
            got = np.empty(v.shape, np.uint16)
            seg.seg_read_denoised(ctx, req, 0, got)
            assert np.array_equal(got, oracle.denoise(v, r)), (v.shape, r)
            seg.seg_release(ctx, req)
        assert seg.seg_get_stats(ctx)["batches"] == 1
    finally:
        seg.seg_destroy(ctx)


@pytest.mark.parametrize("r", range(1, 17))
def test_radii(seg, r):
    # lines of one voxel, of about the window, and of more than one chunk
    # along x (128) and y or z (256)
    dims = [(1, 1, 1), (2 * r, 2 * r + 1, 2 * r + 2), (3 * r + 129, 5, 4), (300, 4, 3), (7, 290, 3), (5, 3, 530),
            (129, 130, 3)]
    check(seg, [noise(d, r + sum(d), 65536 if r % 4 == 0 else 4000) for d in dims], [r] * len(dims))


def test_mixed_radii(seg):
    dims = [(150, 20, 9), (40, 270, 5), (33, 9, 40), (260, 6, 6), (17, 17, 17)]
    radii = [1, 5, 16, 8, 4]
    check(seg, [noise(d, sum(d)) for d in dims], radii)
