"""GPU parity of the denoise front end's box passes in batches large enough for
the register rings (each axis and radius class, rows of whole octets and
ragged ones, lines of one and of several chunks), and of a batch whose volumes
take different routes."""
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


def check(seg, dims, radii):
    vols = [np.random.default_rng(sum(d) + r).integers(0, 65536 if r % 4 == 0 else 4000, size=d[::-1]).astype(np.uint16)
            for d, r in zip(dims, radii)]
    ctx = seg.seg_create(device=0, batch_window_us=30_000_000)
    try:
        reqs = [seg.seg_submit_volume(ctx, v, denoise_radius=r, min_volume=1000) for v, r in zip(vols, radii)]
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
@pytest.mark.parametrize("dims", [(301, 300, 50), (2048, 40, 32)])
def test_lines(seg, dims, r):
    # y and z rings: ragged rows at every radius (y from 3), octets at 3..8
    # (z from 1, and up to 12 for so few planes)
    check(seg, [dims], [r])


@pytest.mark.parametrize("dims,r", [((50, 300, 200), 1), ((50, 300, 200), 5), ((50, 300, 200), 8),
                                    ((200, 800, 200), 1), ((200, 800, 200), 4), ((128, 800, 390), 8),
                                    ((901, 300, 60), 1)])
def test_rows(seg, dims, r):
    check(seg, [dims], [r])


def test_mixed(seg):
    dims = [(301, 300, 50), (2048, 40, 32), (64, 64, 12), (1, 40, 9), (7, 5, 300), (640, 64, 33), (63, 1, 20)]
    check(seg, dims, [12, 5, 16, 1, 3, 9, 8])
