"""The device memory that a request reserves counts its smoothed image once:
in the kept image, in the label image (ragged rows) or in scratch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,scratch", [((64, 30, 20), True), ((514, 30, 20), False), ((67, 31, 9), False),
                                          ((4, 9, 9), False), ((3, 50, 40), True), ((1, 70, 50), True)])
def test_smoothed_image_is_counted_once(dims, scratch):
    import paper_1407_2089_gb300 as seg
    X, Y, Z = dims
    v = np.random.default_rng(1).integers(0, 3000, size=(Z, Y, X)).astype(np.uint16)
    used = []
    for flags in (0, seg.SEG_KEEP_SMOOTHED):
        ctx = seg.seg_create(device=0, flags=flags, batch_window_us=30_000_000)
        try:
            req = seg.seg_submit_volume(ctx, v)
            used.append(seg.seg_get_stats(ctx)["bytes_in_use"])
            seg.seg_flush(ctx)
            assert seg.seg_wait(ctx, req) == seg.SEG_DONE
            seg.seg_release(ctx, req)
            assert seg.seg_get_stats(ctx)["bytes_in_use"] == 0
        finally:
            seg.seg_destroy(ctx)
    image = (2 * v.size + 255) // 256 * 256
    assert used[1] - used[0] == (0 if scratch else image)
