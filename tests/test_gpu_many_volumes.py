"""GPU parity of one batch of more volumes than the kernels index in shared
memory (512) and than the union's pair cache tags (1024): tiny volumes with
components across brick faces, some of them empty."""
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


def volume(i):
    rng = np.random.default_rng(i)
    if i % 7 == 0:
        return np.full((3, 4, 1 + i % 40), 300, np.uint16)  # no foreground
    X, Y, Z = int(rng.integers(1, 45)), int(rng.integers(30, 40)), int(rng.integers(7, 12))
    v = np.full((Z, Y, X), 200.0)
    for _ in range(int(rng.integers(1, 7))):  # bars along x, y or z, which meet at random
        z, y, x = rng.integers(0, [Z, Y, X])
        a = int(rng.integers(0, 3))
        v[slice(None) if a == 0 else slice(z, z + 2), slice(None) if a == 1 else slice(y, y + 2),
          slice(None) if a == 2 else slice(x, x + 2)] = 3000
    return np.rint(v + rng.normal(0, 10, v.shape)).clip(0, 65535).astype(np.uint16)


def test_one_batch(seg):
    n = 1100
    vols = [volume(i) for i in range(n)]
    ctx = seg.seg_create(device=0, max_batch_volumes=1200, batch_window_us=60_000_000)
    try:
        reqs = [seg.seg_submit_volume(ctx, v, min_volume=2) for v in vols]
        seg.seg_flush(ctx)
        for i, (v, req) in enumerate(zip(vols, reqs)):
            assert seg.seg_wait(ctx, req) == seg.SEG_DONE, i
            lab = np.empty(v.shape, np.uint32)
            seg.seg_read_labels(ctx, req, 0, lab)
            cells, thr = seg.seg_read_features(ctx, req, 0)
            assert_matches_oracle(v, lab, cells, thr, min_volume=2, what="volume %d %s" % (i, v.shape))
            runs = seg.seg_read_label_runs(ctx, req, 0)
            assert runs.tobytes() == oracle.label_runs(lab).tobytes(), i
            seg.seg_release(ctx, req)
        assert seg.seg_get_stats(ctx)["batches"] == 1
    finally:
        seg.seg_destroy(ctx)
