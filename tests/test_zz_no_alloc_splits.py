"""The allocation-free Otsu level where its tiles change: heights of 32 and 64
rows, one column cut into many z-chunks, chunks that do not divide Z, and rows
just past a tile; each equal to the level of the regular path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(64, 64, 5000), (33, 20, 3001), (61, 63, 700), (61, 64, 333), (129, 65, 77),
                                  (8, 1, 9001), (1, 33, 40), (700, 32, 203), (1, 1, 1)])
def test_level(dims):
    import torch

    import paper_1407_2089_gb300 as seg
    X, Y, Z = dims
    rng = np.random.default_rng(sum(dims))
    v = rng.normal(300, 30, size=(Z, Y, X))
    v[Z // 3:Z // 3 + max(1, Z // 9)] += 2000
    v[Z - 1, Y - 1, X - 1] = 40000
    v = np.rint(v).clip(0, 65535).astype(np.uint16)
    ctx = seg.seg_create(device=0)
    try:
        (_, _, want), = seg.segment(ctx, v)
    finally:
        seg.seg_destroy(ctx)
    d = torch.from_numpy(v.view(np.int16)).cuda()
    r = torch.full((2,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    seg.seg_otsu_threshold_noalloc(d.data_ptr(), dims, r.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert tuple(int(a) for a in r.cpu()) == (want, 0)
