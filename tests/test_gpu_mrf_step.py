"""GPU parity of the MRF step kernel where its paths meet: octets aligned to
16, 4 and 2 bytes, rows that share a warp, z ranges split between blocks, the
step at which the byte arithmetic of Delta = 1 ends, and Delta > 1."""
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


def noise(dims, seed, sigma, scale=1, mean=400.0):
    X, Y, Z = dims
    v = np.random.default_rng(seed).normal(mean, sigma, size=(Z, Y, X))
    return (np.rint(v).clip(0, 65535 // scale) * scale).astype(np.uint16)


@pytest.mark.parametrize("dims,iters,sigma,scale,mean", [
    ((264, 5, 40), 6, 25.0, 1, 400.0),     # 16-byte octets, 33 of a row: rows cross warps and tiles
    ((258, 7, 33), 6, 25.0, 1, 400.0),     # 4-byte octets, a last octet of two voxels
    ((41, 30, 9), 6, 25.0, 1, 400.0),      # 2-byte octets, a last octet of one voxel
    ((8, 3, 700), 6, 25.0, 1, 400.0),      # three octets a plane: the blocks split z
    ((24, 40, 1), 6, 25.0, 1, 400.0),      # one plane
    ((40, 24, 10), 150, 80.0, 1, 400.0),   # past step 127
    ((22, 24, 10), 150, 80.0, 1, 400.0),
    ((48, 24, 10), 30, 25.0, 3, 100.0),    # Delta = 3, values down to 0
    ((23, 24, 10), 30, 25.0, 700, 60.0),   # Delta = 700, values up to 65535
    ((32, 24, 10), 12, 2.0, 1, 0.0),       # many zeros: no vote below 0
])
def test_step_paths(seg, dims, iters, sigma, scale, mean):
    vol = noise(dims, sum(dims), sigma, scale, mean)
    ctx = seg.seg_create(device=0)
    try:
        req = seg.seg_submit_volume(ctx, vol, mrf_iterations=iters)
        seg.seg_flush(ctx)
        assert seg.seg_wait(ctx, req) == seg.SEG_DONE
        got = np.empty(vol.shape, np.uint16)
        steps = seg.seg_read_denoised(ctx, req, 0, got)
        seg.seg_release(ctx, req)
    finally:
        seg.seg_destroy(ctx)
    want, wsteps = oracle.mrf(vol, iters)
    assert steps == wsteps
    assert np.array_equal(got, want)
