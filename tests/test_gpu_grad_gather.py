"""Voxel gradients gathered from the quads where the gather's chunks of 31 voxels
and sets of 16 rows begin and end, against the oracle's FP64 adjoint: haloed
extents of one less, exactly and one more than a chunk or a set, two of them, and
bricks whose faces are not the volume's."""
import numpy as np
import pytest

import oracle
from paper_2501_01628_gb300 import synth

pytestmark = pytest.mark.gpu

REL = 1e-3  # the adjoint's bar of the differentiation tests, norm-wise


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


@pytest.mark.parametrize("shape,grid", [
    ((6, 13, 28), (1, 1, 1)), ((5, 14, 29), (1, 1, 1)), ((7, 15, 30), (1, 1, 1)),  # 30, 31, 32 by 15, 16, 17
    ((4, 29, 59), (1, 1, 1)), ((3, 30, 60), (1, 1, 1)), ((4, 31, 61), (1, 1, 1)),  # 61, 62, 63 by 31, 32, 33
    ((9, 28, 58), (2, 2, 3)), ((1, 2, 1), (1, 1, 1)),
])
def test_gather_matches_oracle(vr, shape, grid):
    import torch
    rng = np.random.default_rng(sum(shape))
    vol = rng.uniform(0.05, 0.95, shape).astype(np.float32)
    tf = synth.random_tf(rng, alpha_max=0.2)
    part = dict(kind="grid", grid=grid)
    # a view along z: every voxel of the larger faces has several rays
    cam = synth.orbit_camera(150, 120, 10.0, radius=1.3, elevation_deg=12.0,
                             center=tuple(0.5 * np.array(shape[::-1]) / max(shape)))
    G = rng.standard_normal((120, 150, 4)).astype(np.float32)
    ctx = vr.vr_create(0)
    v = None
    try:
        v = vr.vr_volume_create(ctx, vol, "f32", part)
        vr.vr_set_transfer_function(ctx, tf, 0.0, 1.0)
        vr.vr_set_camera(ctx, cam)
        vr.vr_set_render_params(ctx, 0.37, 1.0)
        gtf, gvol = torch.zeros((256, 4), device="cuda"), torch.zeros(shape, device="cuda")
        vr.vr_render_backward(ctx, v, torch.from_numpy(G).cuda(), gtf, gvol)
        vr.vr_sync(ctx)
    finally:
        if v is not None:
            vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
    _, ref = oracle.render_grad(vol, vr.vr_partition_boxes(shape[::-1], part), tf, 0.0, 1.0, cam, G, 0.37)
    assert np.linalg.norm(ref) > 0
    assert np.linalg.norm(gvol.cpu().numpy() - ref) <= REL * np.linalg.norm(ref)
