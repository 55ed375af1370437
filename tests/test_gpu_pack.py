"""The brick pack against numpy where its pairs and steps can go wrong: bricks one
voxel thick, odd and even extents, rows shorter and longer than a round of the
block's threads, bricks of fewer quads than a block, every storage kind; updates
from device memory included."""
import numpy as np
import pytest

from paper_2501_01628_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


@pytest.mark.parametrize("storage,octets", [("f32", False), ("bf16", False), ("f16", False), ("bf16", True), ("f16", True)])
@pytest.mark.parametrize("shape,part", [
    ((1, 1, 1), dict(kind="grid", grid=(1, 1, 1))),
    ((3, 2, 5), dict(kind="grid", grid=(5, 2, 3))),          # one voxel per brick
    ((7, 12, 131), dict(kind="grid", grid=(1, 1, 1))),       # rows of 66 blocks: more than one round
    ((20, 9, 300), dict(kind="grid", grid=(3, 2, 1))),
    ((33, 34, 35), dict(kind="kd", n_bricks=7, cut_fracs=[0.31, 0.66, 0.5, 0.4, 0.6, 0.5])),
])
def test_packed_bricks_hold_the_haloed_voxels(vr, shape, part, storage, octets):
    import torch
    rng = np.random.default_rng(sum(shape))
    first = rng.standard_normal(shape).astype(np.float32)
    vol = rng.standard_normal(shape).astype(np.float32)
    ctx = vr.vr_create(0)
    v = None
    try:
        vr.vr_set_cell_layout(ctx, 1 if octets else 0)
        v = vr.vr_volume_create(ctx, first, storage, part)
        vr.vr_volume_update(v, torch.from_numpy(vol).cuda())
        boxes, _ = vr.vr_volume_info(v)
        want = vol if storage == "f32" else synth.quantize(vol, storage)
        for b, (x0, y0, z0, x1, y1, z1) in enumerate(boxes):
            ix, iy, iz = (np.clip(np.arange(lo - 1, hi + 1), 0, n - 1)
                          for lo, hi, n in ((x0, x1, shape[2]), (y0, y1, shape[1]), (z0, z1, shape[0])))
            np.testing.assert_array_equal(vr.vr_volume_read_brick(v, b, storage), want[np.ix_(iz, iy, ix)])
    finally:
        if v is not None:
            vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
