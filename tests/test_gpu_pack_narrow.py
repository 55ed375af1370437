"""The brick pack where bricks are narrow along x (one quad per thread, by width and
storage) and where a thread's step passes rows and planes at once, against numpy:
widths on both sides of the lines, more and fewer quads than a block writes."""
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


@pytest.mark.parametrize("storage,octets", [("f32", False), ("bf16", False), ("bf16", True), ("f16", True)])
@pytest.mark.parametrize("shape,widths", [
    ((40, 37, 52), (1, 2, 3, 4, 5, 6, 12, 13, 6)),  # narrow and wide bricks in one volume
    ((130, 1, 1), (1,)),                            # one block per plane: planes in steps of 32 and 64
    ((70, 3, 24), (5, 1, 6, 12)),
    ((3, 75, 4), (1, 3)),
])
def test_packed_bricks_hold_the_haloed_voxels(vr, shape, widths, storage, octets):
    import torch
    rng = np.random.default_rng(sum(shape))
    vol = rng.standard_normal(shape).astype(np.float32)
    at = np.concatenate([[0], np.cumsum(widths)])
    assert at[-1] == shape[2]
    part = dict(kind="boxes", boxes=[[x0, 0, 0, x1, shape[1], shape[0]] for x0, x1 in zip(at[:-1], at[1:])])
    ctx = vr.vr_create(0)
    v = None
    try:
        vr.vr_set_cell_layout(ctx, 1 if octets else 0)
        v = vr.vr_volume_create(ctx, torch.from_numpy(vol).cuda(), storage, part)
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
