"""Cycling frames by the march in pairs (small bricks; octets with the general opacity
formula in all but small launches) and by the one with four samples in flight, with each
opacity correction, against counting frames, which march in pairs with the series'
kernel: bit-identical images."""
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
@pytest.mark.parametrize("n,grid,size", [
    (48, (5, 5, 4), (120, 90)),   # pairs: runs of ten samples
    (60, (1, 2, 1), (120, 90)),   # four in flight
    (60, (1, 2, 1), (301, 293)),  # octets with the general formula: pairs
])
def test_choices_give_one_image(vr, storage, octets, n, grid, size):
    import torch
    rng = np.random.default_rng(n)
    vol = synth.blob_volume(n, synth.draw_blobs(rng, 6))
    lo, hi = float(vol.min()), float(vol.max())
    cam = synth.orbit_camera(*size, 35.0)
    ctx = vr.vr_create(0)
    v = None
    try:
        vr.vr_set_cell_layout(ctx, 1 if octets else 0)
        v = vr.vr_volume_create(ctx, vol, storage, dict(kind="grid", grid=grid))
        vr.vr_set_render_mode(ctx, 1)
        vr.vr_set_camera(ctx, cam)
        for alpha, opc in ((0.1, 0.0), (0.1, 0.7), (0.8, 0.7), (0.1, 0.1)):  # off, series, general (table, ratio)
            vr.vr_set_transfer_function(ctx, synth.random_tf(np.random.default_rng(2), alpha_max=alpha), lo, hi)
            vr.vr_set_opacity_correction(ctx, opc)
            for ert in (1.0, 0.9):
                vr.vr_set_render_params(ctx, 0.5, ert)
                images = []
                for count in (True, False):
                    vr.vr_set_count_samples(ctx, count)
                    out = torch.full((size[1], size[0], 4), float("nan"), device="cuda")
                    vr.vr_render_frame(ctx, v, out)
                    vr.vr_sync(ctx)
                    images.append(out)
                assert torch.equal(images[0], images[1])
                assert float(images[0][..., 3].max()) > 0.02
    finally:
        if v is not None:
            vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
