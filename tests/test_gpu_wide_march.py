"""The march with several samples of a ray in flight (small launches and cycling
frames) against the march in pairs, which counting launches take: bit-identical
images for every storage kind, opacity correction, early termination inside a
group, runs of every remainder, and runs shorter than a group."""
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
@pytest.mark.parametrize("step,ert,opc", [(0.5, 1.0, 0.0), (0.31, 0.9, 0.0), (1.3, 0.97, 1.0), (9.0, 1.0, 0.0)])
def test_wide_equals_pairs(vr, storage, octets, step, ert, opc):
    import torch
    rng = np.random.default_rng(3)
    vol = synth.blob_volume(40, synth.draw_blobs(rng, 6))
    tf = synth.random_tf(rng, alpha_max=0.15)
    ctx = vr.vr_create(0)
    vr.vr_set_cell_layout(ctx, 1 if octets else 0)
    v = vr.vr_volume_create(ctx, vol, storage, dict(kind="grid", grid=(2, 3, 2)))
    try:
        vr.vr_set_transfer_function(ctx, tf, float(vol.min()), float(vol.max()))
        vr.vr_set_render_params(ctx, step, ert)
        vr.vr_set_opacity_correction(ctx, opc)
        for cam in (synth.orbit_camera(83, 61, 35.0), synth.orbit_camera(1, 1, 120.0), synth.ortho_camera_z(50, 40)):
            vr.vr_set_camera(ctx, cam)
            for mode in (0, 1):
                vr.vr_set_render_mode(ctx, mode)
                images = []
                for count in (True, False):
                    vr.vr_set_count_samples(ctx, count)
                    out = torch.full((cam["height"], cam["width"], 4), float("nan"), device="cuda")
                    vr.vr_render_frame(ctx, v, out)
                    vr.vr_sync(ctx)
                    images.append(out)
                assert torch.equal(images[0], images[1])
                assert float(images[0][..., 3].max()) > 0.02
    finally:
        vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
