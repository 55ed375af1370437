"""Opacity correction by the series and by the general formula: the counting launch
(branch per sample), the plain one (variant by the table's range), a small launch,
the batch kernel and a table set on the device, whose range the host does not know."""
import numpy as np
import pytest

from paper_2501_01628_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vr():
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


@pytest.mark.parametrize("alpha_max", [0.15, 0.9])
@pytest.mark.parametrize("step", [0.5, 0.75, 1.6, 3.0])
def test_series_and_general(vr, step, alpha_max):
    import torch
    rng = np.random.default_rng(11)
    vol = synth.blob_volume(40, synth.draw_blobs(rng, 6))
    tf = synth.random_tf(rng, alpha_max=alpha_max)
    tf[17, 3] = alpha_max
    lo, hi = float(vol.min()), float(vol.max())
    ctx = vr.vr_create(0)
    v = vr.vr_volume_create(ctx, vol, "f32", dict(kind="grid", grid=(2, 1, 1)))
    try:
        vr.vr_set_render_params(ctx, step, 1.0)
        vr.vr_set_opacity_correction(ctx, 1.0)
        for w, h in ((900, 700), (64, 48)):  # pairs; several samples in flight
            cam = synth.orbit_camera(w, h, 35.0)
            vr.vr_set_camera(ctx, cam)
            images = {}
            for name in ("plain", "counted", "batch", "device"):
                out = torch.full((h, w, 4), float("nan"), device="cuda")
                if name == "device":
                    vr.vr_set_transfer_function_async(ctx, torch.from_numpy(tf).cuda(), lo, hi)
                else:
                    vr.vr_set_transfer_function(ctx, tf, lo, hi)
                vr.vr_set_count_samples(ctx, name == "counted")
                if name == "batch":
                    b = vr.vr_batch_create(ctx, [v], [cam], out[None])
                    vr.vr_batch_launch(b)
                    vr.vr_sync(ctx)
                    vr.vr_batch_release(b)
                else:
                    vr.vr_render_frame(ctx, v, out)
                    vr.vr_sync(ctx)
                images[name] = out
            assert float(images["plain"][..., 3].max()) > 0.1
            assert torch.equal(images["plain"], images["counted"])
            assert torch.equal(images["plain"], images["batch"])
            # a sample's two opacities are at most 2 + 3.2 units of 2^-24 apart, which moves
            # the image by twice that; each of the n samples rounds C and T in both images
            n = np.sqrt(3) * 40 / step
            worst = float((images["plain"] - images["device"]).abs().max())
            assert worst <= 2.0 ** -24 * (12 + 4 * n)
            if alpha_max > 0.25 or step > 2.0:  # the general formula in all of them
                assert worst == 0.0
    finally:
        vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
