"""Frames of vr_render_partials reuse the last released frame's memory: two frames
alive at once, releases in either order, growing and shrinking images, a release
right after the composite's launch followed by a frame on another stream, and an
allocation that finds no room while memory is kept. Every image must equal
vr_render_frame's bit for bit."""
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


def test_reused_frames_equal_render_frame(vr):
    import torch
    vol, tf = synth.small_blob_scene(n=48)
    cams = [synth.orbit_camera(w, h, az) for w, h, az in
            ((160, 120, 10.0), (40, 30, 100.0), (320, 240, 190.0), (160, 120, 280.0))]
    ctx = vr.vr_create(0)
    v = vr.vr_volume_create(ctx, vol, "f32", dict(kind="grid", grid=(2, 3, 2)))
    try:
        vr.vr_set_transfer_function(ctx, tf, float(vol.min()), float(vol.max()))
        want = []
        for cam in cams:
            vr.vr_set_camera(ctx, cam)
            out = torch.empty((cam["height"], cam["width"], 4), device="cuda")
            vr.vr_render_frame(ctx, v, out)
            want.append(out)
        vr.vr_sync(ctx)

        def partials(i, stream=None):
            vr.vr_set_camera(ctx, cams[i])
            return vr.vr_render_partials(ctx, v, stream)

        def image(i, frame, stream=None):
            out = torch.full((cams[i]["height"], cams[i]["width"], 4), float("nan"), device="cuda")
            torch.cuda.synchronize()
            vr.vr_composite(ctx, frame, out, stream)
            return out

        for pair in ((0, 1), (1, 0), (2, 3), (3, 2)):
            for order in ((0, 1), (1, 0)):
                frames = [partials(i) for i in pair]
                outs = [image(i, f) for i, f in zip(pair, frames)]
                for k in order:
                    vr.vr_frame_release(frames[k])
                torch.cuda.synchronize()
                for i, out in zip(pair, outs):
                    assert torch.equal(out, want[i])
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        outs = []
        for k in range(6):
            s = streams[k & 1]
            f = partials(k % 4, s)
            outs.append((k % 4, image(k % 4, f, s)))
            vr.vr_frame_release(f)
        torch.cuda.synchronize()
        for i, out in outs:
            assert torch.equal(out, want[i])
        # the kept memory is given back when an allocation fails once
        vr.vr_debug_inject_fault(vr.VR_FAULT_ALLOC, 0)
        other = vr.vr_volume_create(ctx, vol, "f32", dict(kind="grid", grid=(1, 1, 1)))
        vr.vr_volume_release(other)
        f = partials(2)
        out = image(2, f)
        vr.vr_frame_release(f)
        torch.cuda.synchronize()
        assert torch.equal(out, want[2])
    finally:
        vr.vr_debug_inject_fault(vr.VR_FAULT_NONE, 0)
        vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
