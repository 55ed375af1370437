"""vr_set_transfer_function_async: the table kernel's pairs against the host-built
ones (bit-identical images) for the smallest and largest tables and growing
ones, in stream order with writes to the tensor before and after it."""
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


def test_async_table_equals_the_synchronous_one(vr):
    import torch
    rng = np.random.default_rng(5)
    vol = synth.blob_volume(24, synth.draw_blobs(rng, 5))
    cam = synth.orbit_camera(40, 33, 20.0)
    ctx = vr.vr_create(0)
    v = vr.vr_volume_create(ctx, vol, "f32", dict(kind="grid", grid=(2, 2, 2)))
    stream = torch.cuda.Stream()
    try:
        vr.vr_set_camera(ctx, cam)
        for n in (2, 3, 127, 128, 129, 1024, 64):
            tf = synth.random_tf(rng, n_entries=n, alpha_max=0.1)
            want = torch.empty((33, 40, 4), device="cuda")
            vr.vr_set_transfer_function(ctx, tf, 0.0, 1.5)
            vr.vr_render_frame(ctx, v, want)
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                table = torch.zeros((n, 4), device="cuda")
                table.copy_(torch.from_numpy(tf).pin_memory(), non_blocking=True)
                vr.vr_set_transfer_function_async(ctx, table, 0.0, 1.5)
                table.zero_()  # after the library's kernel in stream order
                got = torch.full((33, 40, 4), float("nan"), device="cuda")
                vr.vr_render_frame(ctx, v, got)
                vr.vr_sync(ctx)
            assert torch.equal(got, want)
        bad = torch.zeros((1, 4), device="cuda")
        for args in ((bad, 0.0, 1.0), (table, 1.0, 1.0), (table, 0.0, float("inf"))):
            with pytest.raises(vr.VrError) as e:
                vr.vr_set_transfer_function_async(ctx, *args)
            assert e.value.status == vr.VR_ERR_ARG
        with pytest.raises(ValueError):
            vr.vr_set_transfer_function_async(ctx, torch.zeros((4, 4)), 0.0, 1.0)
    finally:
        vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
