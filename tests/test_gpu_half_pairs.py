"""16-bit storage is widened and subtracted in one instruction: the image must be
that of the same, quantised values in float32 storage, bit for bit, for both types
and cell layouts, in frames of both modes, small and large, and in a batch; over
ordinary values of both signs, values that are subnormal in the type (for bf16, whose
subnormal range alone has no finite scale, some of them), and values at the ends of
its range."""
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


@pytest.mark.parametrize("storage", ["bf16", "f16"])
@pytest.mark.parametrize("octets", [False, True])
@pytest.mark.parametrize("scale", ["ordinary", "subnormal", "largest"])
def test_equals_float_storage(vr, storage, octets, scale):
    import torch
    rng = np.random.default_rng(5)
    vol = rng.uniform(-1.0, 1.0, (19, 22, 25)).astype(np.float32)
    unit = {"ordinary": 1.0, "subnormal": 2.0 ** -15 if storage == "f16" else 2.0 ** -120,
            "largest": 6.0e4 if storage == "f16" else 1.0e38}[scale]
    dtype = torch.bfloat16 if storage == "bf16" else torch.float16
    vol = torch.from_numpy((vol * unit).astype(np.float32)).to(dtype).float().numpy()
    lo, hi = float(np.float32(-unit)), float(np.float32(unit))
    tf = synth.random_tf(rng, alpha_max=0.1)
    cams = [synth.orbit_camera(700, 500, 35.0), synth.orbit_camera(40, 30, 200.0)]
    ctx = vr.vr_create(0)
    vols = []
    try:
        vr.vr_set_transfer_function(ctx, tf, lo, hi)
        for kind, oct_ in (("f32", False), (storage, octets)):
            vr.vr_set_cell_layout(ctx, 1 if oct_ else 0)
            vols.append(vr.vr_volume_create(ctx, vol, kind, dict(kind="grid", grid=(2, 1, 1))))
        for cam in cams:
            vr.vr_set_camera(ctx, cam)
            for mode in (0, 1):
                vr.vr_set_render_mode(ctx, mode)
                images = []
                for v in vols:
                    out = torch.full((cam["height"], cam["width"], 4), float("nan"), device="cuda")
                    vr.vr_render_frame(ctx, v, out)
                    vr.vr_sync(ctx)
                    images.append(out)
                assert torch.equal(images[0], images[1])
                assert float(images[0][..., 3].max()) > 0.1
        vr.vr_set_render_mode(ctx, 0)
        images = []
        for v in vols:
            out = torch.full((1, 500, 700, 4), float("nan"), device="cuda")
            b = vr.vr_batch_create(ctx, [v], cams[:1], out)
            vr.vr_batch_launch(b)
            vr.vr_sync(ctx)
            vr.vr_batch_release(b)
            images.append(out)
        assert torch.equal(images[0], images[1])
    finally:
        for v in vols:
            vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
