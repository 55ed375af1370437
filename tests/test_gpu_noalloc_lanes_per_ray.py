"""vr_render_frame_noalloc with eight, four, two and one lanes per ray, chosen by the
footprints' pixels, the view direction and early termination, against
vr_render_frame.

The table's opacity is the same in every entry, so both calls take the same T at every
sample and end a ray at the same one; its colours are a ramp over a field in [0, 1].
Positions are rounded differently: each call's within 6e-6 voxels along an axis (two
roundings at 40 voxels and the step's), so values within 4e-5 (differences of neighbouring
voxels are at most 1) and, weighted by opacities that sum to at most 1, colours too;
sums of up to 600 samples add 600 * 2^-24. That is 8e-5; a sample too many or too few
changes a pixel's colour by at least T a r > 0.1 * 0.93 * 0.07 * 0.3 = 2e-3."""
import numpy as np
import pytest

from paper_2501_01628_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 8e-5


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


@pytest.mark.parametrize("view,size,step,ert", [
    ("z", (97, 61), 0.5, 0.9),       # 8 lanes
    ("z", (301, 203), 0.5, 0.9),     # 4
    ("z", (401, 301), 0.5, 0.9),     # 2
    ("z", (701, 503), 0.5, 0.9),     # 1
    ("z", (701, 503), 2.7, 1.0),     # 1, runs of a few samples
    ("x", (401, 403), 0.5, 0.9),     # along the rows: 8
    ("x", (601, 601), 0.5, 0.9),     # 4
    ("x", (901, 901), 0.5, 0.9),     # 2
    ("x", (901, 901), 0.5, 1.0),     # 2
    ("x", (1401, 1401), 0.5, 0.9),   # 1
    ("x", (901, 901), 0.07, 1.0),    # 4: long runs
])
def test_lanes_equal_render_frame(vr, view, size, step, ert):
    import torch
    rng = np.random.default_rng(40)
    vol = rng.uniform(0.0, 1.0, (40, 33, 37)).astype(np.float32)
    tf = synth.ramp_tf(64)
    tf[:, :3] = 0.3 + 0.7 * tf[:, :3]
    tf[:, 3] = 0.07
    part = dict(kind="kd", n_bricks=2, cut_fracs=[0.4])
    ext = np.array([37, 33, 40]) / 40.0
    if view == "z":
        cam = synth.ortho_camera_z(*size, extent=tuple(ext[:2]))
    else:
        cam = synth.orbit_camera(*size, 83.0, elevation_deg=4.0, center=tuple(ext / 2))
    got = torch.full((size[1], size[0], 4), float("nan"), device="cuda")
    vr.vr_render_frame_noalloc(torch.from_numpy(vol).cuda(), part, tf, 0.0, 1.0, cam, got, step, ert)
    ctx = vr.vr_create(0)
    v = None
    try:
        v = vr.vr_volume_create(ctx, vol, "f32", part)
        vr.vr_set_transfer_function(ctx, tf, 0.0, 1.0)
        vr.vr_set_camera(ctx, cam)
        vr.vr_set_render_params(ctx, step, ert)
        want = torch.empty((size[1], size[0], 4), device="cuda")
        vr.vr_render_frame(ctx, v, want)
        vr.vr_sync(ctx)
    finally:
        if v is not None:
            vr.vr_volume_release(v)
        vr.vr_destroy(ctx)
    torch.cuda.synchronize()
    assert float((got - want).abs().max()) <= TOL
    assert float(want[..., 3].max()) > 0.5  # the view meets the volume
