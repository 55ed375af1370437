"""The adjoint's paths against the oracle's FP64 adjoint, where they can go
wrong: runs shorter than a segment and longer than a thread's group of segments,
voxel gradients through quads and straight into the voxels, every storage kind,
table sizes at the ends of their range, an image in several bands, and a run
beyond the refused length."""
import numpy as np
import pytest

import oracle
from paper_2501_01628_gb300 import synth

pytestmark = pytest.mark.gpu

# the adjoint's bar of the differentiation tests: norm-wise 1e-3 (FP32 cells and
# table intervals against FP64 ones, where a sample sits on a knot)
REL = 1e-3


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


def _backward(vr, vol, part, tf, cam, G, step, storage="f32", octets=False, want_volume=True):
    import torch
    ctx = vr.vr_create(0)
    v = None
    try:
        vr.vr_set_cell_layout(ctx, 1 if octets else 0)
        v = vr.vr_volume_create(ctx, vol, storage, part)
        vr.vr_set_transfer_function(ctx, tf, 0.0, 1.0)
        vr.vr_set_camera(ctx, cam)
        vr.vr_set_render_params(ctx, step, 1.0)
        gtf = torch.zeros((tf.shape[0], 4), device="cuda")
        gvol = torch.zeros(vol.shape, device="cuda") if want_volume else None
        vr.vr_render_backward(ctx, v, torch.from_numpy(G.astype(np.float32)).cuda(), gtf, gvol)
        vr.vr_sync(ctx)
        return gtf.cpu().numpy().astype(np.float64), gvol.cpu().numpy().astype(np.float64) if want_volume else None
    finally:
        if v is not None:
            vr.vr_volume_release(v)
        vr.vr_destroy(ctx)


def _scene(rng, shape, ntf=256):
    n = max(shape)
    vol = synth.blob_volume(n, synth.draw_blobs(rng, 5))[:shape[0], :shape[1], :shape[2]].copy()
    vol = (vol - vol.min()) / (vol.max() - vol.min())
    vol = (0.9 * vol + rng.uniform(0.02, 0.08, shape)).astype(np.float32)
    return vol, synth.random_tf(rng, n_entries=ntf, alpha_max=0.2)


def _close(got, ref):
    assert np.linalg.norm(ref) > 0
    assert np.linalg.norm(got - ref) <= REL * np.linalg.norm(ref)


@pytest.mark.parametrize("shape,part,size,step,ntf", [
    ((9, 7, 8), dict(kind="grid", grid=(4, 3, 4)), (33, 21), 0.5, 2),     # runs of a few samples
    ((40, 33, 37), dict(kind="grid", grid=(1, 1, 1)), (17, 35), 0.11, 1024),  # runs of up to 580 samples
    ((48, 48, 48), dict(kind="grid", grid=(2, 1, 1)), (9, 7), 0.5, 256),  # straight into the voxels
    ((21, 40, 30), dict(kind="kd", n_bricks=9, cut_fracs=[0.3, 0.6, 0.5, 0.4, 0.7, 0.35, 0.5, 0.6]), (64, 48), 0.8, 33),
    ((21, 40, 30), dict(kind="grid", grid=(2, 3, 1)), (170, 131), 0.5, 64),  # through quads: many more samples than quads
])
def test_paths_match_oracle(vr, shape, part, size, step, ntf):
    rng = np.random.default_rng(sum(shape) + ntf)
    vol, tf = _scene(rng, shape, ntf)
    cam = synth.orbit_camera(*size, 40.0, elevation_deg=-15.0)
    G = rng.standard_normal((size[1], size[0], 4)).astype(np.float32)
    gtf, gvol = _backward(vr, vol, part, tf, cam, G, step)
    boxes = vr.vr_partition_boxes(vol.shape[::-1], part)
    rtf, rvol = oracle.render_grad(vol, boxes, tf, 0.0, 1.0, cam, G, step)
    _close(gtf, rtf)
    _close(gvol, rvol)
    only, _ = _backward(vr, vol, part, tf, cam, G, step, want_volume=False)
    _close(only, rtf)


@pytest.mark.parametrize("storage,octets", [("bf16", False), ("f16", False), ("bf16", True), ("f16", True)])
def test_storage_kinds_match_oracle(vr, storage, octets):
    rng = np.random.default_rng(3)
    vol, tf = _scene(rng, (26, 31, 29))
    part = dict(kind="grid", grid=(2, 2, 1))
    cam = synth.orbit_camera(41, 30, 205.0, elevation_deg=30.0)
    G = rng.standard_normal((30, 41, 4)).astype(np.float32)
    gtf, gvol = _backward(vr, vol, part, tf, cam, G, 0.5, storage, octets)
    boxes = vr.vr_partition_boxes(vol.shape[::-1], part)
    code = oracle.BF16 if storage == "bf16" else oracle.F16
    rtf, rvol = oracle.render_grad(synth.quantize(vol, storage), boxes, tf, 0.0, 1.0, cam, G, 0.5, dtype=code)
    _close(gtf, rtf)
    _close(gvol, rvol)


def test_image_in_several_bands_matches_oracle(vr):
    """Runs of up to 3700 samples over a 200 x 900 image: over 1 GB of samples, so
    bands of 450 rows; the upstream gradient lives on pixels of both, the rows at
    their edge among them. The ramp table has a slope everywhere
    and leaves the 3700 samples transparent enough for gradients in FP32's range."""
    rng = np.random.default_rng(8)
    vol, _ = _scene(rng, (64, 64, 64))
    tf = synth.ramp_tf(alpha_max=0.002)
    part = dict(kind="grid", grid=(1, 1, 1))
    cam = synth.orbit_camera(200, 900, 30.0, elevation_deg=20.0)
    ys = np.concatenate([np.arange(330, 400), rng.integers(150, 750, 60), np.arange(440, 460)])
    pix = np.unique(np.stack([rng.integers(60, 140, ys.size), ys], axis=1), axis=0)
    g = rng.standard_normal((len(pix), 4)).astype(np.float32)
    G = np.zeros((900, 200, 4), np.float32)
    G[pix[:, 1], pix[:, 0]] = g
    gtf, gvol = _backward(vr, vol, part, tf, cam, G, 0.03)
    boxes = vr.vr_partition_boxes((64,) * 3, part)
    rtf, rvol = oracle.render_grad(vol, boxes, tf, 0.0, 1.0, cam, g, 0.03, pixels=pix)
    _close(gtf, rtf)
    _close(gvol, rvol)


def test_overlong_runs_are_reported_and_the_rest_is_right(vr):
    """One brick with runs of up to 4400 samples: the call reports VR_ERR_BOUNDS
    at vr_sync, and a later call with a legal step is right."""
    import torch
    rng = np.random.default_rng(9)
    vol, tf = _scene(rng, (22, 22, 22))
    part = dict(kind="grid", grid=(1, 1, 1))
    cam = synth.orbit_camera(24, 20, 45.0, elevation_deg=35.0, radius=1.2)
    G = rng.standard_normal((20, 24, 4)).astype(np.float32)
    with pytest.raises(vr.VrError) as e:
        _backward(vr, vol, part, tf, cam, G, 0.005)
    assert e.value.status == vr.VR_ERR_BOUNDS
    gtf, gvol = _backward(vr, vol, part, tf, cam, G, 0.5)
    boxes = vr.vr_partition_boxes((22,) * 3, part)
    rtf, rvol = oracle.render_grad(vol, boxes, tf, 0.0, 1.0, cam, G, 0.5)
    _close(gtf, rtf)
    _close(gvol, rvol)
