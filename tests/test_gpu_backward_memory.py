"""vr_render_backward's memory where there is no room: a workspace or quads that
cannot be had, and what is not asked for again after that; and another allocation
that finds no room while the backward's memory is kept. The failures are injected
on the host. Every gradient against the oracle's FP64 adjoint."""
import numpy as np
import pytest

import oracle
from paper_2501_01628_gb300 import synth

pytestmark = pytest.mark.gpu

REL = 1e-3  # the adjoint's bar of the differentiation tests
SHAPE, SIZE = (21, 40, 30), (170, 131)  # many more samples than quads: through quads
PART = dict(kind="grid", grid=(2, 3, 1))


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


@pytest.fixture()
def scene(vr):
    """backward() checks the gradients of a context's volume; pending() tells whether an
    injected fault is still to come (and clears it)."""
    import torch
    rng = np.random.default_rng(12)
    vol = synth.blob_volume(40, synth.draw_blobs(rng, 5))[:SHAPE[0], :SHAPE[1], :SHAPE[2]].copy()
    vol = (vol - vol.min()) / (vol.max() - vol.min())
    vol = (0.9 * vol + rng.uniform(0.02, 0.08, SHAPE)).astype(np.float32)
    tf = synth.random_tf(rng, n_entries=64, alpha_max=0.2)
    cam = synth.orbit_camera(*SIZE, 40.0, elevation_deg=-15.0)
    G = rng.standard_normal((SIZE[1], SIZE[0], 4)).astype(np.float32)
    boxes = vr.vr_partition_boxes(SHAPE[::-1], PART)
    want = oracle.render_grad(vol, boxes, tf, 0.0, 1.0, cam, G, 0.5)
    ctx, bare = vr.vr_create(0), vr.vr_create(0)
    v = vr.vr_volume_create(ctx, vol, "f32", PART)
    vr.vr_set_transfer_function(ctx, tf, 0.0, 1.0)
    vr.vr_set_camera(ctx, cam)
    vr.vr_set_render_params(ctx, 0.5, 1.0)
    dG = torch.from_numpy(G).cuda()

    def backward():
        gtf, gvol = torch.zeros((64, 4), device="cuda"), torch.zeros(SHAPE, device="cuda")
        vr.vr_render_backward(ctx, v, dG, gtf, gvol)
        vr.vr_sync(ctx)
        for got, ref in zip((gtf, gvol), want):
            assert np.linalg.norm(got.cpu().numpy() - ref) <= REL * np.linalg.norm(ref)

    def pending():
        try:
            vr.vr_volume_release(vr.vr_volume_create(bare, vol, "f32", PART))  # nothing to give back there
        except vr.VrError as e:
            assert e.status == vr.VR_ERR_OOM
            return True
        return False

    yield ctx, v, cam, backward, pending
    vr.vr_debug_inject_fault(vr.VR_FAULT_NONE, 0)
    vr.vr_volume_release(v)
    vr.vr_destroy(ctx)
    vr.vr_destroy(bare)


@pytest.mark.parametrize("refused", [0, 1])  # the workspace; the quads
def test_refused_memory_is_done_without_and_not_asked_for_again(vr, scene, refused):
    _, _, _, backward, pending = scene
    vr.vr_debug_inject_fault(vr.VR_FAULT_ALLOC, refused)
    backward()
    assert not pending()
    vr.vr_debug_inject_fault(vr.VR_FAULT_ALLOC, 0)
    backward()
    assert pending()
    backward()


def test_kept_memory_is_given_back(vr, scene):
    import torch
    ctx, v, cam, backward, _ = scene
    big = synth.orbit_camera(800, 600, 40.0, elevation_deg=-15.0)
    vr.vr_set_camera(ctx, big)
    grad = torch.rand((600, 800, 4), device="cuda")
    vr.vr_render_backward(ctx, v, grad, torch.zeros((64, 4), device="cuda"), torch.zeros(SHAPE, device="cuda"))
    vr.vr_sync(ctx)
    small = torch.rand((4, 4, 4), device="cuda")
    before = torch.cuda.mem_get_info()[0]
    vr.vr_debug_inject_fault(vr.VR_FAULT_ALLOC, 0)
    other = vr.vr_volume_create(ctx, small)
    # the workspace holds 4 bytes for every footprint pixel times the longest run, and more;
    # the device's memory is handed out in pieces of up to 2 MB
    _, rects = vr.vr_plan_view(SHAPE[::-1], PART, big)
    boxes = vr.vr_partition_boxes(SHAPE[::-1], PART)
    runs = np.linalg.norm(boxes[:, 3:] - boxes[:, :3], axis=1) / 0.5
    samples = 4 * int((rects[:, 2] * rects[:, 3] * runs).sum())
    assert samples > 16 << 20
    assert torch.cuda.mem_get_info()[0] - before >= samples - (4 << 20)
    vr.vr_set_camera(ctx, cam)
    backward()
    vr.vr_volume_release(other)
    backward()
