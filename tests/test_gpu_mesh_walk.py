"""The mesh march's start grid, walk and sample pairs against the FP64 oracle
where they can go wrong: bricks of a handful of elements (a start grid of one
cell), strongly graded and jittered elements (the walk's longest way), steps
that skip whole elements, and steps with many samples in one element."""
import numpy as np
import pytest

from paper_2501_01628_gb300 import synth
from gpu_helpers import compare_envelope, oracle_env
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


@pytest.mark.parametrize("n,part,cell,refine,jitter,step,ert", [
    (12, dict(kind="grid", grid=(2, 2, 3)), 12.0, 0.0, 0.0, 0.5, 1.0),    # six elements per brick
    (24, dict(kind="kd", n_bricks=5, cut_fracs=[0.3, 0.7, 0.4, 0.6]), 2.0, 4.0, 0.2, 0.5, 0.97),  # graded, jittered
    (30, dict(kind="grid", grid=(1, 2, 1)), 1.5, 0.0, 0.2, 2.3, 1.0),     # samples several elements apart
    (16, dict(kind="grid", grid=(1, 1, 1)), 8.0, 0.0, 0.1, 0.07, 1.0),    # a hundred samples per element
])
def test_walk_matches_oracle(vr, n, part, cell, refine, jitter, step, ert):
    import torch
    boxes = vr.vr_partition_boxes((n,) * 3, part)
    rng = np.random.default_rng(n)
    verts, tets = synth.tet_mesh((n,) * 3, boxes, rng, cell_voxels=cell, jitter=jitter, refine=refine,
                                 focus=(0.3, 0.6, 0.4))
    vals = synth.mesh_field(rng, verts)
    tf = synth.random_tf(rng, alpha_max=0.04)
    for cam in (synth.orbit_camera(61, 47, 25.0, elevation_deg=10.0), synth.ortho_camera_z(33, 40)):
        ctx = vr.vr_create(0)
        m = vr.vr_mesh_create(ctx, verts, vals, tets, (n,) * 3, part)
        try:
            vr.vr_set_transfer_function(ctx, tf, 0.0, 1.0)
            vr.vr_set_camera(ctx, cam)
            vr.vr_set_render_params(ctx, step, ert)
            out = torch.full((cam["height"], cam["width"], 4), float("nan"), device="cuda")
            vr.vr_render_mesh_frame(ctx, m, out)
            vr.vr_sync(ctx)
        finally:
            vr.vr_mesh_release(m)
            vr.vr_destroy(ctx)
        env = oracle_env(oracle.Mesh(verts, vals, tets, (n,) * 3), boxes, tf, 0.0, 1.0, cam, step, ert)
        compare_envelope(out.cpu().numpy().astype(np.float64), env)
