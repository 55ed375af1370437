"""Meshes whose bricks have faces inside them that no second element shares:
vertices doubled on an interior plane, hanging nodes, and a vertex set per
element. vr_mesh_create accepts them (the elements fill their brick); the image
must be the oracle's, which searches every element, and, as the field is the
same, the conforming mesh's. One of the bricks stays conforming where a mesh has
several."""
import numpy as np
import pytest

import oracle
from paper_2501_01628_gb300 import synth
from gpu_helpers import TOL, compare_envelope, oracle_env

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


def doubled(verts, vals, tets, some, rng):
    """The vertices on the plane of nodes nearest y = 0.5, doubled for the elements above it."""
    y = verts[:, 1].astype(np.float64)
    at = y[np.argmin(np.abs(y - 0.5))]
    on = np.flatnonzero(y == at)
    other = np.arange(len(verts))
    other[on] = len(verts) + np.arange(len(on))
    above = some & (y[tets].mean(axis=1) > at)
    tets = tets.copy()
    tets[above] = other[tets[above]]
    return np.concatenate([verts, verts[on]]), np.concatenate([vals, vals[on]]), tets.astype(np.int32)


def hanging(verts, vals, tets, some, rng):
    """A fifth of the elements cut in two at the middle of their longest edge, their neighbours not."""
    edges = [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]
    p = verts[tets].astype(np.float64)
    longest = np.argmax([np.linalg.norm(p[:, a] - p[:, b], axis=1) for a, b in edges], axis=0)
    cut = some & (rng.uniform(size=len(tets)) < 0.2)
    cut[np.flatnonzero(some)[0]] = True
    new_v, new_s, new_t = [], [], []
    for i in np.flatnonzero(cut):
        a, b = edges[longest[i]]
        mid = len(verts) + len(new_v)
        new_v.append((p[i, a] + p[i, b]) / 2)
        new_s.append((float(vals[tets[i, a]]) + float(vals[tets[i, b]])) / 2)
        for end in (a, b):
            t = tets[i].copy()
            t[end] = mid
            new_t.append(t)
    return (np.concatenate([verts, np.array(new_v, np.float32)]), np.concatenate([vals, np.array(new_s, np.float32)]),
            np.concatenate([tets[~cut], np.array(new_t)]).astype(np.int32))


def apart(verts, vals, tets, some, rng):
    """A vertex set of its own for every element."""
    own = len(verts) + np.arange(tets.size).reshape(-1, 4)
    t = np.where(some[:, None], own, tets).astype(np.int32)
    return np.concatenate([verts, verts[tets].reshape(-1, 3)]), np.concatenate([vals, vals[tets].ravel()]), t


@pytest.mark.parametrize("n,part,cell,jitter,step,ert", [
    (12, dict(kind="grid", grid=(1, 1, 1)), 12.0, 0.0, 0.5, 1.0),   # six elements: a start grid of one cell
    (24, dict(kind="grid", grid=(2, 1, 1)), 3.0, 0.1, 0.5, 0.97),
    (30, dict(kind="kd", n_bricks=4, cut_fracs=[0.4, 0.6, 0.5]), 2.0, 0.2, 2.3, 1.0),  # samples several elements apart
])
@pytest.mark.parametrize("broken", [doubled, hanging, apart])
def test_unmatched_faces_inside_a_brick(vr, broken, n, part, cell, jitter, step, ert):
    import torch
    boxes = vr.vr_partition_boxes((n,) * 3, part)
    rng = np.random.default_rng(n)
    verts, tets = synth.tet_mesh((n,) * 3, boxes, rng, cell_voxels=cell, jitter=jitter)
    vals = synth.mesh_field(rng, verts)
    tf = synth.random_tf(rng, alpha_max=0.04)
    cam = synth.orbit_camera(61, 47, 25.0, elevation_deg=10.0)
    centre = verts[tets].astype(np.float64).mean(axis=1) * n
    some = np.ones(len(tets), bool)
    if len(boxes) > 1:  # the last brick stays as it is
        some = ~((centre >= boxes[-1, :3]) & (centre < boxes[-1, 3:])).all(axis=1)
    meshes = [(verts, vals, tets), broken(verts, vals, tets, some, rng)]
    images = []
    ctx = vr.vr_create(0)
    try:
        vr.vr_set_transfer_function(ctx, tf, 0.0, 1.0)
        vr.vr_set_camera(ctx, cam)
        vr.vr_set_render_params(ctx, step, ert)
        for mesh in meshes:
            m = vr.vr_mesh_create(ctx, *mesh, (n,) * 3, part)
            out = torch.full((cam["height"], cam["width"], 4), float("nan"), device="cuda")
            vr.vr_render_mesh_frame(ctx, m, out)
            vr.vr_sync(ctx)
            vr.vr_mesh_release(m)
            images.append(out.cpu().numpy().astype(np.float64))
    finally:
        vr.vr_destroy(ctx)
    env = oracle_env(oracle.Mesh(*meshes[1], (n,) * 3), boxes, tf, 0.0, 1.0, cam, step, ert)
    compare_envelope(images[1], env)
    if ert >= 1.0:  # no decision that rounding could turn: each within TOL of one field's image
        assert np.abs(images[1] - images[0]).max() <= 2 * TOL
