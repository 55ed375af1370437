"""vr_render_frame_noalloc, whose rays are shared by several lanes, against
vr_render_frame and the FP64 oracle where the sharing can go wrong: runs shorter
than the lanes, runs that end inside a group, image sizes that do not fill a
tile, early termination inside a group, and tables of two and 1024 entries."""
import numpy as np
import pytest

from paper_2501_01628_gb300 import synth
from gpu_helpers import compare_envelope, oracle_env

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vr():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2501_01628_gb300 import vr as _vr
    return _vr


@pytest.mark.parametrize("shape,part,size,step,ert,ntf", [
    ((6, 5, 7), dict(kind="grid", grid=(3, 2, 2)), (13, 9), 0.5, 1.0, 256),      # runs of up to eight samples
    ((33, 20, 41), dict(kind="kd", n_bricks=4, cut_fracs=[0.4, 0.6, 0.5]), (67, 45), 0.5, 0.9, 2),
    ((24, 24, 24), dict(kind="grid", grid=(1, 1, 1)), (1, 1), 0.13, 1.0, 1024),
    ((17, 30, 23), dict(kind="grid", grid=(2, 1, 1)), (34, 27), 2.5, 0.97, 64),
])
def test_lanes_match_oracle_and_render_frame(vr, shape, part, size, step, ert, ntf):
    import torch
    rng = np.random.default_rng(sum(shape))
    n = max(shape)
    vol = synth.blob_volume(n, synth.draw_blobs(rng, 5))[:shape[0], :shape[1], :shape[2]].copy()
    vol += rng.uniform(0, 0.05, vol.shape).astype(np.float32)
    tf = synth.random_tf(rng, n_entries=ntf, alpha_max=0.15)
    lo, hi = synth.volume_range(vol)
    ext = np.array(shape[::-1], dtype=np.float64) / n
    cam = synth.orbit_camera(*size, 70.0, elevation_deg=-20.0, center=tuple(ext / 2))
    out = torch.full((size[1], size[0], 4), float("nan"), device="cuda")
    vr.vr_render_frame_noalloc(torch.from_numpy(vol).cuda(), part, tf, lo, hi, cam, out, step, ert)
    torch.cuda.synchronize()
    boxes = vr.vr_partition_boxes(shape[::-1], part)
    compare_envelope(out.cpu().numpy().astype(np.float64), oracle_env(vol, boxes, tf, lo, hi, cam, step, ert))
