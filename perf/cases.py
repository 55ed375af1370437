"""What the framework is timed on: frames, batches, training steps, streamed and
in-situ time steps, through the calls of paper_2501_01628_gb300 that a user's
program makes.

A case is a dict of plain values; `path` names the calls:
  frame     vr_set_camera + vr_render_frame, sort-last, into device memory
  cycle     the same with ray-state cycling (vr_set_render_mode 1)
  host      the same (sort-last) into pinned host memory, synchronous
  partials  vr_render_partials + vr_composite + vr_frame_release
  batch     one vr_batch_launch of volumes x views
  train     forward of `views` views through autograd.Renderer, a squared image
            loss, backward, and a gradient step on the table and the voxels
  mesh      vr_set_camera + vr_render_mesh_frame of a tetrahedral mesh
  stream    streaming.TimeSeriesRenderer over `steps` time steps in host memory
  insitu    vr_volume_update from device memory, then one frame
  noalloc   vr_render_frame_noalloc on the caller's volume
Volumes are value noise plus Gaussian blobs, tables are random piecewise-linear
ones (synth.random_tf), cameras orbit the volume, all from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2501_01628_gb300 import autograd, streaming, synth, vr

# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------


def _case(path, dims, size, **kw):
    c = dict(path=path, nx=dims[0], ny=dims[1], nz=dims[2], W=size[0], H=size[1], part="grid", gx=1, gy=1, gz=1,
             bricks=1, storage="f32", octets=False, ortho=False, step=0.5, ert=1.0, opc=0.0, radix=False, views=1,
             volumes=1, steps=1)
    c.update(kw)
    if c["part"] == "grid":
        c["bricks"] = c["gx"] * c["gy"] * c["gz"]
    return c


def listed():
    return [
        # an interactive preview of a small field: latency and launches
        _case("frame", (64, 64, 64), (256, 256), gx=2, gy=2, gz=2, ortho=True, name="frame_preview_64"),
        # the frame of an interactive session on a distributed data set, one
        # brick per rank of 36 (the benchmark's frame)
        _case("frame", (512, 512, 512), (1920, 1080), gx=4, gy=3, gz=3, ert=0.99, radix=True, name="frame_orbit_512"),
        # a large data set in 16-bit storage, unevenly split over 64 ranks, a still
        # image without early termination
        _case("frame", (1024, 1024, 1024), (2048, 2048), part="kd", bricks=64, storage="bf16",
              name="frame_bf16_1024"),
        # an orthographic image for a figure: ragged volume and image, float16
        # octets, opacity correction at another step, delivered to host memory
        _case("host", (300, 201, 257), (1283, 721), gx=3, gy=2, gz=2, storage="f16", octets=True, ortho=True,
              step=0.75, opc=1.0, name="host_ortho_octets"),
        # the interactive frame with ray-state cycling and global termination
        _case("cycle", (512, 512, 512), (1920, 1080), gx=4, gy=3, gz=3, ert=0.99, name="cycle_orbit_512"),
        # a rank's own two steps: partial images handed over, then composited
        _case("partials", (255, 255, 255), (1023, 767), gx=3, gy=3, gz=3, radix=True, name="partials_255"),
        # a time-varying multi-field data set seen from several views in one launch
        _case("batch", (256, 256, 256), (512, 512), part="kd", bricks=12, storage="f16", volumes=4, views=8,
              name="batch_4x8_256"),
        # one optimiser step of fitting a volume and its table to images
        _case("train", (256, 256, 256), (512, 512), gx=2, gy=2, gz=2, views=4, name="train_256"),
        # unstructured finite elements, unevenly graded, one part per rank
        _case("mesh", (192, 192, 192), (1280, 720), gx=4, gy=3, gz=3, ert=0.99, radix=True, name="mesh_192"),
        # time steps that do not all fit: upload of the next beside this one's frames
        _case("stream", (256, 256, 256), (1280, 720), gx=2, gy=2, gz=2, ert=0.99, steps=4, views=2,
              name="stream_4x256"),
        # a running simulation hands its device field over and sees a frame of it
        _case("insitu", (384, 384, 384), (1280, 720), gx=2, gy=2, gz=3, ert=0.99, name="insitu_384"),
        # a frame inside a program that allows no device allocation
        _case("noalloc", (128, 128, 128), (400, 300), part="kd", bricks=6, name="noalloc_128"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(most):
        g = dict(gx=rng.randint(1, most), gy=rng.randint(1, most), gz=rng.randint(1, most))
        return g if rng.random() < 0.7 else dict(part="kd", bricks=rng.randint(1, min(64, most ** 3)))

    path = rng.choice(["frame", "frame", "frame", "cycle", "host", "partials", "batch", "train", "mesh", "stream",
                       "insitu", "noalloc"])
    opts = dict(ortho=rng.random() < 0.25, step=rng.choice([0.5, 0.5, 0.5, 0.37, 0.8, 1.0]),
                ert=rng.choice([1.0, 1.0, 0.99, 0.95]))
    if path in ("frame", "cycle", "host", "partials"):
        storage = rng.choice(["f32", "f32", "bf16", "f16"])
        opts.update(grid(4), storage=storage, octets=storage != "f32" and rng.random() < 0.5,
                    opc=rng.choice([0.0, 0.0, 0.0, 1.0]), radix=rng.random() < 0.5)
        return _case(path, (size(40, 512), size(40, 512), size(40, 512)), (size(160, 2048), size(120, 2048)), **opts)
    if path == "batch":
        opts.update(grid(3), storage=rng.choice(["f32", "bf16", "f16"]), volumes=rng.randint(1, 4),
                    views=rng.randint(1, 8))
        return _case(path, (size(40, 256), size(40, 256), size(40, 256)), (size(64, 512), size(64, 512)), **opts)
    if path == "train":
        opts.update(grid(2), ert=1.0, views=rng.randint(1, 4))
        return _case(path, (size(32, 256), size(32, 256), size(32, 256)), (size(64, 512), size(64, 512)), **opts)
    if path == "mesh":
        n = size(48, 192)
        opts.update(gx=rng.randint(1, 4), gy=rng.randint(1, 3), gz=rng.randint(1, 3), radix=rng.random() < 0.5)
        return _case(path, (n, n, n), (size(160, 1280), size(120, 1024)), **opts)
    if path == "stream":
        opts.update(grid(3), steps=rng.randint(2, 4), views=rng.randint(1, 3))
        return _case(path, (size(48, 256), size(48, 256), size(48, 256)), (size(160, 1280), size(120, 1024)), **opts)
    if path == "insitu":
        opts.update(grid(3), storage=rng.choice(["f32", "f32", "bf16", "f16"]))
        return _case(path, (size(48, 384), size(48, 384), size(48, 384)), (size(160, 1280), size(120, 1024)), **opts)
    opts.update(grid(2))  # noalloc: partial images of every brick fit the fixed scratch
    return _case(path, (size(32, 192), size(32, 192), size(32, 192)), (size(64, 400), size(64, 320)), **opts)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------


def _dims(c):
    return c["nx"], c["ny"], c["nz"]


def _volume(c, rng):
    """float32 [nz, ny, nx] on the GPU: value noise of five octaves (4 to 64
    cells per unit) plus eight Gaussian blobs, scaled to [0, 1]."""
    nx, ny, nz = _dims(c)
    nmax = max(nx, ny, nz)
    pos = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / nmax for n in (nz, ny, nx)]
    acc = torch.zeros((nz, ny, nx), dtype=torch.float32, device="cuda")
    for o in range(5):
        cells = 4 * 2 ** o
        lat = torch.from_numpy(rng.random((cells + 1,) * 3, dtype=np.float32)).cuda()
        for axis in (0, 1, 2):
            at = pos[axis] * cells
            i = torch.clamp(torch.floor(at).long(), max=cells - 1)
            w = (at - i).float().reshape([-1 if a == axis else 1 for a in range(3)])
            lo = torch.index_select(lat, axis, i)
            lat = lo.add_((torch.index_select(lat, axis, i + 1).sub_(lo)).mul_(w))
        acc.add_(lat, alpha=0.5 ** o)
        del lat, lo
    acc.mul_(0.5)
    blobs = synth.draw_blobs(rng, 8)
    for mu, s, a in zip(blobs.centers, blobs.sigmas, blobs.amps):
        g = [torch.exp(-((x - m) ** 2) / (2 * s * s)).float() for x, m in zip(pos, mu[::-1])]
        acc.addcmul_((a * g[0])[:, None, None] * g[1][None, :, None], g[2][None, None, :])
    lo, hi = torch.aminmax(acc)
    return acc.sub_(lo).div_(hi - lo)


def _cameras(c, rng, n):
    """Orbit cameras around the volume's centre; orthographic ones see its
    bounding sphere."""
    dims = np.array(_dims(c), dtype=np.float64)
    ext = dims / dims.max()
    cams = []
    for _ in range(n):
        cam = synth.orbit_camera(c["W"], c["H"], float(rng.uniform(0, 360)), elevation_deg=float(rng.uniform(-25, 25)),
                                 center=tuple(ext / 2))
        if c["ortho"]:
            span = 1.05 * float(np.linalg.norm(ext))
            cam.update(ortho=1, fovy_deg=0.0, ortho_w=span * max(1.0, c["W"] / c["H"]),
                       ortho_h=span * max(1.0, c["H"] / c["W"]))
        cams.append(cam)
    return cams


def _partition(c, rng):
    if c["part"] == "grid":
        return dict(kind="grid", grid=(c["gx"], c["gy"], c["gz"]))
    return dict(kind="kd", n_bricks=c["bricks"], cut_fracs=synth.kd_cut_fractions(rng, c["bricks"]))


def _scene(c, seed):
    """What both the framework and exact() take: partition, table, cameras, volumes."""
    rng = np.random.default_rng([seed, 7])
    part = _partition(c, rng)
    tf = synth.random_tf(rng)
    cams = _cameras(c, rng, c["views"])
    n = c["steps"] if c["path"] == "stream" else c["volumes"]
    return part, tf, cams, [_volume(c, rng) for _ in range(n)], rng


def _targets(c, seed):
    """Photographs to fit: smooth RGBA images, one per view."""
    g = torch.Generator().manual_seed(seed)
    low = torch.rand((c["views"], 4, 6, 8), generator=g).cuda()
    big = torch.nn.functional.interpolate(low, size=(c["H"], c["W"]), mode="bilinear", align_corners=True)
    return [t.permute(1, 2, 0).contiguous() for t in big]


class _State:
    """A user's handles and buffers, released with the object."""

    def __init__(self):
        self.ctx, self.vols, self.mesh, self.batch, self.renderer, self.series = None, [], None, None, None, None

    def __del__(self):
        torch.cuda.synchronize()
        if self.series is not None:
            self.series.close()
        if self.batch is not None:
            vr.vr_batch_release(self.batch)
        for v in self.vols:
            vr.vr_volume_release(v)
        if self.mesh is not None:
            vr.vr_mesh_release(self.mesh)
        if self.renderer is not None:
            self.renderer.close()
        if self.ctx is not None:
            vr.vr_destroy(self.ctx)


def _image(c, *lead):
    return torch.empty((*lead, c["H"], c["W"], 4), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    c = case
    s = _State()
    s.case = c
    if c["path"] == "mesh":
        rng = np.random.default_rng([seed, 7])
        s.part = _partition(c, rng)
        tf = synth.random_tf(rng)
        s.cams = _cameras(c, rng, 1)
        boxes = vr.vr_partition_boxes(_dims(c), s.part)
        verts, tets = synth.tet_mesh(_dims(c), boxes, rng, cell_voxels=5.0, jitter=0.2, refine=1.5,
                                     focus=(0.35, 0.55, 0.45))
        vals = synth.mesh_field(rng, verts)
    else:
        s.part, tf, s.cams, fields, _ = _scene(c, seed)
    s.out = _image(c)
    if c["path"] == "noalloc":
        s.tf, s.volume = tf, fields[0]
        return s
    if c["path"] == "train":
        s.renderer = autograd.Renderer(s.part, 0.0, 1.0, step_voxels=c["step"])
        s.tf = torch.from_numpy(tf).cuda().requires_grad_(True)
        s.density = fields[0].requires_grad_(True)
        s.targets = _targets(c, seed)
        s.opt = torch.optim.SGD([s.tf, s.density], lr=1e-3)
        return s
    s.ctx = vr.vr_create(torch.cuda.current_device())
    vr.vr_set_transfer_function(s.ctx, tf, 0.0, 1.0)
    vr.vr_set_render_params(s.ctx, c["step"], c["ert"])
    if c["opc"]:
        vr.vr_set_opacity_correction(s.ctx, c["opc"])
    if c["radix"]:
        vr.vr_set_composite_schedule(s.ctx, (c["gx"], c["gy"], c["gz"]) if c["part"] == "grid" else (c["bricks"],))
    if c["octets"]:
        vr.vr_set_cell_layout(s.ctx, 1)
    if c["path"] == "cycle":
        vr.vr_set_render_mode(s.ctx, 1)
    if c["path"] == "mesh":
        s.mesh = vr.vr_mesh_create(s.ctx, verts, vals, tets, _dims(c), s.part)
        return s
    if c["path"] == "stream":
        s.fields = [f.cpu().pin_memory() for f in fields]
        s.outs = [[_image(c) for _ in s.cams] for _ in range(c["steps"])]
        s.series = streaming.TimeSeriesRenderer(s.ctx, s.fields, s.part, c["storage"], slots=2)
        return s
    s.vols = [vr.vr_volume_create(s.ctx, f, c["storage"], s.part) for f in fields]
    if c["path"] == "batch":
        s.out = _image(c, c["volumes"] * c["views"])
        s.batch = vr.vr_batch_create(s.ctx, s.vols, s.cams, s.out)
        vr.vr_batch_configure(s.batch, packet_width=4, blocks_per_sm=0, order=1)
    if c["path"] == "insitu":
        s.field = fields[0]
    if c["path"] == "host":
        s.out = torch.empty((c["H"], c["W"], 4), dtype=torch.float32).pin_memory()
    return s


def run(state):
    s = state
    path = s.case["path"]
    if path == "noalloc":
        vr.vr_render_frame_noalloc(s.volume, s.part, s.tf, 0.0, 1.0, s.cams[0], s.out, s.case["step"], s.case["ert"])
        return s.out
    if path == "train":
        s.opt.zero_grad(set_to_none=True)
        images = [s.renderer.render(s.tf, s.density, cam) for cam in s.cams]
        loss = sum(((im - t) ** 2).mean() for im, t in zip(images, s.targets)) / len(images)
        loss.backward()
        grads = s.tf.grad, s.density.grad
        s.opt.step()
        return dict(images=[im.detach() for im in images], loss=loss.detach(), grad_tf=grads[0], grad_density=grads[1])
    if path == "batch":
        vr.vr_batch_launch(s.batch)
        return s.out
    if path == "stream":
        for t in range(s.case["steps"]):
            s.series.render_step(t, s.cams, s.outs[t])
        return s.outs
    if path == "insitu":
        vr.vr_volume_update(s.vols[0], s.field)
    vr.vr_set_camera(s.ctx, s.cams[0])
    if path == "mesh":
        vr.vr_render_mesh_frame(s.ctx, s.mesh, s.out)
    elif path == "partials":
        frame = vr.vr_render_partials(s.ctx, s.vols[0])
        vr.vr_composite(s.ctx, frame, s.out)
        vr.vr_frame_release(frame)
    else:
        vr.vr_render_frame(s.ctx, s.vols[0], s.out)
    return s.out


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------


def _basis(cam):
    f = np.array(cam["dir"], dtype=np.float64)
    f /= np.linalg.norm(f)
    r = np.cross(cam["up"], f)
    r /= np.linalg.norm(r)
    return f, r, np.cross(f, r)


def _rays(cam, px, py, xp):
    """Origins and directions (lists of x, y, z) of the pixels' rays; px, py in
    pixels, arrays of numpy or torch (xp), 64-bit."""
    f, r, u = _basis(cam)
    W, H = cam["width"], cam["height"]
    fx, fy = (px + 0.5) / W, (py + 0.5) / H
    if cam["ortho"]:
        a, b = (fx - 0.5) * cam["ortho_w"], (fy - 0.5) * cam["ortho_h"]
        return [cam["eye"][i] + a * r[i] + b * u[i] for i in range(3)], [f[i] + 0 * a for i in range(3)]
    th = math.tan(math.radians(cam["fovy_deg"]) / 2)
    sx, sy = (2 * fx - 1) * th * W / H, (2 * fy - 1) * th
    d = [f[i] + sx * r[i] + sy * u[i] for i in range(3)]
    n = xp.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    return [cam["eye"][i] + 0 * sx for i in range(3)], [x / n for x in d]


def _interval(dims, o, d, xp):
    """[t_in, t_out) of the rays in the volume's box; t_out <= t_in where they miss."""
    nmax = max(dims)
    t0, t1 = 0 * o[0], 0 * o[0] + 1e30
    for i in range(3):
        flat = d[i] == 0
        safe = xp.where(flat, 1 + 0 * d[i], d[i])
        ta, tb = -o[i] / safe, (dims[i] / nmax - o[i]) / safe
        out = flat & ((o[i] < 0) | (o[i] > dims[i] / nmax))
        t0 = xp.where(flat, t0, xp.maximum(t0, xp.minimum(ta, tb)))
        t1 = xp.where(out, 0 * t1, xp.where(flat, t1, xp.minimum(t1, xp.maximum(ta, tb))))
    return t0, t1


def work(case):
    """Bytes: the field's voxels (or the mesh's element data) once in their
    storage type, the images once, and for training the gradients and updated
    values. Flops: 66 for each lattice sample of the rays (position 8, trilinear
    30, classification 19, accumulation 8, termination 1; a training step takes
    three times that), the samples counted on a coarse grid of one orbit view;
    with early termination a ray is taken to end after ln(1/(1-ert)) / 0.025
    samples (0.025: the tables' mean opacity), per brick layer in sort-last."""
    c = case
    cams = _cameras(c, np.random.default_rng(0), 4)
    n = 0.0
    for cam in cams:
        gy, gx = np.meshgrid((np.arange(48) + 0.5) / 48 * c["H"] - 0.5, (np.arange(48) + 0.5) / 48 * c["W"] - 0.5,
                             indexing="ij")
        o, d = _rays(cam, gx, gy, np)
        t0, t1 = _interval(_dims(c), o, d, np)
        k = np.maximum(t1 - t0, 0) * max(_dims(c)) / c["step"]
        if c["ert"] < 1.0:
            layers = 1.0 if c["path"] == "cycle" else c["bricks"] ** (1 / 3)
            k = np.minimum(k, layers * -math.log(1 - c["ert"]) / 0.025)
        n += float(k.mean()) * c["W"] * c["H"] / len(cams)
    voxels = c["nx"] * c["ny"] * c["nz"]
    esize = 4 if c["storage"] == "f32" else 2
    image = c["W"] * c["H"] * 16
    if c["path"] == "train":
        return dict(bytes=voxels * 12 + 3 * c["views"] * image, flops=3 * 66 * n * c["views"])
    if c["path"] == "batch":
        return dict(bytes=c["volumes"] * (voxels * esize + c["views"] * image), flops=66 * n * c["volumes"] * c["views"])
    if c["path"] == "stream":
        return dict(bytes=c["steps"] * (2 * voxels * 4 + c["views"] * image), flops=66 * n * c["steps"] * c["views"])
    if c["path"] == "mesh":  # about 0.19 elements per voxel of the nominal lattice, 4 indices and 1/6 vertex each
        return dict(bytes=0.19 * voxels * 20 + image, flops=66 * n)
    if c["path"] == "insitu":
        return dict(bytes=voxels * (4 + 2 * esize) + image, flops=66 * n)
    return dict(bytes=voxels * esize + image, flops=66 * n)


# ---------------------------------------------------------------------------
# The same in 64 bits, from the definitions
# ---------------------------------------------------------------------------


def _brick_of(c, part):
    """Per cell, the id of its brick: int32 [nz, ny, nx] (any distinct ids)."""
    dims = _dims(c)
    if part["kind"] == "grid":
        ids = 0
        for a, (n, g) in enumerate(zip(dims, part["grid"])):
            at = torch.zeros(n, dtype=torch.int32, device="cuda")
            for j in range(1, g):
                at[n * j // g:] += 1
            ids = ids + (at * 1000 ** a).reshape([-1 if 2 - a == k else 1 for k in range(3)])
        return ids
    boxes = [[0, 0, 0, *dims]]
    for u in part["cut_fracs"]:  # the largest box, halved across its longest axis
        b = max(boxes, key=lambda q: (q[3] - q[0]) * (q[4] - q[1]) * (q[5] - q[2]))
        a = max(range(3), key=lambda i: b[3 + i] - b[i])
        cut = b[a] + math.floor(u * (b[3 + a] - b[a]) + 0.5)
        cut = min(max(cut, b[a] + 1), b[3 + a] - 1)
        high = list(b)
        high[a] = cut
        b[3 + a] = cut
        boxes.append(high)
    ids = torch.zeros((dims[2], dims[1], dims[0]), dtype=torch.int32, device="cuda")
    for i, b in enumerate(boxes):
        ids[b[2]:b[5], b[1]:b[4], b[0]:b[3]] = i
    return ids


def _samples(c, vol, tf, o, d, t_in, t_out, k0, n):
    """Colour [n, P, 3], opacity [n, P] and voxel positions of samples
    k0 .. k0+n-1 of P rays; the opacity is 0 from t_out on."""
    dims, nmax = _dims(c), max(_dims(c))
    k = torch.arange(k0, k0 + n, dtype=torch.float64, device="cuda")[:, None]
    t = t_in[None] + (k + 0.5) * (c["step"] / nmax)
    q = [(o[i][None] + t * d[i][None]) * nmax for i in range(3)]
    at = torch.stack([2 * q[i] / dims[i] - 1 for i in range(3)], dim=-1)
    v = torch.nn.functional.grid_sample(vol[None, None], at[None, :, :, None], mode="bilinear", padding_mode="border",
                                        align_corners=False)[0, 0, :, :, 0]
    x = v.clamp(0.0, 1.0) * (tf.shape[0] - 1)
    i = x.detach().floor().long().clamp(max=tf.shape[0] - 2)
    w = (x - i)[..., None]
    rgba = tf[i] * (1 - w) + tf[i + 1] * w
    alpha = rgba[..., 3]
    if c["opc"]:
        alpha = -torch.expm1(c["step"] / c["opc"] * torch.log1p(-alpha))
    return rgba[..., :3], torch.where(t < t_out[None], alpha, torch.zeros_like(alpha)), q


def _image64(c, part, vol, tf, cam, rows):
    """Rows [rows) of the image; vol [nz, ny, nx] and tf [n, 4] float64."""
    py, px = torch.meshgrid(torch.arange(*rows, dtype=torch.float64, device="cuda"),
                            torch.arange(c["W"], dtype=torch.float64, device="cuda"), indexing="ij")
    o, d = _rays(cam, px.reshape(-1), py.reshape(-1), torch)
    t_in, t_out = _interval(_dims(c), o, d, torch)
    P = t_in.numel()
    total = int(math.ceil(float((t_out - t_in).max().clamp(min=0)) * max(_dims(c)) / c["step"])) + 1
    zero = torch.zeros(P, dtype=torch.float64, device="cuda")
    C, T = torch.zeros((P, 3), dtype=torch.float64, device="cuda"), zero + 1
    ids = _brick_of(c, part) if c["ert"] < 1.0 and c["path"] != "cycle" else None
    Cb, Tb, cur = torch.zeros_like(C), zero + 1, torch.full((P,), -1, dtype=torch.int32, device="cuda")
    limit = 1.0 - float(np.float32(c["ert"]))
    n = max(1, min(64, (1 << 23) // P))
    for k0 in range(0, total, n):
        rgb, alpha, q = _samples(c, vol, tf, o, d, t_in, t_out, k0, n)
        if c["ert"] >= 1.0:
            keep = torch.cumprod(1 - alpha, dim=0)
            front = T * torch.cat([torch.ones_like(keep[:1]), keep[:-1]])
            C = C + ((front * alpha)[..., None] * rgb).sum(0)
            T = T * keep[-1]
            continue
        if ids is not None:
            cell = [q[i].floor().long().clamp(0, _dims(c)[i] - 1) for i in range(3)]
            brick = ids[cell[2], cell[1], cell[0]]
        for j in range(n):
            if ids is not None:  # a brick's own colour and transmittance, folded in when the ray leaves it
                new = brick[j] != cur
                C = torch.where(new[:, None], C + T[:, None] * Cb, C)
                T = torch.where(new, T * Tb, T)
                Cb = torch.where(new[:, None], torch.zeros_like(Cb), Cb)
                Tb = torch.where(new, zero + 1, Tb)
                cur = brick[j]
            a = torch.where(Tb > limit, alpha[j], zero)
            Cb = Cb + (Tb * a)[:, None] * rgb[j]
            Tb = Tb * (1 - a)
    C = C + T[:, None] * Cb
    return torch.cat([C, 1 - (T * Tb)[:, None]], dim=1).reshape(rows[1] - rows[0], c["W"], 4)


def _bands(c):
    """Row ranges of about a million rays (fewer where gradients are kept)."""
    n = max(1, (1 << (13 if c["path"] == "train" else 20)) // c["W"])
    return [(y, min(c["H"], y + n)) for y in range(0, c["H"], n)]


def exact(case, seed):
    c = case
    if c["path"] == "mesh":
        return None  # finding every sample's element in 64 bits takes minutes
    part, tf, cams, fields, _ = _scene(c, seed)
    tf64 = torch.from_numpy(tf).cuda().double()
    if c["path"] == "train":
        vol = fields[0].double().requires_grad_(True)
        tf64.requires_grad_(True)
        images, loss = [], 0.0
        for cam, target in zip(cams, _targets(c, seed)):
            bands = []
            for rows in _bands(c):
                im = _image64(c, part, vol, tf64, cam, rows)
                part_loss = ((im - target[rows[0]:rows[1]]) ** 2).sum() / (target.numel() * len(cams))
                part_loss.backward()
                loss += float(part_loss.detach())
                bands.append(im.detach())
            images.append(torch.cat(bands))
        return dict(images=images, loss=torch.tensor(loss, dtype=torch.float64), grad_tf=tf64.grad,
                    grad_density=vol.grad)
    stored = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[c["storage"]]
    frames = []
    for f in fields:
        vol = f.to(stored).double()
        frames.append([torch.cat([_image64(c, part, vol, tf64, cam, rows) for rows in _bands(c)]) for cam in cams])
    if c["path"] == "batch":
        return torch.stack([im for views in frames for im in views])
    return frames if c["path"] == "stream" else frames[0][0]
