// vr_noalloc.cu -- vr_render_frame_noalloc: a whole frame (per-brick march +
// composite) that allocates no device memory.
//
// Who needs it: a renderer embedded in another program's GPU job -- an
// in-situ plugin inside a simulation that hands all device memory to its own
// pool allocator, or a caller on a latency-critical path where cudaMalloc and
// cudaFree (which synchronise the device) are not allowed. Such a caller owns
// the volume, the output image and the stream; the library supplies only the
// scratch: the per-brick partial images and the transfer-function table, kept in
// one file-scope device array of fixed size, VR_NOALLOC_SCRATCH_BYTES.
//
// The arithmetic is the same as vr_render_frame's. The march reads the
// caller's x-fastest float32 volume directly (edge-clamped trilinear, eight
// scalar loads per sample) instead of the library's packed bricks, because
// packing would need device memory.
#include <cmath>
#include <cstring>
#include <vector>

#include "vr_device.cuh"

namespace vr {
namespace {

// Scratch shared by every call on a device, held until the process exits:
// [0, kTfBytes) transfer-function pairs, then the composite's tile masks (one
// 16-byte mask per 32 x 8 tile of the image), then the partial images (float4).
constexpr size_t kScratchBytes = VR_NOALLOC_SCRATCH_BYTES;
constexpr size_t kTfBytes = 2 * 1024 * sizeof(float4);
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

// Work item of the march: a block's pixels, LANES lanes each.
__host__ __device__ constexpr int tile_w(int lanes) { return lanes == 1 ? 16 : lanes == 8 ? 4 : 8; }
__host__ __device__ constexpr int tile_h(int lanes) { return kMaskThreads / lanes / tile_w(lanes); }

// Device address of g_scratch on the current device. The host-side symbol is
// not a device address; the lookup is repeated on every call (it is cheap once
// the module is loaded), so a device reset or a re-created primary context
// never leaves a stale address behind.
cudaError_t scratch_address(void **out)
{
    *out = nullptr;
    return cudaGetSymbolAddress(out, g_scratch);
}

// March over the caller's global volume (p.data: x-fastest float32 with
// extents p.N). Ray setup, lattice, ownership and samples as in the
// packed-brick march; the grid's first blocks write the composite's tile masks.
//
// LANES neighbouring lanes take consecutive samples of one ray (see lanes_per_ray for
// how many). The transmittance runs through the lanes' samples in order (each lane
// repeats the chain over the group's opacities); the colours are summed per lane and
// added at the end. Bound by issue (52%) and the L1 data pipe (54%) where eight lanes
// fill the chip, by the latency of the voxels' loads else: at 9 blocks per SM (56 registers)
// all eight are in flight, at 10 and 12 the compiler puts some behind others (384^3 along z,
// 800 x 600, step 2, one lane: 432 / 623 / 885 us). With one lane per ray, four samples at a
// time gained nothing, keeping the cell's voxels and loading only new faces a
// fifth (divergent).
static_assert(kMaskThreads == 128, "mask blocks are march blocks");
template <int LANES>
__global__ void __launch_bounds__(128, 9) march_global_kernel(const __grid_constant__ MarchParams p)
{
    if (static_cast<int>(blockIdx.x) < p.mask_blocks) {
        dev::write_tile_mask(blockIdx.x * kMaskThreads + threadIdx.x, p.mask_tiles_x, p.mask_tiles_y, p.nb, p.order,
                             [&](int b) { return make_int4(p.b[b].rect[0], p.b[b].rect[1], p.b[b].rect[2],
                                                           p.b[b].rect[3]); },
                             p.tile_mask);
        return;
    }
    constexpr unsigned all = 0xffffffffu;
    const int item = blockIdx.x - p.mask_blocks;
    const BrickLaunch &B = p.b[dev::find_brick(p, item)];
    const int local = item - B.item_begin;
    const int ty = local / B.tiles_x, tx = local - ty * B.tiles_x;
    const int ray_id = threadIdx.x / LANES, j = threadIdx.x % LANES;
    int rx, ry;
    if constexpr (LANES == 1) {  // four 8 x 4 warp packets
        rx = tx * 16 + (ray_id >> 5 & 1) * 8 + (ray_id & 7);
        ry = ty * 8 + (ray_id >> 6) * 4 + (ray_id >> 3 & 3);
    } else {
        rx = tx * tile_w(LANES) + ray_id % tile_w(LANES);
        ry = ty * tile_h(LANES) + ray_id / tile_w(LANES);
    }
    const bool inside = rx < B.rect[2] && ry < B.rect[3];
    dev::Ray ray;
    dev::ray_setup(p, B.rect[0] + rx, B.rect[1] + ry, ray);
    dev::OwnedRun run;
    dev::brick_run(p, B, ray, run);
    if (!inside) run.kb = run.ka - 1;
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, T = 1.f;
    const float *vol = static_cast<const float *>(p.data);
    const int nx = static_cast<int>(p.N[0]), ny = static_cast<int>(p.N[1]), nz = static_cast<int>(p.N[2]);
    const long long plane = static_cast<long long>(nx) * ny;
    const float xmax = static_cast<float>(p.ntf - 1);
    float base[3], step[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        step[i] = ray.dv[i] * p.dt;
        base[i] = fmaf(ray.t_in, ray.dv[i], ray.ov[i] - 0.5f);  // global voxel-centre coordinates
    }
    // floor(v) (see dev::kFloorOffset) and the fraction
    auto cell = [](float v, float &w) {
        const float y = __fadd_rd(v, dev::kFloorOffset);
        w = v - (y - dev::kFloorOffset);
        return static_cast<int>(__float_as_uint(y) - dev::kFloorBits);
    };
    auto sample = [&](int k, float &a, float &r, float &g, float &b) {
        const float kh = static_cast<float>(k) + 0.5f;
        float wx, wy, wz;
        const int ix = cell(fmaf(kh, step[0], base[0]), wx);
        const int iy = cell(fmaf(kh, step[1], base[1]), wy);
        const int iz = cell(fmaf(kh, step[2], base[2]), wz);
        const int x0 = min(max(ix, 0), nx - 1), x1 = min(max(ix + 1, 0), nx - 1);
        const int y0 = min(max(iy, 0), ny - 1), y1 = min(max(iy + 1, 0), ny - 1);
        const int z0 = min(max(iz, 0), nz - 1), z1 = min(max(iz + 1, 0), nz - 1);
        const float *p0 = vol + z0 * plane, *p1 = vol + z1 * plane;
        const long long r0 = static_cast<long long>(y0) * nx, r1 = static_cast<long long>(y1) * nx;
        const float v000 = __ldg(p0 + r0 + x0), v100 = __ldg(p0 + r0 + x1), v010 = __ldg(p0 + r1 + x0),
                    v110 = __ldg(p0 + r1 + x1), v001 = __ldg(p1 + r0 + x0), v101 = __ldg(p1 + r0 + x1),
                    v011 = __ldg(p1 + r1 + x0), v111 = __ldg(p1 + r1 + x1);
        const float c00 = fmaf(wx, v100 - v000, v000), c10 = fmaf(wx, v110 - v010, v010);
        const float c01 = fmaf(wx, v101 - v001, v001), c11 = fmaf(wx, v111 - v011, v011);
        const float c0 = fmaf(wy, c10 - c00, c00), c1 = fmaf(wy, c11 - c01, c01);
        const float s = fmaf(wz, c1 - c0, c0);
        const float x = fminf(fmaxf(fmaf(s, p.tf_scale, p.tf_bias), 0.0f), xmax);
        float w;
        float4 e0, de;
        dev::ldg_v8(p.tf + 2 * cell(x, w), e0, de);
        r = fmaf(w, de.x, e0.x);
        g = fmaf(w, de.y, e0.y);
        b = fmaf(w, de.z, e0.z);
        a = fmaf(w, de.w, e0.w);
    };
    if constexpr (LANES == 1) {
        for (int k = run.ka; k <= run.kb; ++k) {
            float a, r, g, b;
            sample(k, a, r, g, b);
            const float ta = T * a;
            C0 = fmaf(ta, r, C0);
            C1 = fmaf(ta, g, C1);
            C2 = fmaf(ta, b, C2);
            T = T - ta;
            if (T <= p.ert_T) break;
        }
    } else {
        for (int k = run.ka; __any_sync(all, k <= run.kb); k += LANES) {
            float a = 0.f, r = 0.f, g = 0.f, b = 0.f;
            if (k + j <= run.kb) sample(k + j, a, r, g, b);
            // T before this lane's sample; the ray ends after the first sample with T <= ert_T
            float mine = T;
#pragma unroll
            for (int i = 0; i < LANES; ++i) {
                if (i == j) mine = T;
                const float ai = __shfl_sync(all, a, i, LANES);
                if (!(T <= p.ert_T)) T = T - T * ai;
            }
            if (k + j <= run.kb && !(mine <= p.ert_T)) {
                const float ta = mine * a;
                C0 = fmaf(ta, r, C0);
                C1 = fmaf(ta, g, C1);
                C2 = fmaf(ta, b, C2);
            }
            if (T <= p.ert_T) run.kb = k;  // the same for the ray's lanes
        }
#pragma unroll
        for (int i = 1; i < LANES; i += i) {
            C0 += __shfl_xor_sync(all, C0, i);
            C1 += __shfl_xor_sync(all, C1, i);
            C2 += __shfl_xor_sync(all, C2, i);
        }
    }
    if (inside && j == 0)
        p.partials[B.poff + static_cast<long long>(ry) * B.rect[2] + rx] = make_float4(C0, C1, C2, 1.0f - T);
}

// Lanes per ray of a call with `area` footprint pixels, its view direction's share along x
// (the volume's rows), the mean bound of a ray's samples in a brick, whether rays end
// early, and the row length.
//
// Few pixels leave the chip idle but for the longest rays, whose time falls with the
// lanes. Many fill it, and then lanes that share a ray only repeat its setup and chain and
// load other rows than their neighbours: one lane each is best, whose neighbours' pixels
// share rows. Rays along the rows turn that round: consecutive samples share them, pixels do
// not, the more so the longer the rows. us with 1 / 2 / 4 / 8 lanes:
//   along z   256^3, 30,000 pixels 159 / 132 / 107 / 131; 128^3 in 2 bricks, 121,200
//             160 / 166 / 168 / 205; 236,880 268 / 294 / 305 / 386; 256^3, 816,000
//             1621 / 1858 / 1969 / 2529, opaque with early termination 32 / 43 / 74 / 139
//             384^3 (long rays), 22,500 512 / 299 / 164 / 112
//   oblique   192^3 in 4 bricks, 110,210 363 / 214 / 151 / 119
//   along x   256^3, 163,216 1199 / 663 / 404 / 318; in 8 bricks, 445,264
//             1232 / 778 / 579 / 532; 128^3 in 2 bricks, 437,840 287 / 231 / 235 / 285,
//             opaque with early termination 30 / 34 / 50 / 88
// Over 711 calls (64^3 to 384^3, 900 to 1,000,000 pixels, five directions, steps of 1/2 and 2
// voxels) this choice takes about 0.86 of the time of eight lanes for all, 0.62 of the kernel's
// with one lane before lanes were shared, and is in no call slower than that.
int lanes_per_ray(double area, double along_x, double run, bool early, int row)
{
    if (area <= std::max(20000.0, along_x <= 0.4 ? 24.0 * run : 0.0)) return 8;
    if (along_x <= 0.4) return area <= 140000 ? 4 : area <= 300000 ? 2 : 1;
    if (area <= (early ? 125000 : 150000)) return 8;
    if (early) return area <= 160000 ? 4 : area <= 600000 ? 2 : 1;
    if (along_x > 0.7 && row >= 200 && area <= 300000) return 8;
    return area <= 1500.0 * run ? 4 : area <= 700000 ? 2 : 1;
}

bool normalize3(double v[3])
{
    const double l = std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    if (!(l > 0.0)) return false;
    v[0] /= l;
    v[1] /= l;
    v[2] /= l;
    return true;
}

}  // namespace
}  // namespace vr

using namespace vr;

extern "C" vr_status vr_render_frame_noalloc(const float *volume_dev, const int dims[3], const vr_partition *part,
                                             const float *tf_rgba, int n_tf, float vmin, float vmax,
                                             const vr_camera *cam, float step_voxels, float ert_alpha,
                                             float *out_rgba_dev, void *stream)
{
    if (!volume_dev || !dims || !part || !tf_rgba || !cam || !out_rgba_dev) return VR_ERR_ARG;
    if (n_tf < 2 || n_tf > 1024 || !(vmax > vmin) || !(step_voxels > 0.0f) || !(ert_alpha > 0.0f))
        return VR_ERR_ARG;
    // host-side plan: bricks, front-to-back order and footprint rectangles
    int nb = 0;
    if (vr_partition_boxes(dims, part, &nb, nullptr) != VR_OK || nb < 1 || nb > kMaxBricks) return VR_ERR_ARG;
    std::vector<int> boxes(6 * static_cast<size_t>(nb)), order(nb), rects(4 * static_cast<size_t>(nb));
    vr_partition_boxes(dims, part, &nb, boxes.data());
    if (vr_plan_view(dims, part, cam, order.data(), rects.data()) != VR_OK) return VR_ERR_ARG;

    static thread_local MarchParams mp;
    std::memset(&mp, 0, sizeof(mp));
    long long px = 0;
    for (int b = 0; b < nb; ++b) {
        BrickLaunch &L = mp.b[b];
        const int *bx = &boxes[6 * b];
        const int *r = &rects[4 * b];
        for (int a = 0; a < 3; ++a) {
            L.lo[a] = bx[a];
            L.hi[a] = bx[3 + a];
            L.own_lo[a] = bx[a] == 0 ? -INFINITY : static_cast<float>(bx[a]);
            L.own_hi[a] = bx[3 + a] == dims[a] ? INFINITY : static_cast<float>(bx[3 + a]);
        }
        std::memcpy(L.rect, r, sizeof(L.rect));
        L.poff = px;
        px += static_cast<long long>(r[2]) * r[3];
        px = (px + 7) & ~7LL;
    }
    // the frame's partial images must fit the fixed scratch
    const int tiles_x = (cam->width + kCompW - 1) / kCompW, tiles_y = (cam->height + kCompTileH - 1) / kCompTileH;
    const size_t mask_bytes = static_cast<size_t>(tiles_x) * tiles_y * sizeof(uint4);
    if (static_cast<size_t>(px) * sizeof(float4) + mask_bytes > kScratchBytes - kTfBytes) return VR_ERR_ARG;

    double f[3] = {cam->dir[0], cam->dir[1], cam->dir[2]}, r[3], u[3];
    if (!normalize3(f)) return VR_ERR_ARG;
    r[0] = cam->up[1] * f[2] - cam->up[2] * f[1];
    r[1] = cam->up[2] * f[0] - cam->up[0] * f[2];
    r[2] = cam->up[0] * f[1] - cam->up[1] * f[0];
    if (!normalize3(r)) return VR_ERR_ARG;
    u[0] = f[1] * r[2] - f[2] * r[1];
    u[1] = f[2] * r[0] - f[0] * r[2];
    u[2] = f[0] * r[1] - f[1] * r[0];
    const double th = std::tan(cam->fovy_deg * M_PI / 360.0);
    const double nmax = std::max(dims[0], std::max(dims[1], dims[2]));
    for (int a = 0; a < 3; ++a) {
        mp.eye[a] = static_cast<float>(cam->eye[a]);
        mp.r[a] = static_cast<float>(r[a]);
        mp.u[a] = static_cast<float>(u[a]);
        mp.f[a] = static_cast<float>(f[a]);
        mp.N[a] = static_cast<float>(dims[a]);
    }
    mp.tany = static_cast<float>(th);
    mp.tanx = static_cast<float>(th * static_cast<double>(cam->width) / cam->height);
    mp.ow = static_cast<float>(cam->ortho_w);
    mp.oh = static_cast<float>(cam->ortho_h);
    mp.ortho = cam->ortho ? 1 : 0;
    mp.W = cam->width;
    mp.H = cam->height;
    mp.inv_W = static_cast<float>(1.0 / cam->width);
    mp.inv_H = static_cast<float>(1.0 / cam->height);
    mp.nmax = static_cast<float>(nmax);
    const double dt = static_cast<double>(step_voxels) / nmax;
    mp.dt = static_cast<float>(dt);
    mp.inv_dt = static_cast<float>(1.0 / dt);
    mp.ert_T = ert_alpha < 1.0f ? static_cast<float>(1.0 - static_cast<double>(ert_alpha)) : -1.0f;
    const double scale = (n_tf - 1) / (static_cast<double>(vmax) - vmin);
    mp.tf_scale = static_cast<float>(scale);
    mp.tf_bias = static_cast<float>(-static_cast<double>(vmin) * scale);
    mp.ntf = n_tf;
    mp.nb = nb;
    double area = 0.0, samples = 0.0;
    for (int b = 0; b < nb; ++b) {
        const BrickLaunch &L = mp.b[b];
        const double px_b = static_cast<double>(L.rect[2]) * L.rect[3];
        double d2 = 0.0;
        for (int a = 0; a < 3; ++a) d2 += static_cast<double>(L.hi[a] - L.lo[a]) * (L.hi[a] - L.lo[a]);
        area += px_b;
        samples += px_b * std::sqrt(d2) / step_voxels;
    }
    const int lanes = lanes_per_ray(area, std::fabs(f[0]), area > 0.0 ? samples / area : 0.0, ert_alpha < 1.0f, dims[0]);
    int items = 0;
    for (int b = 0; b < nb; ++b) {
        BrickLaunch &L = mp.b[b];
        L.item_begin = items;
        L.tiles_x = (L.rect[2] + tile_w(lanes) - 1) / tile_w(lanes);
        items += L.tiles_x * ((L.rect[3] + tile_h(lanes) - 1) / tile_h(lanes));
    }
    mp.n_items = items;
    mp.data = volume_dev;

    // transfer-function pairs (T[i], T[i+1] - T[i]), last difference 0
    std::vector<float> pairs(8 * static_cast<size_t>(n_tf));
    for (int i = 0; i < n_tf; ++i)
        for (int c = 0; c < 4; ++c) {
            const float a = tf_rgba[4 * i + c];
            const float b = i + 1 < n_tf ? tf_rgba[4 * (i + 1) + c] : a;
            pairs[8 * i + c] = a;
            pairs[8 * i + 4 + c] = b - a;
        }

    void *scratch = nullptr;
    if (scratch_address(&scratch) != cudaSuccess || !scratch) return VR_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    float4 *tf_dev = static_cast<float4 *>(scratch);
    uint4 *masks = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(scratch) + kTfBytes);
    float4 *partials = reinterpret_cast<float4 *>(static_cast<unsigned char *>(scratch) + kTfBytes + mask_bytes);
    // pageable source: the copy has left `pairs` before cudaMemcpyAsync returns
    if (cudaMemcpyAsync(tf_dev, pairs.data(), pairs.size() * sizeof(float), cudaMemcpyHostToDevice, s) !=
        cudaSuccess)
        return VR_ERR_CUDA;
    mp.tf = tf_dev;
    mp.partials = partials;
    mp.tile_mask = masks;
    mp.mask_tiles_x = tiles_x;
    mp.mask_tiles_y = tiles_y;
    mp.mask_blocks = (tiles_x * tiles_y + kMaskThreads - 1) / kMaskThreads;
    for (int j = 0; j < nb; ++j) mp.order[j] = order[j];
    const int grid = mp.mask_blocks + items;
    switch (lanes) {
    case 1: march_global_kernel<1><<<grid, kMaskThreads, 0, s>>>(mp); break;
    case 2: march_global_kernel<2><<<grid, kMaskThreads, 0, s>>>(mp); break;
    case 4: march_global_kernel<4><<<grid, kMaskThreads, 0, s>>>(mp); break;
    default: march_global_kernel<8><<<grid, kMaskThreads, 0, s>>>(mp); break;
    }
    if (cudaGetLastError() != cudaSuccess) return VR_ERR_CUDA;
    // direct front-to-back composite with the existing kernel
    static thread_local CompositeParams cp;
    std::memset(&cp, 0, sizeof(cp));
    cp.W = cam->width;
    cp.H = cam->height;
    cp.nb = nb;
    cp.n_levels = 1;
    for (int j = 0; j < nb; ++j) cp.order[j] = order[j];
    for (int b = 0; b < nb; ++b) {
        std::memcpy(cp.rect[b], &rects[4 * b], 4 * sizeof(int));
        cp.poff[b] = mp.b[b].poff;
    }
    cp.partials = partials;
    cp.out = reinterpret_cast<float4 *>(out_rgba_dev);
    cp.tile_mask = masks;
    cp.tiles_x = tiles_x;
    cp.tiles_y = tiles_y;
    if (launch_composite(cp, s) != cudaSuccess) return VR_ERR_CUDA;
    return VR_OK;
}
