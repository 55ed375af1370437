// vr_mesh.cu -- march kernel (sm_103a) of tetrahedral-mesh volumes: the same
// per-brick emission-absorption runs on the global lattice as the voxel march
// (Sec. 2.2: each rank renders the samples of its share of the data), with the
// value taken from the brick's elements instead of a voxel grid.
//
// Per pixel and brick: the owned run [ka, kb] of lattice samples (ownership by
// the sample's cell, exactly as for voxel bricks), the element containing the
// first sample from the brick's start grid and a walk towards the sample, then a
// walk through face neighbours along the ray. In an element the value is linear
// in t and the ray leaves through the face whose barycentric coordinate falls to 0
// first; every sample with t up to that exit parameter is classified and
// accumulated from the element's line along the ray.
//
// Bound by instruction issue (68% of slots) at 23 of 32 lanes, since rays in a warp
// meet elements of different size. What was measured (1.3 M elements, 1280 x 720,
// ms per frame; 25 M elements at 1920 x 1080 2.11 -> 1.63):
//   0.540  a BVH point location per ray and brick, all samples of an element before
//          the next element, the record kept for them
//   0.530  five numbers per element instead of the record, one sample per iteration
//   0.461  start grid and walk instead of the BVH (which stays for the rays whose
//          walk or element steps do not end)
//   0.404  two samples per iteration, warp-converged, the BVH outside the loop (inside,
//          its registers spill in the loop: 0.551)
//   0.407  a walk ends only in an element that holds the sample (without that test, in
//          any element whose faces towards the sample have no neighbour: wrong values
//          where vertices are doubled, hang or are not merged inside a brick). Such
//          meshes pay for the BVH, ms with all rays located in it / now: a hundredth of
//          the elements cut in two but not their neighbours 1.18 / 0.92, a fifth
//          5.98 / 4.08, a vertex set per element 9.77 / 9.82 (10.83 with 128-bit record loads
//          in the BVH's leaves, which spill 12 bytes less and leave the rest 0.3% faster)
// Waiting until 4 to 24 lanes can step together: 0.452 to 0.461; lanes left to
// diverge: 0.596; 6, 7, 9 blocks per SM: 0.480, 0.500, 0.717 (spills).
#include "vr_device.cuh"
#include "vr_mesh.h"

namespace vr {
namespace {

using dev::find_brick;
using dev::ldg_v8;

// Smallest barycentric coordinate of q in the element (record at rec).
__device__ __forceinline__ float min_bary(const float4 *rec, float qx, float qy, float qz)
{
    float4 r0, r1, r2, r3;
    ldg_v8(rec, r0, r1);
    ldg_v8(rec + 2, r2, r3);
    const float dx = qx - r0.x, dy = qy - r0.y, dz = qz - r0.z;
    const float l1 = fmaf(r1.x, dx, fmaf(r1.y, dy, fmaf(r1.z, dz, 0.25f)));
    const float l2 = fmaf(r2.x, dx, fmaf(r2.y, dy, fmaf(r2.z, dz, 0.25f)));
    const float l3 = fmaf(r3.x, dx, fmaf(r3.y, dy, fmaf(r3.z, dz, 0.25f)));
    const float l0 = 1.0f - l1 - l2 - l3;
    return fminf(fminf(l0, l1), fminf(l2, l3));
}

// Brick-local element containing q: a stackless preorder walk of the brick's
// BVH (node indices only increase), keeping the element with the largest
// smallest-barycentric among the leaves whose boxes hold q and stopping at the
// first element that holds q. Returns -1 only when no leaf box holds q.
__device__ int locate(const MeshNode *nodes, const float4 *rec, float qx, float qy, float qz)
{
    constexpr float eps = 1.0e-3f;  // voxel units
    int best = -1;
    float best_m = -3.0e38f;
    const int end = nodes[0].skip;
    int node = 0;
    while (node < end) {
        const MeshNode nd = nodes[node];
        const bool in = qx >= nd.lo[0] - eps && qx <= nd.hi[0] + eps && qy >= nd.lo[1] - eps &&
                        qy <= nd.hi[1] + eps && qz >= nd.lo[2] - eps && qz <= nd.hi[2] + eps;
        if (in && nd.leaf == 0) {
            ++node;
            continue;
        }
        if (in) {
            const int first = nd.leaf & ((1 << 28) - 1), count = nd.leaf >> 28;
            for (int i = 0; i < count; ++i) {
                const float m = min_bary(rec + kMeshRec * (first + i), qx, qy, qz);
                if (m > best_m) {
                    best_m = m;
                    best = first + i;
                }
            }
            if (best_m >= 0.0f) return best;
        }
        node = nd.skip;
    }
    return best;
}

// A mask block writes one tile mask per thread.
static_assert(kMaskThreads == 128, "mask blocks are march blocks");
template <bool COUNT, int OPC>
__global__ void __launch_bounds__(128, 8) march_mesh_kernel(const __grid_constant__ MeshParams P)
{
    const MarchParams &p = P.m;
    // pipelined frames: the next grid may start once every block of this one
    // is running; the mask blocks write only after the preceding grid
    // completes, and the march blocks store their partials once the composite
    // that last read their pool is done (as in march_kernel); outside such
    // launches both waits return at once
    asm volatile("griddepcontrol.launch_dependents;");
    if (static_cast<int>(blockIdx.x) < p.mask_blocks) {  // the composite's tile masks
        asm volatile("griddepcontrol.wait;" ::: "memory");
        dev::write_tile_mask(blockIdx.x * kMaskThreads + threadIdx.x, p.mask_tiles_x, p.mask_tiles_y, p.nb, p.order,
                             [&](int b) { return make_int4(p.b[b].rect[0], p.b[b].rect[1], p.b[b].rect[2],
                                                           p.b[b].rect[3]); },
                             p.tile_mask);
        return;
    }
    const int item = blockIdx.x - p.mask_blocks;
    const int bi = find_brick(p, item);
    const BrickLaunch &B = p.b[bi];
    const int local = item - B.item_begin;
    const int ty = local / B.tiles_x, tx = local - ty * B.tiles_x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rx = tx * p.tile_w + (warp & 1) * p.pw + (lane & (p.pw - 1));
    const int ry = ty * p.tile_h + (warp >> 1) * (32 / p.pw) + lane / p.pw;
    const bool inside = rx < B.rect[2] && ry < B.rect[3];
    const int px = B.rect[0] + rx, py = B.rect[1] + ry;

    dev::Ray ray;
    dev::ray_setup(p, px, py, ray);
    dev::OwnedRun run;
    dev::brick_run(p, B, ray, run);
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, T = 1.f;
    unsigned long long executed = 0;
    const float4 *rec = P.rec + kMeshRec * P.rec_base[bi];
    const int4 *nbr = P.nbr + P.rec_base[bi];
    const float xmax = static_cast<float>(p.ntf - 1);
    // transfer-function pair i at tf + 2 i, addressed from the floor's bits
    const uintptr_t tf_base = reinterpret_cast<uintptr_t>(p.tf) - static_cast<uintptr_t>(dev::kFloorBits) * 32u;
    const float kh_end = static_cast<float>(run.kb) + 0.5f;
    float kh = static_cast<float>(run.ka) + 0.5f;   // the next sample, k + 1/2
    float t = fmaf(kh, p.dt, ray.t_in);
    // Along the ray an element is a linear function: table coordinate
    // x0 + slope (t - t0) up to the exit parameter, then the neighbour nx across
    // the exit face. So a lane carries five numbers of its element, not its record.
    float x0 = 0.f, slope = 0.f, t0 = 0.f, t_exit = -3.0e38f;
    int e = 0, nx = -1;   // -1: from the start grid
    int stall = 0, walk = 0;
    bool live = inside && run.ka <= run.kb;
    bool lost = false, located = false;
    for (;;) {
        while (__any_sync(0xffffffffu, live)) {
            if (live && t > t_exit) do {
                // the next sample lies beyond the element: the neighbour across the exit
                // face. At first, and after a boundary face, the element the start grid
                // gives for the sample's cell and from there a walk towards the sample.
                const float dvx = ray.dv[0], dvy = ray.dv[1], dvz = ray.dv[2];
                const float qx = fmaf(t, dvx, ray.ov[0]), qy = fmaf(t, dvy, ray.ov[1]), qz = fmaf(t, dvz, ray.ov[2]);
                if (nx < 0) {
                    const MeshGrid &g = P.grid[bi];
                    auto cell = [&](float q, int a) {
                        const float c = (q - static_cast<float>(B.lo[a])) * g.scale[a];
                        return min(max(static_cast<int>(c), 0), g.n[a] - 1);
                    };
                    const int cx = cell(qx, 0), cy = cell(qy, 1), cz = cell(qz, 2);
                    nx = __ldg(P.start + g.base + (static_cast<long long>(cz) * g.n[1] + cy) * g.n[0] + cx);
                    walk = kMeshWalkSteps;
                } else if (walk > 0 ? --walk == 0 : ++stall > kMeshStallSteps) {
                    lost = true;
                    live = false;
                    break;
                }
                e = nx;
                float4 r0, r1, r2, r3;
                ldg_v8(rec + kMeshRec * e, r0, r1);
                ldg_v8(rec + kMeshRec * e + 2, r2, r3);
                const int4 nb = __ldg(nbr + e);
                // exit parameter: the first decreasing barycentric coordinate to reach 0,
                // t + min lambda / -beta, the minimum by cross-multiplication
                const float dx = qx - r0.x, dy = qy - r0.y, dz = qz - r0.z;
                const float b1 = fmaf(r1.x, dvx, fmaf(r1.y, dvy, r1.z * dvz));
                const float b2 = fmaf(r2.x, dvx, fmaf(r2.y, dvy, r2.z * dvz));
                const float b3 = fmaf(r3.x, dvx, fmaf(r3.y, dvy, r3.z * dvz));
                const float g1 = fmaf(r1.x, dx, fmaf(r1.y, dy, r1.z * dz));
                const float g2 = fmaf(r2.x, dx, fmaf(r2.y, dy, r2.z * dz));
                const float g3 = fmaf(r3.x, dx, fmaf(r3.y, dy, r3.z * dz));
                const float l0 = 0.25f - (g1 + g2 + g3), l1 = 0.25f + g1, l2 = 0.25f + g2, l3 = 0.25f + g3;
                float num = 3.0e38f, den = 1.0f;
                nx = -1;
                auto exit_face = [&](float beta, float lam, int other) {
                    if (beta < 0.0f && lam * den < num * -beta) {
                        num = lam;
                        den = -beta;
                        nx = other;
                    }
                };
                exit_face(-(b1 + b2 + b3), l0, nb.x);
                exit_face(b1, l1, nb.y);
                exit_face(b2, l2, nb.z);
                exit_face(b3, l3, nb.w);
                t_exit = t + __fdividef(num, den);
                if (walk > 0) {  // on through the face the sample lies furthest behind, if any
                    float low = -kMeshInside;
                    int on = -2;  // none; -1: a face without a neighbour
                    auto behind = [&](float lam, int other) {
                        if (lam < low) {
                            low = lam;
                            on = other;
                        }
                    };
                    behind(l0, nb.x);
                    behind(l1, nb.y);
                    behind(l2, nb.z);
                    behind(l3, nb.w);
                    if (on == -2) {
                        walk = 0;
                        located = true;
                    } else {
                        // this element does not hold the sample; without a neighbour to
                        // go to, the walk ends in the BVH
                        nx = on < 0 ? e : on;
                        if (on < 0) walk = 1;
                        t_exit = -3.0e38f;
                    }
                }
                // a located element takes its first sample whatever the rounding says
                if (located) t_exit = fmaxf(t_exit, t);
                located = false;
                // value(q) = s_mean + sum_i (s_i - s_0) n_i . (q - c)
                const float s = fmaf(r1.w, g1, fmaf(r2.w, g2, fmaf(r3.w, g3, r0.w)));
                x0 = fmaf(s, p.tf_scale, p.tf_bias);
                slope = fmaf(r1.w, b1, fmaf(r2.w, b2, r3.w * b3)) * p.tf_scale;
                t0 = t;
            } while (false);
            __syncwarp();
            // up to two samples of the element, both table entries requested first
            const float tb = fmaf(kh + 1.0f, p.dt, ray.t_in);
            const bool one = live && !(t > t_exit), two = one && !(tb > t_exit) && kh < kh_end;
            auto entry = [&](float at, float &w, float4 &e0, float4 &de) {
                const float x = fminf(fmaxf(fmaf(slope, at - t0, x0), 0.0f), xmax);
                const float y = __fadd_rd(x, dev::kFloorOffset);
                w = x - (y - dev::kFloorOffset);
                ldg_v8(reinterpret_cast<const float4 *>(tf_base + static_cast<uintptr_t>(__float_as_uint(y)) * 32u),
                       e0, de);
            };
            auto accumulate = [&](float w, const float4 &e0, const float4 &de) {
                float al = fmaf(w, de.w, e0.w);
                if (OPC) al = dev::corrected_opacity<OPC>(al, p.opc);
                const float ta = T * al;
                C0 = fmaf(ta, fmaf(w, de.x, e0.x), C0);
                C1 = fmaf(ta, fmaf(w, de.y, e0.y), C1);
                C2 = fmaf(ta, fmaf(w, de.z, e0.z), C2);
                T = T - ta;
                if (COUNT) ++executed;
                live = !(T <= p.ert_T || kh >= kh_end);
                kh += 1.0f;
            };
            float wa, wb;
            float4 ea, da, eb, db;
            if (one) entry(t, wa, ea, da);
            if (two) entry(tb, wb, eb, db);
            if (one) {
                stall = 0;
                accumulate(wa, ea, da);
                t = tb;
                if (two && live) {
                    accumulate(wb, eb, db);
                    t = fmaf(kh, p.dt, ray.t_in);
                }
            }
        }
        if (!__any_sync(0xffffffffu, lost)) break;
        if (lost) {
            // too many steps without a sample (rounding near edges and vertices) or of a
            // walk, or a walk that came to a face without a neighbour: a point location
            nx = locate(P.nodes + P.node_base[bi], rec, fmaf(t, ray.dv[0], ray.ov[0]), fmaf(t, ray.dv[1], ray.ov[1]),
                        fmaf(t, ray.dv[2], ray.ov[2]));
            if (nx < 0) {
                atomicOr(P.error, 8);
                nx = e;
            }
            walk = stall = 0;
            located = live = true;
            lost = false;
        }
    }
    if (!inside) return;
    if (!dev::pool_ready(p.pool_done, p.pool, p.pool_frame, P.error)) return;
    p.partials[B.poff + static_cast<long long>(ry) * B.rect[2] + rx] = make_float4(C0, C1, C2, 1.0f - T);
    if (COUNT && executed) atomicAdd(p.sample_counter, executed);
}

}  // namespace

cudaError_t launch_march_mesh(const MeshParams &p, cudaStream_t s, bool after_frame)
{
    const int grid = p.m.n_items + p.m.mask_blocks;
    if (grid <= 0) return cudaSuccess;
    const bool count = p.m.sample_counter != nullptr;
    const int opc = opacity_kind(p.m.opc);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(128);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = after_frame ? 1 : 0;
    if (count) return opc ? cudaLaunchKernelEx(&cfg, march_mesh_kernel<true, kOpacitySeries>, p)
                          : cudaLaunchKernelEx(&cfg, march_mesh_kernel<true, kOpacityOff>, p);
    return opc == kOpacitySeries    ? cudaLaunchKernelEx(&cfg, march_mesh_kernel<false, kOpacitySeries>, p)
           : opc == kOpacityGeneral ? cudaLaunchKernelEx(&cfg, march_mesh_kernel<false, kOpacityGeneral>, p)
                                    : cudaLaunchKernelEx(&cfg, march_mesh_kernel<false, kOpacityOff>, p);
}

}  // namespace vr
