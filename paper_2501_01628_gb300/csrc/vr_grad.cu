// vr_grad.cu -- adjoint kernels of the frame: gradients of a loss on the image
// with respect to the transfer-function table and the voxel values.
//
// The paper renders only forward; its sort-last pipeline (Sec. 2.2 per-rank
// rendering, Sec. 3/4 compositing) is differentiated here with the chain rule.
// "Over" is associative, so a pixel is one sequence of samples through its
// bricks front to back, I = sum_k T_k a_k c_k, I_A = 1 - T_n, and its adjoint is
// one backward recurrence with lambda_T(n) = -dL/dI_A and lambda_C = dL/dI_rgb:
//     dL/dc_k = lambda_C T_k a_k, dL/da_k = T_k (lambda_C . c_k - lambda_T(k+1)),
//     lambda_T(k) = lambda_T(k+1) (1 - a_k) + a_k (lambda_C . c_k);
//   table lerp and trilinear weights as in the forward pass.
// No transmittance is ever obtained by dividing by (1 - a): each owned run is cut
// into groups of kGradGroup segments of kGradSeg samples, and
//   1. grad_groups_kernel composites each group alone, u = lambda_C . C and t,
//      keeping each sample's table coordinate and T at each segment's start;
//   2. grad_scan_kernel walks a pixel's groups through all its bricks: back to
//      front lambda_T <- t lambda_T + u, front to back T <- T t, leaving for each
//      group the lambda_T behind it and the T in front of it;
//   3. grad_samples_kernel walks a group back to front from its lambda_T (T of a
//      segment's samples again forward from the segment's start) and adds every
//      sample's gradients.
// Steps 1 and 3 are independent per group, so a launch has one thread per (pixel,
// brick, group) -- about seven times the threads of one per (pixel, brick), whose
// runs of different length left a third of the lanes and a quarter of the
// multiprocessors idle -- and every voxel is sampled once.
#include <algorithm>

#include "vr_device.cuh"
#include "vr_grad.h"

namespace vr {
namespace {

using dev::Quad;

// A brick's storage as the sample loops need it: the quad index of a cell is the
// separable form of quad_index on the floors' bit patterns (see
// dev::march_accumulate), clamped to the storage.
struct GradBrick {
    unsigned ay, az, c0, py, pz, dz, last;
    __device__ __forceinline__ explicit GradBrick(const BrickLaunch &B)
    {
        const unsigned nbx = static_cast<unsigned>(B.sx / 2), nby = static_cast<unsigned>(B.sy / 2);
        const unsigned nbz = static_cast<unsigned>(B.hi[2] - B.lo[2] + 3) / 2;
        last = nbx * nby * nbz * 8u - 1u;
        ay = 4u * nbx;
        az = 4u * nbx * nby;
        c0 = 0u - (4u + ay + az) * dev::kFloorBits;
        py = 2u - ay;
        pz = 4u - az;
        dz = 2u * az - 8u;
    }
};

// A sample's cell (floors as kFloorBits + cell) and weights.
struct GradCell {
    unsigned bx, by, bz;
    float wx, wy, wz;
    // quad index of the cell's plane k, and of plane k + 1
    __device__ __forceinline__ unsigned place(const GradBrick &G) const
    {
        unsigned c = bz * G.az + G.c0;
        c = by * G.ay + c;
        c = bx * 4u + c;
        c = (bx & 1u) * (0u - 3u) + c;
        c = (by & 1u) * G.py + c;
        return (bz & 1u) * G.pz + c;
    }
    __device__ __forceinline__ void quads(const GradBrick &G, unsigned &c, unsigned &c1) const
    {
        const unsigned at = place(G);
        c = min(at, G.last);
        c1 = min(at + 4u + (bz & 1u) * G.dz, G.last);
    }
    // the same two by the parity of their plane
    __device__ __forceinline__ void planes(const GradBrick &G, unsigned &even, unsigned &odd) const
    {
        unsigned c = by * G.ay + G.c0;
        c = bx * 4u + c;
        c = (bx & 1u) * (0u - 3u) + c;
        c = (by & 1u) * G.py + c;
        even = min(((bz + 1u) & ~1u) * G.az + c, G.last);
        odd = min((bz & ~1u) * G.az + c + 4u, G.last);
    }
};

// floor(v) as kFloorBits + floor and the fraction
__device__ __forceinline__ unsigned grad_floor(float v, float &w)
{
    const float y = __fadd_rd(v, dev::kFloorOffset);
    w = v - (y - dev::kFloorOffset);
    return __float_as_uint(y);
}

__device__ __forceinline__ void grad_cell(const dev::OwnedRun &run, float h, GradCell &q)
{
    q.bx = grad_floor(fmaf(h, run.step[0], run.base[0]), q.wx);
    q.by = grad_floor(fmaf(h, run.step[1], run.base[1]), q.wy);
    q.bz = grad_floor(fmaf(h, run.step[2], run.base[2]), q.wz);
}

// The table coordinate (not clamped) of sample kk.
template <typename S>
__device__ __forceinline__ float grad_value(const MarchParams &m, const typename Quad<S>::type *vox,
                                            const GradBrick &G, const dev::OwnedRun &run, int kk)
{
    GradCell q;
    grad_cell(run, static_cast<float>(kk) + 0.5f, q);
    unsigned c, c1;
    q.quads(G, c, c1);
    float4 a0, a1;
    if constexpr (Quad<S>::octet) {
        Quad<S>::load2(vox + c, a0, a1);
    } else {
        a0 = Quad<S>::load(vox + c);
        a1 = Quad<S>::load(vox + c1);
    }
    return fmaf(dev::trilinear<S>(a0, a1, q.wx, q.wy, q.wz), m.tf_scale, m.tf_bias);
}

// The table interval of coordinate x and the weight of its upper entry.
__device__ __forceinline__ int grad_interval(float x, float xmax, float &w)
{
    return static_cast<int>(grad_floor(fminf(fmaxf(x, 0.0f), xmax), w) - dev::kFloorBits);
}

// A thread's pixel of its block's (brick, tile) and its group.
struct GradItem {
    int b, px, py;
    long long pixel;   // index in the brick's rect
    long long area;
    int n;             // samples of the owned run
    int s0, s1;        // segments [s0, s1) of this thread
    dev::OwnedRun run;
    float4 g;          // dL/dI
};

// False where the thread has no segment. The first group's threads write their
// pixel's group count (COUNT).
template <bool COUNT>
__device__ __forceinline__ bool grad_item(const GradParams &p, GradItem &it)
{
    const MarchParams &m = p.m;
    it.b = dev::find_brick(m, blockIdx.x);
    const BrickLaunch &B = m.b[it.b];
    it.s0 = blockIdx.y * kGradGroup;
    if (it.s0 >= p.nseg[it.b]) return false;
    const int local = blockIdx.x - B.item_begin;
    const int ty = local / B.tiles_x, tx = local - ty * B.tiles_x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rx = tx * m.tile_w + (warp & 1) * m.pw + (lane & (m.pw - 1));
    const int ry = ty * m.tile_h + (warp >> 1) * (32 / m.pw) + lane / m.pw;
    if (rx >= B.rect[2] || ry >= B.rect[3]) return false;
    it.px = B.rect[0] + rx;
    it.py = B.rect[1] + ry;
    it.pixel = static_cast<long long>(ry) * B.rect[2] + rx;
    it.area = static_cast<long long>(B.rect[2]) * B.rect[3];
    it.g = __ldg(p.grad_img + static_cast<long long>(it.py) * m.W + it.px);
    it.n = 0;
    if (it.g.x != 0.f || it.g.y != 0.f || it.g.z != 0.f || it.g.w != 0.f) {
        dev::owned_run(m, B, it.px, it.py, it.run);
        it.n = it.run.kb - it.run.ka + 1;
    }
    const int segs = min((it.n + kGradSeg - 1) / kGradSeg, p.nseg[it.b]);
    it.s1 = min(it.s0 + kGradGroup, segs);
    if (COUNT && blockIdx.y == 0)
        p.count[B.poff + it.pixel] = static_cast<unsigned short>((segs + kGradGroup - 1) / kGradGroup);
    return it.s0 < it.s1;
}

// Step 1, bound by the march's loads and its stores of the coordinates: 256^3
// volume, 8 bricks, 512^2 view (35M samples) 0.22 ms. The samples come in batches of kGradSeg without a branch (past the end
// the last sample is repeated with opacity 0), so a batch's loads are in flight
// together. Keeping the coordinates (4 bytes per sample) instead of sampling the
// voxels again in step 3 measured the same time and half the code.
template <typename S>
__global__ void __launch_bounds__(128) grad_groups_kernel(const __grid_constant__ GradParams p)
{
    GradItem it;
    if (!grad_item<true>(p, it)) return;
    const MarchParams &m = p.m;
    const BrickLaunch &B = m.b[it.b];
    const typename Quad<S>::type *vox = static_cast<const typename Quad<S>::type *>(m.data) + B.base;
    const GradBrick G(B);
    const float xmax = static_cast<float>(m.ntf - 1);
    const long long seg0 = p.soff[it.b] + it.pixel;
    float u = 0.0f, T = 1.0f;
    for (int s = it.s0; s < it.s1; ++s) {
        // the last kept segment of an over-long run takes all the rest
        const int ks = it.run.ka + s * kGradSeg;
        const int k1 = s == p.nseg[it.b] - 1 ? it.run.kb : min(it.run.kb, ks + kGradSeg - 1);
        p.front[seg0 + s * it.area] = T;
        float *xs = p.x + p.soff[it.b] * kGradSeg + s * it.area * kGradSeg + it.pixel;
        for (int k0 = ks; k0 <= k1; k0 += kGradSeg) {
#pragma unroll
            for (int j = 0; j < kGradSeg; ++j) {
                const float x = grad_value<S>(m, vox, G, it.run, min(k0 + j, k1));
                if (k0 == ks) xs[j * it.area] = x;
                float w;
                const int ti = grad_interval(x, xmax, w);
                float4 e0, de;
                dev::ldg_v8(m.tf + 2 * ti, e0, de);
                const float a = k0 + j <= k1 ? fmaf(w, de.w, e0.w) : 0.0f;
                const float gc = it.g.x * fmaf(w, de.x, e0.x) + it.g.y * fmaf(w, de.y, e0.y) +
                                 it.g.z * fmaf(w, de.z, e0.z);
                const float ta = T * a;
                u = fmaf(ta, gc, u);
                T = T - ta;
            }
        }
    }
    p.group[p.goff[it.b] + blockIdx.y * it.area + it.pixel] = make_float2(u, T);
}

// Step 2, one thread per pixel of the band, bound by the latency of a few dependent
// loads per brick: 0.04 ms for a 512^2 view of 8 bricks (0.14 ms over segments
// of 8 samples, 0.48 ms with each load behind the previous store).
__global__ void __launch_bounds__(256) grad_scan_kernel(const __grid_constant__ GradParams p)
{
    __shared__ int s_brick[kMaxBricks];
    __shared__ int s_m;
    const MarchParams &m = p.m;
    const int tx0 = blockIdx.x * kCompW, ty0 = p.band_y0 + blockIdx.y * kCompH;
    const int tid = threadIdx.y * kCompW + threadIdx.x;
    if (tid < 32) {
        int n = 0;
        for (int j0 = 0; j0 < m.nb; j0 += 32) {
            const int j = j0 + tid;
            bool ov = false;
            int b = 0;
            if (j < m.nb) {
                b = m.order[j];
                const int *r = m.b[b].rect;
                ov = r[0] < tx0 + kCompW && tx0 < r[0] + r[2] && r[1] < ty0 + kCompH && ty0 < r[1] + r[3];
            }
            const unsigned bal = __ballot_sync(0xffffffffu, ov);
            if (ov) s_brick[n + __popc(bal & ((1u << tid) - 1u))] = b;
            n += __popc(bal);
        }
        if (tid == 0) s_m = n;
    }
    __syncthreads();
    const int px = tx0 + threadIdx.x, py = ty0 + threadIdx.y;
    if (px >= m.W || py >= p.band_y0 + p.band_h) return;
    // groups of the pixel in listed brick i: grp + s * area, s < the count
    auto at = [&](int i, float2 *&grp, long long &area) {
        const int b = s_brick[i];
        const int *r = m.b[b].rect;
        const int x = px - r[0], y = py - r[1];
        if (x < 0 || x >= r[2] || y < 0 || y >= r[3]) return 0;
        const long long pixel = static_cast<long long>(y) * r[2] + x;
        area = static_cast<long long>(r[2]) * r[3];
        grp = p.group + p.goff[b] + pixel;
        return static_cast<int>(p.count[m.b[b].poff + pixel]);
    };
    // kScan groups at a time: their loads are in flight together
    constexpr int kScan = 8;
    float lam = -p.grad_img[static_cast<long long>(py) * m.W + px].w;
    for (int i = s_m - 1; i >= 0; --i) {
        float2 *grp = nullptr;
        long long area = 0;
        for (int s = at(i, grp, area); s > 0; s -= kScan) {
            float2 v[kScan];
#pragma unroll
            for (int j = 0; j < kScan; ++j)
                if (s - 1 - j >= 0) v[j] = grp[(s - 1 - j) * area];
#pragma unroll
            for (int j = 0; j < kScan; ++j)
                if (s - 1 - j >= 0) {
                    grp[(s - 1 - j) * area].x = lam;
                    lam = fmaf(v[j].y, lam, v[j].x);
                }
        }
    }
    float T = 1.0f;
    for (int i = 0; i < s_m; ++i) {
        float2 *grp = nullptr;
        long long area = 0;
        const int n = at(i, grp, area);
        for (int s = 0; s < n; s += kScan) {
            float t[kScan];
#pragma unroll
            for (int j = 0; j < kScan; ++j)
                if (s + j < n) t[j] = grp[(s + j) * area].y;
#pragma unroll
            for (int j = 0; j < kScan; ++j)
                if (s + j < n) {
                    grp[(s + j) * area].y = T;
                    T *= t[j];
                }
        }
    }
}

__device__ __forceinline__ void red_v4(float4 *dst, const float (&v)[4])
{
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(v[0]), "f"(v[1]),
                 "f"(v[2]), "f"(v[3])
                 : "memory");
}

// Step 3. The samples of a segment are walked back to front; past the end the
// last sample is repeated with T and opacity 0, so nothing branches on the
// length and the segment's loads are in flight together. Gradients of
// consecutive samples in one cell, and in one table interval, are summed in
// registers before they are added to memory: the table with a 16-byte
// reduction per entry left behind into one of the copies (float atomics in shared
// memory are compare-and-swap loops), the voxels with a 16-byte reduction per
// quad left behind into quads laid out as the brick's own (QUADS;
// grad_voxels_kernel then adds them to the voxels), or with one reduction per
// corner on the original volume's indexing (halo copies alias their neighbours'
// voxels).
// Bound by issue (64% of slots) at 26.5 of 32 lanes, then by the reductions on their
// way to L2 (39% of its rate): 0.32 ms for a 512^2 view of a 256^3 volume. A whole backward of 512^2 views of a 256^3 volume: 0.703 ms
// with the sums by parity of their place, 0.743 ms with them moved between lower and
// upper (0.37 ms here); one thread per run with shared-memory table gradients and
// three samplings took 2.1 ms. 4 and 6 blocks per SM: 0.718 and 0.743 ms; segments of 4
// samples 0.76, groups of 6 and 16 segments 0.718 and 0.701 (0.21 against 0.16 for a 256^2
// view of 128^3).
template <bool QUADS>
__global__ void __launch_bounds__(128, 5) grad_samples_kernel(const __grid_constant__ GradParams p)
{
    GradItem it;
    if (!grad_item<false>(p, it)) return;
    const MarchParams &m = p.m;
    const BrickLaunch &B = m.b[it.b];
    if (it.n > kGradMaxRun) {
        atomicOr(p.error, 1);
        return;
    }
    const GradBrick G(B);
    const float xmax = static_cast<float>(m.ntf - 1);
    // neighbouring lanes, whose samples often share an interval, add into different copies
    const unsigned which = ((blockIdx.x + blockIdx.y) * kGradLaneCopies + threadIdx.x % kGradLaneCopies) % kGradCopies;
    float4 *copy = reinterpret_cast<float4 *>(p.tf_copies) + static_cast<long long>(which) * (m.ntf + 1);
    const bool voxels = QUADS || p.grad_vol;
    float4 *gquads = QUADS ? p.grad_quads + B.base : nullptr;
    // Sums in registers by the parity of their place: of the two table entries of an
    // interval, and of the two planes of a cell, one is even and one is odd, so that
    // what the next sample shares stays where it is and what it leaves behind goes.
    int cur_e = -1, cur_o = -1;  // entries being summed (negative: none)
    float tab_e[4], tab_o[4], pl_e[4], pl_o[4];
    unsigned quad_e = ~0u, quad_o = ~0u;          // QUADS: quads of the planes (~0: none)
    unsigned cur_x = 0, cur_y = 0, cur_z = 0;     // else: the cell's floors (0: no cell)
#pragma unroll
    for (int c = 0; c < 4; ++c) tab_e[c] = tab_o[c] = pl_e[c] = pl_o[c] = 0.0f;
    auto leave = [&](float4 *dst, bool any, float (&sum)[4]) {
        if (any) red_v4(dst, sum);
#pragma unroll
        for (int c = 0; c < 4; ++c) sum[c] = 0.0f;
    };
    auto leave_cell = [&]() {  // the eight corners of (cur_x, cur_y, cur_z) into the voxels
        const int i = static_cast<int>(cur_x - dev::kFloorBits), j = static_cast<int>(cur_y - dev::kFloorBits),
                  k = static_cast<int>(cur_z - dev::kFloorBits);
        const int gx0 = min(max(B.lo[0] - 1 + i, 0), p.N[0] - 1), gx1 = min(max(B.lo[0] + i, 0), p.N[0] - 1);
        const int gy0 = min(max(B.lo[1] - 1 + j, 0), p.N[1] - 1), gy1 = min(max(B.lo[1] + j, 0), p.N[1] - 1);
        const int ge = min(max(B.lo[2] - 1 + ((k + 1) & ~1), 0), p.N[2] - 1);
        const int go = min(max(B.lo[2] - 1 + (k | 1), 0), p.N[2] - 1);
        const long long nx = p.N[0], nxy = static_cast<long long>(p.N[0]) * p.N[1];
        float *gv = p.grad_vol;
        atomicAdd(gv + ge * nxy + gy0 * nx + gx0, pl_e[0]);
        atomicAdd(gv + ge * nxy + gy0 * nx + gx1, pl_e[1]);
        atomicAdd(gv + ge * nxy + gy1 * nx + gx0, pl_e[2]);
        atomicAdd(gv + ge * nxy + gy1 * nx + gx1, pl_e[3]);
        atomicAdd(gv + go * nxy + gy0 * nx + gx0, pl_o[0]);
        atomicAdd(gv + go * nxy + gy0 * nx + gx1, pl_o[1]);
        atomicAdd(gv + go * nxy + gy1 * nx + gx0, pl_o[2]);
        atomicAdd(gv + go * nxy + gy1 * nx + gx1, pl_o[3]);
    };
    // on to cell q
    auto next_cell = [&](const GradCell &q) {
        if constexpr (QUADS) {
            unsigned e, o;
            q.planes(G, e, o);
            if (e != quad_e) {
                leave(gquads + quad_e, quad_e != ~0u, pl_e);
                quad_e = e;
            }
            if (o != quad_o) {
                leave(gquads + quad_o, quad_o != ~0u, pl_o);
                quad_o = o;
            }
        } else if (q.bx != cur_x || q.by != cur_y || q.bz != cur_z) {
            if (cur_x != 0) leave_cell();
#pragma unroll
            for (int c = 0; c < 4; ++c) pl_e[c] = pl_o[c] = 0.0f;
            cur_x = q.bx;
            cur_y = q.by;
            cur_z = q.bz;
        }
    };
    const unsigned area = static_cast<unsigned>(it.area);  // a band's coordinates stay below 2^32
    const float2 ends = p.group[p.goff[it.b] + blockIdx.y * it.area + it.pixel];
    float lamT = ends.x;
    for (int s = it.s1 - 1; s >= it.s0; --s) {
        const int k0 = it.run.ka + s * kGradSeg, left = it.run.kb - k0;  // samples 0 .. min(left, kGradSeg - 1)
        const float h0 = static_cast<float>(k0) + 0.5f;
        const float *x = p.x + p.soff[it.b] * kGradSeg + s * it.area * kGradSeg + it.pixel;
        float T = ends.y * p.front[p.soff[it.b] + s * it.area + it.pixel];
        float xs[kGradSeg], Ts[kGradSeg];
#pragma unroll
        for (int j = 0; j < kGradSeg; ++j) xs[j] = __ldcs(x + static_cast<unsigned>(min(j, left)) * area);
#pragma unroll
        for (int j = 0; j < kGradSeg; ++j) {
            float w;
            const float *e = reinterpret_cast<const float *>(m.tf + 2 * grad_interval(xs[j], xmax, w));
            Ts[j] = j <= left ? T : 0.0f;
            T = T - T * fmaf(w, __ldg(e + 7), __ldg(e + 3));
        }
#pragma unroll
        for (int j = kGradSeg - 1; j >= 0; --j) {
            float w, xj = xs[j];
            asm volatile("" : "+f"(xj));  // weights again, not kept in registers from the loop above
            const int ti = grad_interval(xj, xmax, w);
            float4 e0, de;
            dev::ldg_v8(m.tf + 2 * ti, e0, de);
            const float a = j <= left ? fmaf(w, de.w, e0.w) : 0.0f;
            const float gc = it.g.x * fmaf(w, de.x, e0.x) + it.g.y * fmaf(w, de.y, e0.y) +
                             it.g.z * fmaf(w, de.z, e0.z);
            const float ta = Ts[j] * a;
            const float g4[4] = {it.g.x * ta, it.g.y * ta, it.g.z * ta, Ts[j] * (gc - lamT)};
            lamT = lamT * (1.0f - a) + a * gc;
            // table: rgba = (1-w) T[i] + w T[i+1]
            const int ie = (ti + 1) & ~1, io = ti | 1;
            if (ie != cur_e) {
                leave(copy + cur_e, cur_e >= 0, tab_e);
                cur_e = ie;
            }
            if (io != cur_o) {
                leave(copy + cur_o, cur_o >= 0, tab_o);
                cur_o = io;
            }
            const float w0 = 1.0f - w, we = ti & 1 ? w : w0, wo = ti & 1 ? w0 : w;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                tab_e[c] = fmaf(we, g4[c], tab_e[c]);
                tab_o[c] = fmaf(wo, g4[c], tab_o[c]);
            }
            // scalar: ds = (g . (T[i+1] - T[i])) dx/ds where the table coordinate is not clamped
            if (voxels && j <= left && xj > 0.0f && xj < xmax) {
                const float ds = (g4[0] * de.x + g4[1] * de.y + g4[2] * de.z + g4[3] * de.w) * m.tf_scale;
                GradCell q;
                grad_cell(it.run, h0 + static_cast<float>(j), q);
                next_cell(q);
                const float ux = 1.0f - q.wx, uy = 1.0f - q.wy, uz = 1.0f - q.wz;
                const bool odd = q.bz & 1u;
                const float de_ = ds * (odd ? q.wz : uz), do_ = ds * (odd ? uz : q.wz);
                pl_e[0] = fmaf(de_, ux * uy, pl_e[0]);
                pl_e[1] = fmaf(de_, q.wx * uy, pl_e[1]);
                pl_e[2] = fmaf(de_, ux * q.wy, pl_e[2]);
                pl_e[3] = fmaf(de_, q.wx * q.wy, pl_e[3]);
                pl_o[0] = fmaf(do_, ux * uy, pl_o[0]);
                pl_o[1] = fmaf(do_, q.wx * uy, pl_o[1]);
                pl_o[2] = fmaf(do_, ux * q.wy, pl_o[2]);
                pl_o[3] = fmaf(do_, q.wx * q.wy, pl_o[3]);
            }
        }
    }
    if constexpr (QUADS) {
        if (quad_e != ~0u) red_v4(gquads + quad_e, pl_e);
        if (quad_o != ~0u) red_v4(gquads + quad_o, pl_o);
    } else {
        if (cur_x != 0) leave_cell();
    }
    if (cur_e >= 0) red_v4(copy + cur_e, tab_e);
    if (cur_o >= 0) red_v4(copy + cur_o, tab_o);
}

// Step 4 (QUADS): every haloed voxel of every brick sums its share of the four
// quads that hold it and adds it to the volume's voxel (halo copies alias their
// neighbours' voxels). A warp takes 31 voxels along x (lane 0 has the quad on their
// left) and kGradVoxelRows rows: a quad is loaded once, the row below's half stays in
// registers and the left neighbour's comes from the lane below, and the quads' index
// is stepped. Bound by HBM:
// 0.069 ms for 256^3 (0.28 GB of quads, 0.35 GB read with the voxels, 73% of the peak
// DRAM rate); one row per warp, both quads of a voxel loaded and indexed anew, took
// 0.080 ms.
__global__ void __launch_bounds__(256) grad_voxels_kernel(const __grid_constant__ GradVoxelParams p)
{
    int lo = 0, hi = p.nb - 1;
    const int task = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (task >= p.n_tasks) return;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.b[mid].task_begin <= task) lo = mid;
        else hi = mid - 1;
    }
    const GradVoxelBrick &B = p.b[lo];
    const int local = task - B.task_begin;
    const int nx = grad_voxel_chunks(B.s[0]), ny = grad_voxel_row_sets(B.s[1]);
    const int yz = local / nx, cx = local - yz * nx, lz = yz / ny, y0 = (yz - lz * ny) * kGradVoxelRows;
    const int lx = cx * 31 - 1 + lane;
    const int qx = B.s[0] - 1, qy = B.s[1] - 1, nbx = B.s[0] / 2, nby = B.s[1] / 2;
    const bool quad = lx >= 0 && lx < qx, voxel = lane > 0 && lx < B.s[0];
    const float4 *at = p.quads + B.base + quad_index(quad ? lx : 0, y0, lz, nbx, nby);  // row y0 is even
    const int gx = min(max(B.lo[0] + lx - 1, 0), p.N[0] - 1);
    const int gz = min(max(B.lo[2] + lz - 1, 0), p.N[2] - 1);
    float *out = p.grad_vol + static_cast<long long>(gz) * p.N[1] * p.N[0] + gx;
    const long long down = 8LL * nbx;  // two rows on
    float bz = 0.0f, bw = 0.0f;        // the row below's quad
    if (quad && y0 > 0) {
        const float4 b = __ldg(at + 2 - down);
        bz = b.z;
        bw = b.w;
    }
    const int y1 = min(y0 + kGradVoxelRows, B.s[1]);
#pragma unroll 4
    for (int ly = y0; ly < y1; ++ly) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (quad && ly < qy) a = __ldg(at + ((ly - y0) >> 1) * down + 2 * (ly & 1));
        const float own = a.x + bz, next = a.y + bw;
        const float v = own + __shfl_up_sync(0xffffffffu, next, 1);
        bz = a.z;
        bw = a.w;
        const int gy = min(max(B.lo[1] + ly - 1, 0), p.N[1] - 1);
        if (voxel && v != 0.0f) atomicAdd(out + static_cast<long long>(gy) * p.N[0], v);
    }
}

// The copies of the table gradient, summed and added: a block takes 32
// consecutive values of grad_tf, a warp every eighth copy.
__global__ void __launch_bounds__(256) grad_table_kernel(const float *copies, int ntf, float *grad_tf)
{
    __shared__ float s_sum[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int v = blockIdx.x * 32 + lane;
    float sum = 0.0f;
    if (v < 4 * ntf) {
#pragma unroll
        for (int k = warp; k < kGradCopies; k += 8) {
            sum += copies[static_cast<long long>(k) * 4 * (ntf + 1) + v];
        }
    }
    s_sum[warp][lane] = sum;
    __syncthreads();
    if (warp == 0 && v < 4 * ntf) {
        float t = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += s_sum[k][lane];
        if (t != 0.0f) atomicAdd(grad_tf + v, t);
    }
}

__global__ void __launch_bounds__(128) table_pairs_kernel(const float4 *rgba, int n, float4 *pairs)
{
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= n) return;
    const float4 a = rgba[i], b = rgba[min(i + 1, n - 1)];
    pairs[2 * i] = a;
    pairs[2 * i + 1] = i + 1 < n ? make_float4(b.x - a.x, b.y - a.y, b.z - a.z, b.w - a.w)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
}

}  // namespace

cudaError_t launch_table_pairs(const float4 *rgba, int n, float4 *pairs, cudaStream_t s)
{
    table_pairs_kernel<<<(n + 127) / 128, 128, 0, s>>>(rgba, n, pairs);
    return cudaGetLastError();
}

cudaError_t launch_grad_groups(const GradParams &p, int kind, int groups, cudaStream_t s)
{
    if (p.m.n_items <= 0 || groups <= 0) return cudaSuccess;
    const dim3 grid(p.m.n_items, groups);
    switch (kind) {
    case kStoreF32: grad_groups_kernel<float><<<grid, 128, 0, s>>>(p); break;
    case kStoreBF16: grad_groups_kernel<__nv_bfloat16><<<grid, 128, 0, s>>>(p); break;
    case kStoreF16: grad_groups_kernel<__half><<<grid, 128, 0, s>>>(p); break;
    case kStoreBF16Oct: grad_groups_kernel<dev::Octet<__nv_bfloat16>><<<grid, 128, 0, s>>>(p); break;
    case kStoreF16Oct: grad_groups_kernel<dev::Octet<__half>><<<grid, 128, 0, s>>>(p); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_grad_scan(const GradParams &p, cudaStream_t s)
{
    if (p.m.n_items <= 0) return cudaSuccess;
    const dim3 grid((p.m.W + kCompW - 1) / kCompW, (p.band_h + kCompH - 1) / kCompH), block(kCompW, kCompH);
    grad_scan_kernel<<<grid, block, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_grad_samples(const GradParams &p, int groups, cudaStream_t s)
{
    if (p.m.n_items <= 0 || groups <= 0) return cudaSuccess;
    const dim3 grid(p.m.n_items, groups);
    if (p.grad_quads) grad_samples_kernel<true><<<grid, 128, 0, s>>>(p);
    else grad_samples_kernel<false><<<grid, 128, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_grad_voxels(const GradVoxelParams &p, cudaStream_t s)
{
    if (p.n_tasks <= 0) return cudaSuccess;
    grad_voxels_kernel<<<(p.n_tasks + 7) / 8, 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_grad_table(const float *tf_copies, int ntf, float *grad_tf, cudaStream_t s)
{
    grad_table_kernel<<<(4 * ntf + 31) / 32, 256, 0, s>>>(tf_copies, ntf, grad_tf);
    return cudaGetLastError();
}

}  // namespace vr
