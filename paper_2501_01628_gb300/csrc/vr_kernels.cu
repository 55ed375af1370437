// vr_kernels.cu -- CUDA kernels (sm_103a) of the brick pack and the per-brick
// emission-absorption march (the sort-last "over" composite is in
// vr_composite.cu, the ray-state cycling frame in vr_cycle.cu).
//
// Sec. 2.2 of arXiv:2501.01628: data is spatially distributed, each rank
// renders its share. Sec. 3/4: the per-rank images are composited into one
// framebuffer. The optical model is the standard emission-absorption one; the
// exact per-sample definitions are stated in include/vr.h.
#include <algorithm>

#include "vr_device.cuh"

namespace vr {
namespace {

using dev::Quad;
using dev::find_brick;

// ---------------------------------------------------------------------------
// Pack: global x-fastest float32 volume -> every brick's xy-quads (halo of one
// voxel, edge-clamped), converted to the storage type with round-to-nearest.
// One launch for all bricks; a block writes kPackChunk consecutive quads of one
// brick's storage (2x2x2 blocks of quads, blocks x-fastest), so a warp's writes
// are contiguous. Quads of the padding that rounds a brick's storage up to
// whole blocks are not written.
//
// Bound by memory: the volume once and the quads once (384^3: 0.23 + 0.93 GB). A
// thread writes the two quads (i, i + 1) that share a sector: six loads for eight
// voxels, one store (one quad in narrow bricks, see kPackNarrow). Its place in the
// storage is divided out once and then stepped by the brick's PackBrick::step, and all its
// loads are in flight together. 384^3 in 12 bricks: 0.190 ms, 6.0 TB/s (88% of
// a device copy); with one quad per thread 0.204, and with two 64-bit divisions per
// quad, most of its instructions, 0.263. A step that carried row by row took
// 64 turns in a brick one block wide (2048 x 2048 x 1: 52.5 us, now 27.4).
// ---------------------------------------------------------------------------
constexpr int kPackThreads = 256;
// two consecutive elements at an address aligned to both
__device__ __forceinline__ void store_pair(float4 *p, const float4 &a, const float4 &b)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}
__device__ __forceinline__ void store_pair(uint4 *p, const uint4 &a, const uint4 &b)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z),
                 "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
__device__ __forceinline__ void store_pair(uint2 *p, const uint2 &a, const uint2 &b)
{
    *reinterpret_cast<uint4 *>(p) = make_uint4(a.x, a.y, b.x, b.y);
}
// One block's chunk of a brick, E consecutive quads (1 or 2) per thread and round.
template <typename T, int E>
__device__ __forceinline__ void pack_chunk(const PackParams &p, const PackBrick &B, int chunk)
{
    constexpr int kRound = E * kPackThreads;         // quads per round of the block
    constexpr int kUnroll = kPackChunk / kRound;     // rounds, their loads in flight together
    static_assert(kRound / 8 == (E == 2 ? kPackStep : kPackStepNarrow), "2x2x2 blocks per round");
    using Q = typename Quad<T>::type;
    Q *dst = static_cast<Q *>(B.dst);
    const int qx = B.s[0] - 1, qy = B.s[1] - 1, nbx = B.s[0] / 2, nby = B.s[1] / 2;
    // a brick holds less than 2^31 quads; inverse of quad_index for the thread's first
    const unsigned q = static_cast<unsigned>(chunk) * kPackChunk + E * threadIdx.x;
    const unsigned q1 = static_cast<unsigned>(B.quads);
    const unsigned bl = q >> 3, rest = bl / static_cast<unsigned>(nbx);
    int bx = static_cast<int>(bl - rest * nbx), bz = static_cast<int>(rest / static_cast<unsigned>(nby));
    int by = static_cast<int>(rest) - bz * nby;
    const int ox = static_cast<int>(q & 1), oy = static_cast<int>((q >> 1) & 1), oz = static_cast<int>((q >> 2) & 1);
    constexpr int kPlanes = Quad<T>::octet ? 2 : 1;
    float v[kUnroll][kPlanes][2][E + 1];  // plane, row, x .. x + E
    bool in[kUnroll], both[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
        const int lx = 2 * bx + ox, ly = 2 * by + oy, lz = 2 * bz + oz;
        in[u] = q + u * kRound < q1 && lx < qx && ly < qy && lz < B.s[2];
        both[u] = in[u] && E == 2 && lx + 1 < qx;
        if (in[u]) {
            int gx[E + 1];
#pragma unroll
            for (int i = 0; i <= E; ++i) gx[i] = min(max(B.lo[0] + lx - 1 + i, 0), p.N[0] - 1);
#pragma unroll
            for (int k = 0; k < kPlanes; ++k) {  // plane lz, and for octets plane lz + 1
                const int gz = min(max(B.lo[2] + lz - 1 + k, 0), p.N[2] - 1);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int gy = min(max(B.lo[1] + ly - 1 + j, 0), p.N[1] - 1);
                    const float *row = p.src + (static_cast<long long>(gz) * p.N[1] + gy) * p.N[0];
#pragma unroll
                    for (int i = 0; i <= E; ++i) v[u][k][j][i] = __ldg(row + gx[i]);
                }
            }
        }
        bx += B.step[0];  // the next round's 2x2x2 block
        by += B.step[1];
        bz += B.step[2];
        if (bx >= nbx) {
            bx -= nbx;
            ++by;
        }
        if (by >= nby) {
            by -= nby;
            ++bz;
        }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
        if (!in[u]) continue;
        Q e[E];
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const float (&a)[2][E + 1] = v[u][0], (&b)[2][E + 1] = v[u][kPlanes - 1];
            if constexpr (Quad<T>::octet)
                e[i] = Quad<T>::make8(a[0][i], a[0][i + 1], a[1][i], a[1][i + 1], b[0][i], b[0][i + 1], b[1][i],
                                      b[1][i + 1]);
            else
                e[i] = Quad<T>::make(a[0][i], a[0][i + 1], a[1][i], a[1][i + 1]);
        }
        Q *d = dst + q + u * kRound;
        if (both[u]) store_pair(d, e[0], e[E - 1]);
        else *d = e[0];
    }
}

template <typename T>
__global__ void __launch_bounds__(kPackThreads) pack_kernel(const __grid_constant__ PackParams p)
{
    int lo = 0, hi = p.nb - 1;  // the block's brick (the same for all its threads)
    const int blk = blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.b[mid].block_begin <= blk) lo = mid;
        else hi = mid - 1;
    }
    const PackBrick &B = p.b[lo];
    if (B.narrow) pack_chunk<T, 1>(p, B, blk - B.block_begin);
    else pack_chunk<T, 2>(p, B, blk - B.block_begin);
}

// ---------------------------------------------------------------------------
// March: one thread per pixel of a brick's footprint. A block is a tile of
// 2x2 warp packets of pw x (32/pw) pixels (pw = p.pw: 4, 8 or 16). The transfer
// function is read as (T[i], T[i+1]-T[i]) pairs (the last difference is 0)
// through L1: one cached copy per SM instead of one shared-memory copy per block.
// ---------------------------------------------------------------------------
template <typename S, bool COUNT, int OPC, bool WIDE>
__device__ __forceinline__ void march_block(const MarchParams &p)
{
    // the composite launched after this march may start once every block of
    // this grid is running; it reads the masks and partials only after this
    // grid has completed
    asm volatile("griddepcontrol.launch_dependents;");
    // Launched as a programmatic dependent of the previous frame's composite
    // (pipelined frames), this grid reads only the bricks and the table before
    // it waits; its writes (masks, partials) go to a pool that the frame before
    // the previous one read. The mask blocks wait for the preceding grid's
    // completion (so this grid completes only after it); the march blocks wait
    // only for the composite that last read their pool (pool_ready). Outside
    // such a launch both waits return at once.
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
    if (rx >= B.rect[2] || ry >= B.rect[3]) return;
    const int px = B.rect[0] + rx, py = B.rect[1] + ry;

    unsigned long long executed = 0;
    dev::OwnedRun run;
    dev::owned_run(p, B, px, py, run);
    float4 c;
    if constexpr (WIDE) {
        float C0 = 0.f, C1 = 0.f, C2 = 0.f, T = 1.f;
        dev::march_accumulate_wide<S, OPC, kWideSamples>(p.data, B, run, p.tf, p.tf_scale, p.tf_bias, p.ntf, p.ert_T, C0,
                                                         C1, C2, T, p.opc);
        c = make_float4(C0, C1, C2, 1.0f - T);
    } else {
        c = dev::march_run<S, COUNT, OPC>(p.data, B, run, p.tf, p.tf_scale, p.tf_bias, p.ntf, p.ert_T, executed,
                                          p.opc, p.count_error);
    }
    // the composite reads the partial next: keep it in L2 ahead of the streamed bricks
    float4 *dst = p.partials + B.poff + static_cast<long long>(ry) * B.rect[2] + rx;
    if (!dev::pool_ready(p.pool_done, p.pool, p.pool_frame, p.count_error)) return;
    unsigned long long policy;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(policy));
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(dst), "f"(c.x), "f"(c.y),
                 "f"(c.z), "f"(c.w), "l"(policy)
                 : "memory");
    if (COUNT && executed) atomicAdd(p.sample_counter, executed);
}

template <typename S, bool COUNT, int OPC>
__global__ void __launch_bounds__(128) march_kernel(const __grid_constant__ MarchParams p)
{
    march_block<S, COUNT, OPC, false>(p);
}

// For launches that do not fill the chip (wide_march in vr_host.cpp has the rule
// and its figures).
template <typename S, int OPC>
__global__ void __launch_bounds__(128) march_wide_kernel(const __grid_constant__ MarchParams p)
{
    march_block<S, false, OPC, true>(p);
}

}  // namespace

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
cudaError_t launch_pack(const PackParams &p, int kind, cudaStream_t s)
{
    if (p.n_blocks <= 0) return cudaSuccess;
    switch (kind) {
    case kStoreF32: pack_kernel<float><<<p.n_blocks, kPackThreads, 0, s>>>(p); break;
    case kStoreBF16: pack_kernel<__nv_bfloat16><<<p.n_blocks, kPackThreads, 0, s>>>(p); break;
    case kStoreF16: pack_kernel<__half><<<p.n_blocks, kPackThreads, 0, s>>>(p); break;
    case kStoreBF16Oct: pack_kernel<dev::Octet<__nv_bfloat16>><<<p.n_blocks, kPackThreads, 0, s>>>(p); break;
    case kStoreF16Oct: pack_kernel<dev::Octet<__half>><<<p.n_blocks, kPackThreads, 0, s>>>(p); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_march(const MarchParams &p, int kind, cudaStream_t s, bool after_composite, bool wide)
{
    if (p.n_items + p.mask_blocks <= 0) return cudaSuccess;
    const int grid = p.n_items + p.mask_blocks;
    const bool count = p.sample_counter != nullptr;
    const int opc = opacity_kind(p.opc);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(128);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = after_composite ? 1 : 0;
#define VR_MARCH(T)                                                                                      \
    (wide && !count ? (opc ? cudaLaunchKernelEx(&cfg, march_wide_kernel<T, kOpacitySeries>, p)           \
                           : cudaLaunchKernelEx(&cfg, march_wide_kernel<T, kOpacityOff>, p))             \
     : count ? (opc ? cudaLaunchKernelEx(&cfg, march_kernel<T, true, kOpacitySeries>, p)                 \
                    : cudaLaunchKernelEx(&cfg, march_kernel<T, true, kOpacityOff>, p))                   \
     : opc == kOpacitySeries    ? cudaLaunchKernelEx(&cfg, march_kernel<T, false, kOpacitySeries>, p)    \
       : opc == kOpacityGeneral ? cudaLaunchKernelEx(&cfg, march_kernel<T, false, kOpacityGeneral>, p)   \
                                : cudaLaunchKernelEx(&cfg, march_kernel<T, false, kOpacityOff>, p))
    cudaError_t e = cudaErrorInvalidValue;
    switch (kind) {
    case kStoreF32: e = VR_MARCH(float); break;
    case kStoreBF16: e = VR_MARCH(__nv_bfloat16); break;
    case kStoreF16: e = VR_MARCH(__half); break;
    case kStoreBF16Oct: e = VR_MARCH(dev::Octet<__nv_bfloat16>); break;
    case kStoreF16Oct: e = VR_MARCH(dev::Octet<__half>); break;
    default: return cudaErrorInvalidValue;
    }
#undef VR_MARCH
    return e;
}

}  // namespace vr
