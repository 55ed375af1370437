// vr_cycle.cu -- CUDA kernel (sm_103a) of the ray-state cycling frame: one
// thread per pixel carries its ray's state through the bricks in visibility
// order (the ray-queue cycling of Sec. 2.2 and 3 of arXiv:2501.01628, restated
// for bricks on one GPU) and writes the final pixel; no partials, no composite.
#include <algorithm>

#include "vr_device.cuh"

namespace vr {
namespace {

// ---------------------------------------------------------------------------
// Ray-state cycling: one thread per image pixel carries (C, T) through the
// bricks in front-to-back order (the paper's ray-queue cycling, Sec. 2.2 and 3,
// where every ray visits every rank, restated for bricks on one GPU). No
// partial images and no composite; early termination is global.
// ---------------------------------------------------------------------------
// Bound by the latency of a ray's chain of loads (a launch has one thread per
// pixel, each with all its bricks' samples), so each ray keeps kWideSamples samples
// in flight, at 8 blocks per SM (36 to 48 bytes of spill stores). ms per frame, samples in
// pairs with the previous cell's quads reused / four in flight: 512^3, 36 bricks, 1080p
// 0.581 / 0.544; 256^3 at 1024^2 0.491 / 0.461, at 512^2 0.334 / 0.307, at 256^2 0.156 /
// 0.122; 64^3 at 256^2 0.0214 / 0.0198. (Six or eight in flight: 0.269 and 0.230 at 512^2,
// but 0.146 and 0.134 at 256^2, 0.481 and 0.476 at 1024^2.) Pairs stay where they are
// better (cycle_pairs in vr_host.cpp) and for counting, whose quads' bounds they check.
template <typename S, bool COUNT, int OPC, bool WIDE>
__device__ __forceinline__ void cycle_block(const MarchParams &p, float4 *out)
{
    // pipelined frames: the next frame's kernel may start once every block of
    // this grid is running, and this grid's image store waits for the
    // preceding grid (see march_kernel); outside such launches both are no-ops
    asm volatile("griddepcontrol.launch_dependents;");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int px = blockIdx.x * p.tile_w + (warp & 1) * p.pw + (lane & (p.pw - 1));
    const int py = blockIdx.y * p.tile_h + (warp >> 1) * (32 / p.pw) + lane / p.pw;
    if (px >= p.W || py >= p.H) return;
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, T = 1.f;
    unsigned long long executed = 0;
    dev::Ray ray;
    dev::ray_setup(p, px, py, ray);  // once per pixel; each brick only intersects it
    for (int j = 0; ray.hit && j < p.nb; ++j) {
        const BrickLaunch &B = p.b[p.order[j]];
        if (px < B.rect[0] || px >= B.rect[0] + B.rect[2] || py < B.rect[1] || py >= B.rect[1] + B.rect[3])
            continue;
        dev::OwnedRun run;
        dev::brick_run(p, B, ray, run);
        if constexpr (WIDE)
            dev::march_accumulate_wide<S, OPC, kWideSamples>(p.data, B, run, p.tf, p.tf_scale, p.tf_bias, p.ntf,
                                                             p.ert_T, C0, C1, C2, T, p.opc);
        else
            dev::march_accumulate<S, COUNT, OPC>(p.data, B, run, p.tf, p.tf_scale, p.tf_bias, p.ntf, p.ert_T, C0, C1,
                                                 C2, T, executed, p.opc, p.count_error);
        if (T <= p.ert_T) break;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    out[static_cast<long long>(py) * p.W + px] = make_float4(C0, C1, C2, 1.0f - T);
    if (COUNT && executed) atomicAdd(p.sample_counter, executed);
}

template <typename S, int OPC>
__global__ void __launch_bounds__(128, 8) march_cycle_kernel(const __grid_constant__ MarchParams p, float4 *out)
{
    cycle_block<S, false, OPC, true>(p, out);
}

template <typename S, bool COUNT, int OPC>
__global__ void __launch_bounds__(128) march_cycle_pairs_kernel(const __grid_constant__ MarchParams p, float4 *out)
{
    cycle_block<S, COUNT, OPC, false>(p, out);
}

}  // namespace

cudaError_t launch_march_cycle(const MarchParams &p, int kind, float4 *out, cudaStream_t s, bool after_frame,
                               bool pairs)
{
    if (p.W <= 0 || p.H <= 0) return cudaSuccess;
    const dim3 grid((p.W + p.tile_w - 1) / p.tile_w, (p.H + p.tile_h - 1) / p.tile_h);
    const bool count = p.sample_counter != nullptr;
    const int opc = opacity_kind(p.opc);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(128);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = after_frame ? 1 : 0;
#define VR_PAIRS(T, C, O) cudaLaunchKernelEx(&cfg, march_cycle_pairs_kernel<T, C, O>, p, out)
#define VR_WIDE(T, O) cudaLaunchKernelEx(&cfg, march_cycle_kernel<T, O>, p, out)
#define VR_CYCLE(T)                                                                                       \
    (count   ? (opc ? VR_PAIRS(T, true, kOpacitySeries) : VR_PAIRS(T, true, kOpacityOff))                  \
     : pairs ? (opc == kOpacitySeries    ? VR_PAIRS(T, false, kOpacitySeries)                              \
                : opc == kOpacityGeneral ? VR_PAIRS(T, false, kOpacityGeneral)                             \
                                         : VR_PAIRS(T, false, kOpacityOff))                                \
             : (opc == kOpacitySeries    ? VR_WIDE(T, kOpacitySeries)                                      \
                : opc == kOpacityGeneral ? VR_WIDE(T, kOpacityGeneral)                                     \
                                         : VR_WIDE(T, kOpacityOff)))
    cudaError_t e = cudaErrorInvalidValue;
    switch (kind) {
    case kStoreF32: e = VR_CYCLE(float); break;
    case kStoreBF16: e = VR_CYCLE(__nv_bfloat16); break;
    case kStoreF16: e = VR_CYCLE(__half); break;
    case kStoreBF16Oct: e = VR_CYCLE(dev::Octet<__nv_bfloat16>); break;
    case kStoreF16Oct: e = VR_CYCLE(dev::Octet<__half>); break;
    default: return cudaErrorInvalidValue;
    }
#undef VR_CYCLE
#undef VR_WIDE
#undef VR_PAIRS
    return e;
}

}  // namespace vr
