// vr_internal.h -- structures shared by the host runtime (vr_host.cpp) and the
// CUDA kernels (vr_kernels.cu). Not part of the public ABI.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/vr.h"

namespace vr {

constexpr int kMaxBricks = VR_MAX_BRICKS;

// Opacity correction for a step of `ratio` reference steps, 1 - (1 - a)^ratio,
// where |a| <= cut by the binomial series a (c[0] + a (c[1] + ...)), c[k] =
// (-1)^k binom(ratio, k + 1). The cut is where the terms left out reach 2^-27 of
// the result: 0.19 for ratios near 0, 0.25 at most. There is none (-1) for ratios
// above 2, whose terms cancel more, and for tables that reach above it, so that
// the lanes of a warp do not part (256^3 in 12 bricks, 1280 x 720, f32: table up
// to 0.05, general formula 241 us / series 212 us; table up to 1, lanes on both
// sides 256 us / general formula for all 241 us). Series against formula, table up
// to 0.05: f16 octets 220 / 181 us, ray-state cycling 367 / 276 us, staged march of
// 128^3 114 / 93 us, batch of four 512^2 views of it 323 / 266 us, mesh of its size
// 280 / 235 us.
constexpr int kOpacityTerms = 10;
struct OpacityStep {
    float ratio;  // step / reference step (1: off)
    float cut;
    float c[kOpacityTerms];
};
// Template argument of the march kernels: no correction, the general formula for
// all samples, or the series up to the cut. The last gives any launch's image; the
// second, without the branch, is for launches without a cut: the branch keeps two
// samples' formulas from overlapping (241 / 257 us in sort-last frames; where
// samples are not in pairs, or one frame is too short to matter, there is none).
enum { kOpacityOff = 0, kOpacityGeneral = 1, kOpacitySeries = 2 };
inline int opacity_kind(const OpacityStep &o)
{
    return o.ratio == 1.0f ? kOpacityOff : o.cut < 0.0f ? kOpacityGeneral : kOpacitySeries;
}
// alpha_max: the largest |opacity| in the table (infinity: not known).
inline OpacityStep opacity_step(float ratio, float alpha_max)
{
    OpacityStep o = {};
    o.ratio = ratio;
    o.cut = -1.0f;
    if (!(ratio > 0.0f && ratio <= 2.0f && ratio != 1.0f)) return o;
    const double r = ratio;
    double c = r;
    for (int k = 0; k < kOpacityTerms; ++k) {
        o.c[k] = static_cast<float>(c);
        c *= (k + 1 - r) / (k + 2);
    }
    // the terms left out: at most |c| a^10 (1 + a + a^2 + ...) of a, a <= 1/4
    const float cut = static_cast<float>(std::fmin(
        0.25, std::pow(0.75 * r / 134217728.0 / std::fmax(std::fabs(c), 1e-30), 1.0 / kOpacityTerms)));
    if (alpha_max <= cut) o.cut = cut;
    return o;
}

// Brick storage kind: the storage type and the cell layout -- xy-quads (four
// voxels of one plane per element; two loads per sample) or, for the 16-bit
// types, octets (both planes of a cell, 16 bytes per element; one load per
// sample). The first three equal vr_dtype's values.
enum StorageKind { kStoreF32 = 0, kStoreBF16 = 1, kStoreF16 = 2, kStoreBF16Oct = 3, kStoreF16Oct = 4 };
inline int storage_kind(vr_dtype t, bool octets) { return static_cast<int>(t) + (octets && t != VR_F32 ? 2 : 0); }
constexpr int kMaxFactors = 8;

// Composite: 256-thread blocks of 32 x 8 threads, one thread per pixel of a
// 32 x 8 image tile with one brick mask per tile (the composite adjoint takes the
// same tiles).
constexpr int kCompW = 32;
constexpr int kCompH = 8;
constexpr int kCompTileH = kCompH;  // forward composite tile: kCompW x kCompTileH pixels
constexpr int kMaskThreads = 128;                // threads (tiles) per mask block of a march grid

// Brick storage index of quad (i, j, k): quads are grouped in 2x2x2 blocks of
// 128 bytes (one L1 line for float32), blocks x-fastest; nbx, nby = blocks per
// row and per plane. A warp's 8x4 ray packet then touches about the same
// number of lines whatever the view direction.
__host__ __device__ __forceinline__ int quad_index(int i, int j, int k, int nbx, int nby)
{
    return ((((k >> 1) * nby + (j >> 1)) * nbx + (i >> 1)) << 3) | ((k & 1) << 2) | ((j & 1) << 1) | (i & 1);
}

// Per-brick data of one frame, as the march kernel needs it.
struct BrickLaunch {
    int lo[3], hi[3];   // voxel box, half-open
    float own_lo[3];    // ownership bounds in voxel units (-inf / +inf on volume faces)
    float own_hi[3];
    int sx, sy;         // haloed brick extents in x and y (elements)
    long long base;     // quad offset of the brick's haloed xy-quad storage
    int rect[4];        // x0, y0, w, h of the footprint rectangle
    long long poff;     // float4 offset of the brick's partial
    int item_begin;     // first work item (tile) of this brick
    int tiles_x;        // tiles per rectangle row
};

// Everything one march launch needs; passed by value as the kernel parameter.
struct MarchParams {
    // camera, all FP32 (basis computed on the host in FP64)
    float eye[3], r[3], u[3], f[3];
    float tanx, tany;   // perspective: tan(fovy/2)*W/H, tan(fovy/2)
    float ow, oh;       // orthographic image-plane extent
    int ortho;
    int W, H;
    float inv_W, inv_H;  // 1/W, 1/H
    int pw;              // ray packet: a warp marches pw x (32/pw) pixels (pw = 4, 8 or 16)
    int tile_w, tile_h;  // work item: 2 x 2 packets = (2 pw) x (64/pw) pixels
    // volume
    float nmax;         // voxels per world unit
    float N[3];         // volume extent in voxels
    float dt, inv_dt;   // sample spacing (world units) and its inverse
    float ert_T;        // terminate a brick when T <= ert_T (negative: never)
    OpacityStep opc;    // opacity correction
    // classification
    float tf_scale, tf_bias;  // x = s*scale + bias = (s - vmin)/(vmax - vmin)*(ntf-1)
    int ntf;
    const float4 *tf;   // 2*ntf float4: (T[i], T[i+1]-T[i]) pairs, last difference 0
    const void *data;   // brick storage
    float4 *partials;   // partial pool
    unsigned long long *sample_counter;  // non-null: count executed samples
    int *count_error;   // device error word; bit 4: in a counting launch, an executed
                        // sample's quad index fell outside its brick's storage
    // composite tile masks written by the first mask_blocks blocks of the
    // march grid (null: none): bit j of tile t's mask = the brick at visibility
    // position j overlaps composite tile t (kCompW x kCompTileH pixels)
    uint4 *tile_mask;
    int mask_tiles_x, mask_tiles_y, mask_blocks;
    // pipelined frames: the partial pool this frame writes was last read by the
    // composite of frame pool_frame - 2, which sets pool_done[pool] to its own
    // frame number when it is done; the march blocks wait for that (null: no
    // wait) before storing their partials
    const unsigned long long *pool_done;
    unsigned long long pool_frame;
    int pool;
    int nb;
    int n_items;        // march work items (the grid adds mask_blocks in front)
    int order[kMaxBricks];  // brick ids front to back (ray-state cycling)
    BrickLaunch b[kMaxBricks];
};

struct CompositeParams {
    int W, H;
    int nb;
    int n_levels;                     // 1 = direct
    int order[kMaxBricks];            // brick ids front to back
    unsigned long long gid[kMaxBricks + 1];   // radix-k: byte l-1 = group index of position q at level l
                                              // (entry nb: one past the last group at every level)
    int rect[kMaxBricks][4];          // by brick id
    long long poff[kMaxBricks];       // by brick id
    const float4 *partials;
    float4 *out;
    uint4 *tile_mask;                 // per tile: visibility positions of the bricks overlapping it
    int tiles_x, tiles_y;             // composite tiles per row / column (kCompW x kCompTileH)
    // pipelined frames: the grid's last block to finish sets pool_done[pool] =
    // pool_frame (pool_count counts finished blocks; null: nothing published)
    unsigned long long *pool_done;
    unsigned int *pool_count;
    unsigned long long pool_frame;
    int pool;
};

// Batched form: per view, the camera fields that dev::owned_run reads (same
// names as MarchParams) and the view's work-item counts.
struct BatchView {
    float eye[3], r[3], u[3], f[3];
    float tanx, tany;
    float ow, oh;
    int ortho;
    int W, H;
    float inv_W, inv_H;
    float nmax;
    float N[3];
    float dt, inv_dt;
    int march_items;  // (brick, tile) items of one render of this view
    int comp_items;   // composite tiles of one render of this view
};

constexpr int kBatchCompW = 16;  // composite tile of the batched kernel (128 threads)
constexpr int kBatchCompH = 8;

struct BatchParams {
    int n_renders, n_views, nb;
    int mode;                        // 0: unit = one render; 1: unit = one volume, all views, brick-major
    int n_units;
    const int *unit_march;           // per unit: march items
    const int *unit_comp;            // per unit: composite tiles
    const long long *bw_begin;       // mode 1: nb x n_views + 1 tile offsets, (brick, view) order
    long long view_stride;           // mode 1: partial pixels per view inside a unit's ring slot
    int pw;                          // ray-packet width: a warp marches pw x (32/pw) pixels
    long long total_items;
    const long long *render_begin;   // n_units + 2 segment starts: segment g = march items of
                                     // unit g, then composite tiles of unit g-1
    const BatchView *views;          // n_views
    const BrickLaunch *vb;           // n_views x nb; rect/poff/item_begin/tiles_x per view
    const int *order;                // n_views x nb, front to back
    const void *const *vol_data;     // per volume: brick storage
    const float2 *vol_tf;            // per volume: (tf_scale, tf_bias)
    const float4 *tf;                // (T, dT) pairs
    int ntf;
    float ert_T;
    OpacityStep opc;                 // opacity correction
    float4 *ring;                    // slots x slot_px partial pixels
    long long slot_px;               // partial pixels per ring slot (one unit)
    int slots;
    float4 *out;                     // n_renders x H x W
    unsigned long long *claim;       // work counter
    int *march_done;                 // per unit: finished march items
    int *comp_done;                  // per unit: finished composite tiles
    int *error;                      // bit 1: a bounded wait gave up
    int wait_limit;                  // spin iterations (about 128 ns each) before giving up
    int wait_extra;                  // added to unit 0's march target by composite waits (test hook; 0)
};

// "over" of n images, front to back, pixel by pixel (vr_composite_images).
struct ImagesParams {
    const float4 *img[kMaxBricks];
    int n;
    long long pixels;
    float4 *out;
};

// Pack of all bricks of a volume in one launch: block j of brick b (counted
// from that brick's block_begin) writes the brick's storage quads
// [j*kPackChunk, (j+1)*kPackChunk), in storage order.
constexpr int kPackChunk = 1024;
// A thread writes two quads in turn, or one in narrow bricks, and goes on by this many
// 2x2x2 blocks.
constexpr int kPackStep = 64, kPackStepNarrow = 32;
// Bricks of at most this many voxels along x, in rows of four times as many at least. A
// warp with two quads per thread reads twice the rows of the volume per load
// instruction, three loads per row instead of two: a row of a narrow brick is in one or
// two sectors, so its loads are bound by the rows, wider ones by their bytes. 512 x 512 x 128 in
// equal bricks, us, two / one quads per thread, f32 | bf16 quads | f16 octets: 1 wide 704 /
// 502 | 680 / 476 | 1344 / 923, 4 wide 279 / 250 | 250 / 216 | 451 / 380, 5 wide 203 / 182
// | 183 / 160 | 345 / 293, 6 wide 192 / 193 | 154 / 165 | 274 / 239, 12 wide octets
// 225 / 206, 16 wide 203 / 209; half of a row of 16 (165 / 170 | 117 / 134 | 185 / 201) and whole
// rows of any width are faster with two.
constexpr int kPackNarrow = 5, kPackNarrowOctets = 12;
struct PackBrick {
    void *dst;             // the brick's storage
    long long quads;       // quads in the brick's storage (whole 2x2x2 blocks)
    int lo[3];             // voxel box origin
    int s[3];              // haloed extents (the brick stores (s0-1)(s1-1)s2 quads)
    int block_begin;       // first block of this brick
    int row;               // scalar copies: padded row length in elements (multiple of 4)
    bool narrow;           // one quad per thread (else two)
    int step[3];           // kPackStep (narrow: kPackStepNarrow) blocks on, as blocks along x, rows, planes
};
struct PackParams {
    const float *src;      // x-fastest float32 volume
    int N[3];
    int nb;
    int n_blocks;
    PackBrick b[kMaxBricks];
};

// Staged march (vr_staged.cu): scalar copies of the bricks, haloed, rows padded
// to a multiple of 4 elements; kStageCap floats per shared-memory stage (two
// stages per block).
constexpr int kStageCap = 4096;
struct StagedBricks {
    const float *scalar;          // all bricks' scalar copies
    long long sbase[kMaxBricks];  // element offset of each brick (a multiple of 32)
    int sxp[kMaxBricks];          // padded row length (elements)
};

constexpr int kWideSamples = 4;  // samples in flight per ray of a wide march (dev::march_accumulate_wide)

// Launchers (vr_kernels.cu). They return the launch's cudaError_t.
// `kind` is a StorageKind.
cudaError_t launch_pack(const PackParams &p, int kind, cudaStream_t s);
// after_composite: launch as a programmatic dependent of the preceding kernel
// (the previous pipelined frame's composite); see march_kernel.
// wide: the march for launches that do not fill the chip (same image).
cudaError_t launch_march(const MarchParams &p, int kind, cudaStream_t s, bool after_composite = false,
                         bool wide = false);
// after_frame: launch as a programmatic dependent of the preceding kernel (the
// previous pipelined frame); see march_cycle_kernel. pairs: two samples of a ray in
// flight instead of four (same image).
cudaError_t launch_march_cycle(const MarchParams &p, int kind, float4 *out, cudaStream_t s, bool after_frame,
                               bool pairs);
// max_blocks > 0: a grid of at most that many blocks, each compositing tiles in
// turn; 0: one block per tile.
cudaError_t launch_composite(const CompositeParams &p, cudaStream_t s, int max_blocks = 0);
cudaError_t launch_composite_images(const ImagesParams &p, cudaStream_t s);
// Persistent batched kernel: cooperative launch of `blocks` blocks of 128 threads.
cudaError_t launch_batch(const BatchParams &p, int kind, int blocks, cudaStream_t s);
int batch_max_blocks_per_sm(int kind);
// Staged march and the scalar brick pack (vr_staged.cu).
cudaError_t launch_march_staged(const MarchParams &p, const StagedBricks &sb, cudaStream_t s);
cudaError_t launch_scalar_pack(const PackParams &p, cudaStream_t s);

}  // namespace vr
