// vr_grad.h -- structures shared by the host side of the adjoint (vr_host.cpp)
// and its kernels (vr_grad.cu). Not part of the public ABI.
#pragma once

#include "vr_internal.h"

namespace vr {

// A brick's owned run of a ray is cut into segments of kGradSeg samples, counted
// from the run's first sample, and groups of kGradGroup segments, one thread's
// work. A run of more than kGradMaxRun samples is reported (its samples get no
// gradient), and its last segment takes everything from sample kGradMaxRun on.
constexpr int kGradSeg = 8;
constexpr int kGradGroup = 8;
constexpr int kGradMaxRun = 4096;
// Copies of the table gradient ((ntf + 1) x 4 floats each), spread over blocks and
// lanes so that few reductions meet on one entry. 4 views of 512^2, ms per training step,
// 64 / 256 / 512 / 1024 / 2048 copies by block and lane % 8: 256^3 blobs 5.16 / 5.00 / 5.00 /
// 5.11 / 5.12, noise 7.21 / 6.49 / 6.31 / 6.38 / 6.33; 512 by block alone 5.12 and 6.34, by
// block and lane 5.06 and 6.38. (16 copies by block, an earlier kernel: 7.29 against 6.44
// with 64.)
constexpr int kGradCopies = 512;
constexpr int kGradLaneCopies = 8;
// Voxel gradients go through quads (at most two 16-byte reductions per cell, then
// one pass over the volume's quads) when the view's samples, bounded by rect areas
// times longest runs, are over this many times the quads, else straight into the
// voxels (eight reductions per cell). One backward of 8 bricks, us, quads / direct:
// 256^3 at 256^2 (ratio 1.6) 416 / 351, at 384^2 (3.6 to 4.4) 527 / 557, at 512^2 (5.8
// to 7.4) 692 / 865; 128^3 at 256^2 (6.4) 156 / 186; 64^3 at 256^2 118 / 155.
constexpr long long kGradQuadsRatio = 3;
constexpr long long kGradBandBytes = 1LL << 30;  // per-sample workspace of one band of image rows

struct GradParams {
    MarchParams m;                // camera, lattice, table, bricks (rects clipped to the image band)
    const float4 *grad_img;       // dL/dI, H x W
    // Workspace, [...][pixel of the brick's rect]; the offsets count segments and groups.
    float *x;                     // per sample: its table coordinate (not clamped)
    float *front;                 // per segment: T in front of it, from the group's start
    float2 *group;                // per group: (lambda_C . C, T) of the group alone, then
                                  // (lambda_T behind it, T in front of it) along the whole ray
    long long soff[kMaxBricks], goff[kMaxBricks];
    int nseg[kMaxBricks];         // segments kept per pixel
    unsigned short *count;        // per (brick, pixel), at BrickLaunch::poff: groups of the run
    float *tf_copies;             // kGradCopies x (ntf + 1) x 4, zeroed before the launches
    float *grad_vol;              // Nz x Ny x Nx, or null
    float4 *grad_quads;           // quads of voxel gradients laid out as the bricks', or null
                                  // (reductions straight into grad_vol)
    int N[3];
    int band_y0, band_h;          // image rows of this launch
    int *error;                   // device error word: bit 0 = a run exceeded kGradMaxRun
};

// Voxel gradients gathered from the quads (grad_voxels_kernel): a warp's task is a
// chunk of 31 voxels along x in a set of rows of one plane.
constexpr int kGradVoxelRows = 16;  // even: a set starts at the lower row of the quads' blocks
__host__ __device__ inline int grad_voxel_chunks(int sx) { return (sx + 30) / 31; }
__host__ __device__ inline int grad_voxel_row_sets(int sy) { return (sy + kGradVoxelRows - 1) / kGradVoxelRows; }
struct GradVoxelBrick {
    long long base;   // quad offset of the brick's storage
    int lo[3];        // voxel box origin
    int s[3];         // haloed extents
    int task_begin;   // first of the brick's s[2] x row sets x chunks
};
struct GradVoxelParams {
    const float4 *quads;
    float *grad_vol;
    int N[3];
    int nb;
    int n_tasks;
    GradVoxelBrick b[kMaxBricks];
};

// The adjoint's steps for one band of image rows (see vr_grad.cu), in order:
// groups, scan, samples. `groups`: the largest number of groups of a brick. launch_grad_table adds the copies into grad_tf (ntf x 4).
cudaError_t launch_grad_groups(const GradParams &p, int kind, int groups, cudaStream_t s);
cudaError_t launch_grad_scan(const GradParams &p, cudaStream_t s);
cudaError_t launch_grad_samples(const GradParams &p, int groups, cudaStream_t s);
cudaError_t launch_grad_voxels(const GradVoxelParams &p, cudaStream_t s);
cudaError_t launch_grad_table(const float *tf_copies, int ntf, float *grad_tf, cudaStream_t s);

// The table as the kernels read it, (T[i], T[i+1] - T[i]) pairs with the last
// difference 0, from a device table (vr_set_transfer_function_async: fitting a
// table changes it every step, and a copy to the host and back waits for the GPU).
cudaError_t launch_table_pairs(const float4 *rgba, int n, float4 *pairs, cudaStream_t s);

}  // namespace vr
