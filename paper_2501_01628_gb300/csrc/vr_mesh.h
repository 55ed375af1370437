// vr_mesh.h -- structures shared by the host runtime of tetrahedral-mesh volumes
// (vr_mesh_host.cpp) and their march kernel (vr_mesh.cu). Not part of the
// public ABI.
//
// The paper's data set is a mixed finite-element mesh distributed over ranks
// (Sec. 5); elements here are tetrahedra, each held by one brick. Within an
// element the value is linear, so along a ray it is linear in t, and a ray
// leaves the element through the face whose barycentric coordinate reaches 0
// first. A ray's run inside a brick therefore starts with one point location (the
// brick's start grid and a walk through face neighbours or, where that walk does
// not end, the brick's BVH, the acceleration structure of Sec. 2.1) and then
// walks face neighbours.
#pragma once

#include "vr_internal.h"

namespace vr {

// Element record, 4 float4 (64 B), voxel units:
//   r0 = (c.x, c.y, c.z, s_mean)   centroid and mean vertex value
//   ri = (n_i.x, n_i.y, n_i.z, s_i - s_0), i = 1..3
// with n_i the gradient of barycentric coordinate lambda_i, so that
// lambda_i(q) = 1/4 + n_i . (q - c) for i = 1..3, n_0 = -(n_1 + n_2 + n_3),
// and value(q) = s_mean + g . (q - c), g = sum_{i=1..3} (s_i - s_0) n_i.
// Face i is the face opposite vertex i (lambda_i = 0 on it).
constexpr int kMeshRec = 4;

// BVH node over a brick's elements (voxel units), nodes in preorder: an inner
// node's first child is the next node; `skip` is the first node after the
// node's subtree (the root's skip is the node count), so a point query needs no
// stack. leaf = 0 for an inner node, else (count << 28) | first: count elements
// from brick-local element index first.
struct MeshNode {
    float lo[3];
    int skip;
    float hi[3];
    int leaf;
};

constexpr int kMeshLeafMax = 4;        // elements per leaf
constexpr int kMeshMaxElems = 1 << 28; // elements per brick (leaf encoding)
constexpr int kMeshStallSteps = 32;    // element steps without a sample before re-locating

// Start grid of a brick: n[0] x n[1] x n[2] equal cells of its box, each with an
// element near the cell's centre (brick-local), from which a walk through face
// neighbours reaches a sample in the cell in a step or two. Bricks are convex and
// filled, so where all faces inside a brick are shared the walk always has a
// neighbour to go to. Vertices doubled on an interior surface, hanging nodes or
// unmerged vertices leave faces inside that no second element shares: a walk that
// comes to one ends in the BVH. About kMeshGridElems elements per cell.
struct MeshGrid {
    long long base;   // first cell in MeshParams::start
    int n[3];
    float scale[3];   // cells per voxel
};
constexpr int kMeshGridElems = 2;
constexpr int kMeshWalkSteps = 64;     // of a walk before the BVH is asked instead
constexpr float kMeshInside = 1.0e-6f; // barycentric slack of a sample on a face (FP32 rounding)

struct MeshParams {
    MarchParams m;                    // camera, lattice, transfer function, tiles, bricks
    const float4 *rec;                // kMeshRec float4 per element
    const int4 *nbr;                  // brick-local neighbour across face i, -1 if no element of the brick shares it
    const MeshNode *nodes;
    const int *start;                 // start grids
    MeshGrid grid[kMaxBricks];
    long long rec_base[kMaxBricks];   // first element of each brick
    long long node_base[kMaxBricks];  // first BVH node of each brick
    int *error;                       // bit 3: a point location found no element (empty brick)
};

// The grid starts with p.m.mask_blocks blocks that write the composite's tile
// masks. after_frame: launch as a programmatic dependent of the preceding
// kernel (the previous pipelined frame).
cudaError_t launch_march_mesh(const MeshParams &p, cudaStream_t s, bool after_frame = false);

}  // namespace vr
