// dlo_kernels.h -- launch entry points of the device kernels (host side of each .cu file).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include "dlo_internal.h"

namespace dlo {

// Shared memory of one rod (of at most NV vertices) in the forward and recompute kernels: nine
// float4 arrays of NV (displacements, positions, velocities, base frames + twist, base tangents +
// rest lengths, hinge state, three exchanged between neighbours) and, with self-contact, 4 NV
// pair slots (two float4 of projection data each, one packed index pair) plus an int4 fixed-point
// accumulator per vertex.
constexpr int kPairsPerVertex = 4;
__host__ __device__ constexpr size_t warp_smem_bytes(int NV, bool contact) {
    return (size_t)(9 * NV) * 16 +
           (contact ? ((size_t)(2 * kPairsPerVertex * NV) * 16 + (size_t)NV * 16 + (size_t)(kPairsPerVertex * NV) * 4)
                    : 0);
}

// Per size class (dlo_nv*.cu).
cudaError_t launch_forward_nv32(const FwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int forward_occ_nv32(bool c, int warps);
cudaError_t launch_rec_nv32(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rec_occ_nv32(bool c, int warps);
cudaError_t launch_rev_nv32(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rev_occ_nv32(bool c, int warps);
cudaError_t launch_forward_nv64(const FwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int forward_occ_nv64(bool c, int warps);
cudaError_t launch_rec_nv64(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rec_occ_nv64(bool c, int warps);
cudaError_t launch_rev_nv64(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rev_occ_nv64(bool c, int warps);
cudaError_t launch_forward_nv128(const FwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int forward_occ_nv128(bool c, int warps);
cudaError_t launch_rec_nv128(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rec_occ_nv128(bool c, int warps);
cudaError_t launch_rev_nv128(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rev_occ_nv128(bool c, int warps);
cudaError_t launch_forward_nv192(const FwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int forward_occ_nv192(bool c, int warps);
cudaError_t launch_rec_nv192(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rec_occ_nv192(bool c, int warps);
cudaError_t launch_rev_nv192(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rev_occ_nv192(bool c, int warps);
cudaError_t launch_forward_nv224(const FwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int forward_occ_nv224(bool c, int warps);
cudaError_t launch_rec_nv224(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rec_occ_nv224(bool c, int warps);
cudaError_t launch_rev_nv224(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rev_occ_nv224(bool c, int warps);
cudaError_t launch_forward_nv256(const FwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int forward_occ_nv256(bool c, int warps);
cudaError_t launch_rec_nv256(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rec_occ_nv256(bool c, int warps);
cudaError_t launch_rev_nv256(const BwdParams& P, bool c, int grid, int warps, cudaStream_t st);
int rev_occ_nv256(bool c, int warps);
// the backward's recompute and reverse kernels (dlo_adjoint.cu dispatches to the size classes)
cudaError_t launch_rec(const BwdParams& P, int nv_max, bool contact, int grid, int warps, cudaStream_t st);
int rec_blocks_per_sm(int nv_max, bool contact, int warps);
cudaError_t launch_rev(const BwdParams& P, int nv_max, bool contact, int grid, int warps, cudaStream_t st);
int rev_blocks_per_sm(int nv_max, bool contact, int warps);
// Substeps whose gripper blocks (256 B each) are formed together.
constexpr int kPoseBatch = 8;
// Shared memory of one rod: the arrays above, 256 B of group-reduction scratch, and the gripper
// blocks, the pose and the actions (144 B), in whole 256 B.
__host__ __device__ constexpr size_t rod_smem_bytes(int NV, bool contact) {
    return warp_smem_bytes(NV, contact) + 512 + 256 * kPoseBatch;
}

// Rod size classes: a rod of nv vertices runs in the kernels instantiated for the smallest
// class that holds it: threads, shared memory, records and candidate slots are sized per class.  In the
// reverse two rods of any class above 128 share an SM; 192 and 224 leave a thread more registers
// and move fewer record bytes than 256 does.  608 ropes, 2 frames with their gradient: x 150
// 0.55 ms (0.64 in class 256), x 180 0.98 (1.09), x 200 1.09 (1.11), x 224 1.16 (1.18).
constexpr int kNumSizeClasses = 6;
__host__ __device__ constexpr int size_class_at(int k) {
    return k == 0 ? 32 : k == 1 ? 64 : k == 2 ? 128 : k == 3 ? 192 : k == 4 ? 224 : 256;
}
__host__ __device__ constexpr int size_class(int nv) {
    return nv <= 32 ? 32 : nv <= 64 ? 64 : nv <= 128 ? 128 : nv <= 192 ? 192 : nv <= 224 ? 224 : 256;
}

// Threads that step one rod of size class NV: one per vertex.
__host__ __device__ constexpr int threads_per_rod(int NV) { return NV; }

cudaError_t launch_forward(const FwdParams& P, int nv_max, bool contact, int grid, int warps, cudaStream_t st);
int forward_blocks_per_sm(int nv_max, bool contact, int warps);

struct InitParams {
    const RodInfo* rods;
    int B;
    const float4* xin;       // [V][4] positions (w ignored)
    const float4* vin;       // [V][4] or null
    const float* thin;       // [Etot] or null
    const float2* mass;      // [V] (mass, inverse mass)
    const float2* ES;        // [Etot] (rest length, 1/inertia)
    float4* rest;            // [V] rest hinge data (kbar0 x, kbar0 y, mbar, unused)
    StateRef S;
    const float* GP0;        // [B][2][12] initial gripper poses
    int rest_mode;           // 1: compute the rest twist from xin into rest[].z only
    // the rods of up to 32 vertices (nv_small at most), when they take the kernel that packs several
    // into a warp (n_small > 0)
    const int* small;
    int n_small, nv_small;
};
// nv_max: the largest size class of the batch (threads per block)
cudaError_t launch_init(const InitParams& P, int nv_max, cudaStream_t st);
// Reverse of launch_init's frame construction: from the cotangents of the base tangents and
// directors, adds the cotangents of the positions to gx0.
cudaError_t launch_frames_adjoint(const RodInfo* rods, int B, int nv_max, const float4* X0, const float4* gtb0,
                                  const float4* gd1b0, float4* gx0, cudaStream_t st);

}  // namespace dlo
