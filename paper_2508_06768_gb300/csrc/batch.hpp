// What the translation units of the batched path share: the device view of a
// plan and the launches of the marches.
#pragma once

#include "host.hpp"
#include "march_tile.cuh"

namespace dfs {

struct PlanPose {
    int32_t n_rays, S;
    FanDev fan;
    float a2;
    int32_t W;
    int64_t img_off;
    double a2d;
    float l2_hi, l2_lo;      // log2(a^2) split (depth-gain reading)
    int32_t ld, pad;         // row_stride(S)
    int64_t pad_off;         // the pose's first internal row
};

// What the forward keeps for the adjoint of the same call (each nullable).
struct FwdKeep {
    float4 *ckpt;
    float *mbuf;
    float2 *kbuf;
    float4 *bcar;
    float *zbuf, *rbuf;   // one warp per ray: impedance and r rows (gz_stride)
};

struct BatchDev {
    const PlanPose *pose;
    const int32_t *ray_pose, *ray_j, *order;
    const int64_t *row_off, *gz_off, *ck_off;   // row_off: packed image rows
    const int64_t *pad_off;                     // internal rows (row_stride)
    int64_t total_rays;
};

// The forward's launch: fwd_form 0 one warp per ray, 1 tiles with one lane
// per ray (grid = CTAs per SM x SMs of kTileWarps warps).
struct FwdLaunch {
    int grid, form;
    const TileDesc *tiles;
    int64_t n_tiles;
    const float *spk_in;   // speckle factors drawn ahead (one warp per ray only), or null
    bool padded;           // the output rows are internal rows
};

inline int sm_count()
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// The forward march of rays q0 .. q0+qn-1 of the queue (and, when sel lists
// rays, the refined pass), and the adjoint march.
int launch_batch_fwd(int dtype, int warps, const void *vol, const MarchArgs &A, const BatchDev &B, const RayGeo *geo,
                     float *out, int *valid, uint32_t *status, unsigned *counter, const FwdKeep &kp,
                     const FwdLaunch &fl, const RefineSel &sel, const PoseFrame *frames, const VolPlace &vp, int64_t q0,
                     int64_t qn, cudaStream_t s);
int launch_batch_bwd(int dtype, int warps, const void *vol, const MarchArgs &A, const BatchDev &B, const RayGeo *geo,
                     const float *gy, bool gy_padded, float *gz, double *part, float4 *ckpt, unsigned *counter,
                     const float *mbuf, const float *zbuf, const float *rbuf, int grid, bool pose, int64_t q0,
                     int64_t qn, cudaStream_t s);

}  // namespace dfs
