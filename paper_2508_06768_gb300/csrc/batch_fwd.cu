// Forward marches of the batched path: one warp per ray, one lane per ray,
// and the refined pass.
#include "batch.hpp"

using namespace dfs;

namespace {

// Persistent forward: each warp takes rays from the queue (longest first).
// TRACK (refinement on, sel.rinfo set): it is the FP32 pass, which lists the
// rays that need the refined pass.  Bound by L1 wavefronts (90 to 92 % of peak,
// two thirds of them the eight corner loads, 4.4 lines each) with the issue slots
// at 76 to 78 %.  512 uneven frames with everything kept for the adjoint: 1433 us
// with packed rows, per-row tests and per-sample neighbour exchange, 1097 us
// as it stands (225 and 181 warp instructions per 32 samples).
template <typename T, int WARPS, int MODE, bool TRACK>
__global__ void __launch_bounds__(WARPS * 32, kFwdThreadsPerSM / (WARPS * 32))
    k_batch_fwd(const T *__restrict__ vol, MarchArgs A, BatchDev B, const RayGeo *__restrict__ geo,
                float *__restrict__ out, int *__restrict__ valid, uint32_t *__restrict__ status,
                unsigned *__restrict__ counter, float4 *__restrict__ ckpt, float *__restrict__ zbuf,
                float *__restrict__ rbuf, const float *__restrict__ spk_in, RefineSel sel, int64_t q0, int64_t qn,
                bool padded)
{
    __shared__ float2 buf[WARPS][kSegPad];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (;;) {
        unsigned q = 0;
        if (lane == 0) q = atomicAdd(counter, 1u);
        q = __shfl_sync(0xffffffffu, q, 0);
        if ((int64_t)q >= qn) break;   // entries q0 .. q0+qn-1 of the ray order
        const int r = B.order[q0 + q];
        RayGeo rg = geo[r];
        MarchArgs Ap = A;
        if (!A.atten) Ap.a2 = B.pose[rg.pose].a2;   // the depth-gain reading keeps a2 = 1 (lossless systems)
        const int64_t po = B.pad_off[r], go = B.gz_off[r];
        RayOut o{out + (padded ? po : B.row_off[r]), valid ? valid + r : nullptr, status,
                 ckpt ? ckpt + B.ck_off[r] : nullptr, zbuf ? zbuf + go : nullptr, rbuf ? rbuf + go : nullptr,
                 spk_in ? spk_in + po : nullptr, TRACK ? sel.rinfo + r : nullptr, sel.rlist, sel.rcount, r, padded};
        march_fwd_ray<T, MODE, TRACK, false, true>(vol, Ap, rg, o, buf[w]);
        __syncwarp();
    }
}

// Persistent forward with one lane per ray: each warp takes tiles of 32
// consecutive rays of a pose from the queue (longest first).
template <typename T, bool KEEP>
__global__ void __launch_bounds__(kTileWarps * 32, kFwdThreadsPerSM / (kTileWarps * 32)) k_batch_fwd_tiles(const T *__restrict__ vol, MarchArgs A, BatchDev B,
                                                          const RayGeo *__restrict__ geo,
                                                          const TileDesc *__restrict__ tiles, int64_t n_tiles,
                                                          float *__restrict__ out, int *__restrict__ valid,
                                                          uint32_t *__restrict__ status,
                                                          unsigned *__restrict__ counter, float4 *__restrict__ ckpt,
                                                          float *__restrict__ mbuf, float2 *__restrict__ kbuf,
                                                          float4 *__restrict__ bcar, RefineSel sel, bool padded)
{
    __shared__ TileSmem sm[kTileWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (;;) {
        unsigned q = 0;
        if (lane == 0) q = atomicAdd(counter, 1u);
        q = __shfl_sync(0xffffffffu, q, 0);
        if ((int64_t)q >= n_tiles) break;
        const TileDesc *tl = tiles + q;
        MarchArgs Ap = A;
        if (!A.atten) Ap.a2 = B.pose[tl->pose].a2;   // the depth-gain reading keeps a2 = 1
        march_fwd_tile<T, KEEP>(vol, Ap, tl, geo, out, valid, status, ckpt, mbuf, kbuf, bcar, sel, padded, sm[w]);
        __syncwarp();
    }
}

// Refined pass of the batch over the rays the FP32 pass listed (in the order
// it listed them, which follows its longest-first queue).
template <typename T, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, kRefineWarpsPerSM / WARPS) k_batch_refine(const T *__restrict__ vol, MarchArgs A, BatchDev B,
                                                                const RayGeo *__restrict__ geo,
                                                                const PoseFrame *__restrict__ frames, VolPlace vp,
                                                                float *__restrict__ out, int *__restrict__ valid,
                                                                uint32_t *__restrict__ status,
                                                                float4 *__restrict__ ckpt,
                                                                const float *__restrict__ spk_in, RefineSel sel,
                                                                bool padded)
{
    __shared__ float buf[WARPS][kSegPad];
    __shared__ float2 dbuf[WARPS][kSegPad];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned n = *sel.rcount;
    for (;;) {
        unsigned q = 0;
        if (lane == 0) q = atomicAdd(sel.ticket, 1u);
        q = __shfl_sync(0xffffffffu, q, 0);
        if (q >= n) break;
        const int r = sel.rlist[q];
        const RayGeo rg = geo[r];
        const PlanPose pp = B.pose[rg.pose];
        MarchArgs Ap = A;
        if (!A.atten) {
            Ap.a2 = pp.a2;
            Ap.a2d = pp.a2d;
        }
        const FanDev &fd = pp.fan;
        RayOut o{out + (padded ? B.pad_off[r] : B.row_off[r]), valid ? valid + r : nullptr, status,
                 ckpt ? ckpt + B.ck_off[r] : nullptr, nullptr, nullptr, spk_in ? spk_in + B.pad_off[r] : nullptr, nullptr,
                 nullptr, nullptr, r, padded};
        refine_ray<T, true>(vol, Ap, rg, frames[rg.pose], fd, vp, o, sel.rinfo[r], buf[w], dbuf[w]);
        __syncwarp();
    }
}

template <typename T, int WARPS>
void launch_fwd_t(const void *vol, const MarchArgs &A, const BatchDev &B, const RayGeo *geo, float *out, int *valid,
                  uint32_t *status, unsigned *counter, const FwdKeep &kp, const FwdLaunch &fl, const RefineSel &sel,
                  const PoseFrame *frames, const VolPlace &vp, int64_t q0, int64_t qn, cudaStream_t s)
{
    if (fl.form == 1) {
        const bool keep = kp.ckpt || kp.mbuf || kp.kbuf || kp.bcar;
        auto kernel = keep ? k_batch_fwd_tiles<T, true> : k_batch_fwd_tiles<T, false>;
        kernel<<<fl.grid, kTileWarps * 32, 0, s>>>((const T *)vol, A, B, geo, fl.tiles, fl.n_tiles, out, valid, status,
                                                   counter, kp.ckpt, kp.mbuf, kp.kbuf, kp.bcar, sel, fl.padded);
    } else {
#define DFS_BF(MODE, TRACK)                                                                                         \
    k_batch_fwd<T, WARPS, MODE, TRACK><<<fl.grid, WARPS * 32, 0, s>>>((const T *)vol, A, B, geo, out, valid, status, \
                                                                      counter, kp.ckpt, kp.zbuf, kp.rbuf, fl.spk_in, \
                                                                      sel, q0, qn, fl.padded)
        const bool track = sel.rinfo != nullptr;
        if (A.mode == DIFFUS_MODE_LITERAL) {
            if (track) DFS_BF(DIFFUS_MODE_LITERAL, true);
            else DFS_BF(DIFFUS_MODE_LITERAL, false);
        } else {
            if (track) DFS_BF(DIFFUS_MODE_SIGNED, true);
            else DFS_BF(DIFFUS_MODE_SIGNED, false);
        }
#undef DFS_BF
    }
    if (sel.rinfo)
        k_batch_refine<T, WARPS><<<kRefineWarpsPerSM / WARPS * sm_count(), WARPS * 32, 0, s>>>(
            (const T *)vol, A, B, geo, frames, vp, out, valid, status, kp.ckpt, fl.spk_in, sel, fl.padded);
}

template <typename T>
int launch_fwd_w(int warps, const void *vol, const MarchArgs &A, const BatchDev &B, const RayGeo *geo, float *out,
                 int *valid, uint32_t *status, unsigned *counter, const FwdKeep &kp, const FwdLaunch &fl,
                 const RefineSel &sel, const PoseFrame *frames, const VolPlace &vp, int64_t q0, int64_t qn,
                 cudaStream_t s)
{
    switch (warps) {
    case 2: launch_fwd_t<T, 2>(vol, A, B, geo, out, valid, status, counter, kp, fl, sel, frames, vp, q0, qn, s); break;
    case 4: launch_fwd_t<T, 4>(vol, A, B, geo, out, valid, status, counter, kp, fl, sel, frames, vp, q0, qn, s); break;
    case 8: launch_fwd_t<T, 8>(vol, A, B, geo, out, valid, status, counter, kp, fl, sel, frames, vp, q0, qn, s); break;
    default: return DIFFUS_E_PLAN;
    }
    return DIFFUS_OK;
}

}  // namespace

namespace dfs {

int launch_batch_fwd(int dtype, int warps, const void *vol, const MarchArgs &A, const BatchDev &B, const RayGeo *geo,
                     float *out, int *valid, uint32_t *status, unsigned *counter, const FwdKeep &kp,
                     const FwdLaunch &fl, const RefineSel &sel, const PoseFrame *frames, const VolPlace &vp, int64_t q0,
                     int64_t qn, cudaStream_t s)
{
    if (dtype == DIFFUS_F32)
        return launch_fwd_w<float>(warps, vol, A, B, geo, out, valid, status, counter, kp, fl, sel, frames, vp, q0, qn,
                                   s);
    return launch_fwd_w<unsigned short>(warps, vol, A, B, geo, out, valid, status, counter, kp, fl, sel, frames, vp, q0,
                                        qn, s);
}

}  // namespace dfs
