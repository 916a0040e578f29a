// Adjoint march of the batched path, one warp per ray.
#include <atomic>

#include "batch.hpp"
#include "march_bwd.cuh"

using namespace dfs;

namespace {

// POSE: the pose-only call, which samples Z and dZ/dp itself; otherwise the
// march reads the rows that the forward of the same call kept (STORED) and
// never touches the volume, whatever its type.  STORED is bound by issue (77 %)
// and L1 wavefronts (64 to 68 %): 512 uneven frames 1535 us with the kept pairs
// transposed through shared memory and scalar rows, 942 us with each lane
// loading its chunks of the kept rows (249 and 155 warp instructions per 32
// samples).
template <typename T, int WARPS, bool POSE, int MODE>
__global__ void __launch_bounds__(WARPS * 32, (POSE ? kBwdThreadsPerSM : kBwdValThreadsPerSM) / (WARPS * 32))
    k_batch_bwd(const T *__restrict__ vol, MarchArgs A, BatchDev B, const RayGeo *__restrict__ geo,
                const float *__restrict__ gy, bool gy_padded, float *__restrict__ gz, double *__restrict__ part,
                float4 *__restrict__ ckpt, unsigned *__restrict__ counter, const float *__restrict__ mbuf,
                const float *__restrict__ zbuf, const float *__restrict__ rbuf, int64_t q0, int64_t qn)
{
    // WARPS slots of BwdSmem, in dynamic shared memory (above the 48 KB of
    // static arrays with 8 warps and POSE)
    extern __shared__ __align__(16) unsigned char bwd_smem[];
    BwdSmem<POSE, !POSE> *sm = reinterpret_cast<BwdSmem<POSE, !POSE> *>(bwd_smem);
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
        march_bwd_ray<T, MODE, POSE, !POSE>(vol, Ap, rg, gy + (gy_padded ? po : B.row_off[r]), gz + go,
                                            part + 6 * (size_t)r, ckpt + B.ck_off[r], sm[w], gy_padded, true,
                                            mbuf ? mbuf + po : nullptr, zbuf + go, rbuf + go);
        __syncwarp();
    }
}

// Opt the kernel in to its dynamic shared memory, once per kernel and device
// (the attribute is not a stream operation, so this is safe inside a
// capture).  Returns nonzero on failure.
template <typename T, int WARPS, bool POSE, int MODE>
int bwd_smem_optin(size_t bytes)
{
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return 0;
    if (cudaFuncSetAttribute(k_batch_bwd<T, WARPS, POSE, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)bytes) != cudaSuccess)
        return 1;
    done.fetch_or(bit, std::memory_order_acq_rel);
    return 0;
}

struct BwdCall {
    const void *vol;
    const MarchArgs &A;
    const BatchDev &B;
    const RayGeo *geo;
    const float *gy;
    bool gy_padded;
    float *gz;
    double *part;
    float4 *ckpt;
    unsigned *counter;
    const float *mbuf, *zbuf, *rbuf;
    int grid;
    int64_t q0, qn;
    cudaStream_t s;
};

template <typename T, int WARPS, bool POSE, int MODE>
int launch_one(const BwdCall &c)
{
    const size_t sb = WARPS * sizeof(BwdSmem<POSE, !POSE>);
    if (bwd_smem_optin<T, WARPS, POSE, MODE>(sb)) return DIFFUS_E_LAUNCH;
    k_batch_bwd<T, WARPS, POSE, MODE><<<c.grid, WARPS * 32, sb, c.s>>>(
        (const T *)c.vol, c.A, c.B, c.geo, c.gy, c.gy_padded, c.gz, c.part, c.ckpt, c.counter, c.mbuf, c.zbuf, c.rbuf,
        c.q0, c.qn);
    return DIFFUS_OK;
}

template <typename T, bool POSE, int MODE>
int launch_w(int warps, const BwdCall &c)
{
    switch (warps) {
    case 2: return launch_one<T, 2, POSE, MODE>(c);
    case 4: return launch_one<T, 4, POSE, MODE>(c);
    case 8: return launch_one<T, 8, POSE, MODE>(c);
    default: return DIFFUS_E_PLAN;
    }
}

template <typename T, bool POSE>
int launch_m(int warps, const BwdCall &c)
{
    return c.A.mode == DIFFUS_MODE_LITERAL ? launch_w<T, POSE, DIFFUS_MODE_LITERAL>(warps, c)
                                           : launch_w<T, POSE, DIFFUS_MODE_SIGNED>(warps, c);
}

}  // namespace

namespace dfs {

int launch_batch_bwd(int dtype, int warps, const void *vol, const MarchArgs &A, const BatchDev &B, const RayGeo *geo,
                     const float *gy, bool gy_padded, float *gz, double *part, float4 *ckpt, unsigned *counter,
                     const float *mbuf, const float *zbuf, const float *rbuf, int grid, bool pose, int64_t q0,
                     int64_t qn, cudaStream_t s)
{
    const BwdCall c{vol,     A,    B,    geo,  gy,   gy_padded, gz, part, ckpt,
                    counter, mbuf, zbuf, rbuf, grid, q0,        qn, s};
    if (!pose) return launch_m<float, false>(warps, c);
    return dtype == DIFFUS_F32 ? launch_m<float, true>(warps, c) : launch_m<unsigned short, true>(warps, c);
}

}  // namespace dfs
