// CT pre-pass: Hounsfield units to acoustic impedance through a
// user-supplied piecewise-linear calibration table, written as an FP32 or
// BF16 impedance volume that the renderer then samples.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "host.hpp"

using namespace dfs;

namespace {

constexpr int kHuMax = 64;

struct HuTable {
    int m;
    float hu[kHuMax];      // breakpoints, strictly increasing
    float z[kHuMax];       // impedance at the breakpoints
    float slope[kHuMax];   // (z[i+1] - z[i]) / (hu[i+1] - hu[i]), from FP64
};

__device__ __forceinline__ float hu_map(const HuTable &t, float h)
{
    if (h <= t.hu[0]) return t.z[0];
    if (h >= t.hu[t.m - 1]) return t.z[t.m - 1];
    int lo = 0, hi = t.m - 1;          // hu[lo] < h < hu[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (h > t.hu[mid]) lo = mid; else hi = mid;
    }
    return fmaf(h - t.hu[lo], t.slope[lo], t.z[lo]);
}

__device__ __forceinline__ void hu_store(float *zf, unsigned short *zb, int64_t v, float z)
{
    if (zf) zf[v] = z;
    else zb[v] = __bfloat16_as_ushort(__float2bfloat16_rn(z));
}

// Eight voxels per thread with 16-byte loads where the pointers allow it;
// the values themselves are exact in float (|hu| < 2^15).
__global__ void k_hu_to_z(const int16_t *__restrict__ hu, int64_t n, HuTable tab, float *__restrict__ zf,
                          unsigned short *__restrict__ zb, int vec)
{
    __shared__ HuTable t;
    for (int i = threadIdx.x; i < (int)(sizeof(HuTable) / 4); i += blockDim.x)
        ((float *)&t)[i] = ((const float *)&tab)[i];
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n8 = vec ? n / 8 : 0;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n8; g += stride) {
        const uint4 raw = __ldg(reinterpret_cast<const uint4 *>(hu) + g);
        const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
        float z[8];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            z[2 * i] = hu_map(t, (float)(int16_t)(w[i] & 0xFFFFu));
            z[2 * i + 1] = hu_map(t, (float)(int16_t)(w[i] >> 16));
        }
        if (zf) {
            float4 *o = reinterpret_cast<float4 *>(zf) + 2 * g;
            o[0] = make_float4(z[0], z[1], z[2], z[3]);
            o[1] = make_float4(z[4], z[5], z[6], z[7]);
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) hu_store(zf, zb, 8 * g + i, z[i]);
        }
    }
    for (int64_t v = 8 * n8 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        hu_store(zf, zb, v, hu_map(t, (float)hu[v]));
}

// The same map through a table of every whole HU value between the
// breakpoints' ends, built once per block in shared memory by hu_map itself:
// a voxel is one clamped lookup instead of a search, which leaves the pass to
// HBM (6 bytes per voxel).  lo..hi: the table's HU range; values outside it
// map as its ends do.  The block's first voxels are loaded ahead of the table,
// the next ones ahead of the stores (256^3 voxels from and to HBM: 21.7 us
// without, 20.7 with; BF16 16.2 and 14.5 us).
constexpr int kLutThreads = 1024;
constexpr int kLutMax = 24576;        // entries: two blocks' tables fit an SM's shared memory

__global__ void __launch_bounds__(kLutThreads, 2) k_hu_lut(const int16_t *__restrict__ hu, int64_t n,
                                                        const __grid_constant__ HuTable tab, int lo, int hi,
                                                        float *__restrict__ zf, unsigned short *__restrict__ zb, int vec)
{
    extern __shared__ float lut[];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n8 = vec ? n / 8 : 0;
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint4 raw = make_uint4(0, 0, 0, 0);
    if (g < n8) raw = __ldcs(reinterpret_cast<const uint4 *>(hu) + g);
    for (int i = threadIdx.x; i <= hi - lo; i += blockDim.x) lut[i] = hu_map(tab, (float)(lo + i));
    __syncthreads();
    auto look = [&](int h) { return lut[min(max(h, lo), hi) - lo]; };
    for (; g < n8; g += stride) {
        const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
        float z[8];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            z[2 * i] = look((int)(int16_t)(w[i] & 0xFFFFu));
            z[2 * i + 1] = look((int)(int16_t)(w[i] >> 16));
        }
        if (g + stride < n8) raw = __ldcs(reinterpret_cast<const uint4 *>(hu) + g + stride);
        if (zf) {
            float4 *o = reinterpret_cast<float4 *>(zf) + 2 * g;
            o[0] = make_float4(z[0], z[1], z[2], z[3]);
            o[1] = make_float4(z[4], z[5], z[6], z[7]);
        } else {
            uint32_t p[4];
#pragma unroll
            for (int i = 0; i < 4; i++)
                p[i] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(z[2 * i])) |
                       ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(z[2 * i + 1])) << 16);
            reinterpret_cast<uint4 *>(zb)[g] = make_uint4(p[0], p[1], p[2], p[3]);
        }
    }
    for (int64_t v = 8 * n8 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        hu_store(zf, zb, v, look((int)hu[v]));
}

// Opt k_hu_lut in to its dynamic shared memory, once per device (the attribute
// is not a stream operation, so this is safe inside a capture).
int lut_smem_optin()
{
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return 0;
    if (cudaFuncSetAttribute(k_hu_lut, cudaFuncAttributeMaxDynamicSharedMemorySize, kLutMax * (int)sizeof(float)) !=
        cudaSuccess)
        return 1;
    done.fetch_or(bit, std::memory_order_acq_rel);
    return 0;
}

}  // namespace

extern "C" int diffus_hu_to_z(const int16_t *hu, int64_t n, const double *hu_pts, const double *z_pts, int32_t m,
                              void *z_out, int32_t out_dtype, diffus_stream_t stream)
{
    NvtxRange nvtx_range("diffus_hu_to_z");
    if (!hu || !hu_pts || !z_pts || !z_out) return DIFFUS_E_NULL;
    if (n < 0 || m < 1 || m > kHuMax) return DIFFUS_E_PARAM;
    if (out_dtype != DIFFUS_F32 && out_dtype != DIFFUS_BF16) return DIFFUS_E_DTYPE;
    if (((uintptr_t)hu) % 2 || ((uintptr_t)z_out) % (out_dtype == DIFFUS_F32 ? 4 : 2)) return DIFFUS_E_ALIGN;
    HuTable t{};
    t.m = m;
    for (int i = 0; i < m; i++) {
        if (!std::isfinite(hu_pts[i]) || !std::isfinite(z_pts[i])) return DIFFUS_E_PARAM;
        if (i > 0 && !(hu_pts[i] > hu_pts[i - 1])) return DIFFUS_E_PARAM;
        if ((float)hu_pts[i] != hu_pts[i]) return DIFFUS_E_PARAM;   // breakpoints are HU values (exact in float)
        t.hu[i] = (float)hu_pts[i];
        t.z[i] = (float)z_pts[i];
        t.slope[i] = i + 1 < m ? (float)((z_pts[i + 1] - z_pts[i]) / (hu_pts[i + 1] - hu_pts[i])) : 0.0f;
    }
    if (n == 0) return DIFFUS_OK;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // the lookup table pays when its entries, built once per block, are few
    // beside the voxels (16.7 M voxels, 7 breakpoints, 3001 entries, 304
    // blocks, from and to HBM: 33.0 us with the search, 20.7 with the table;
    // 3 breakpoints 23.4 and 20.5), but not for an FP32 map of one piece, whose
    // search is two comparisons (19.5 and 20.1 us; 17.7 and 20.2 us where the
    // L2 holds half of it)
    const double lo_d = std::max(-32768.0, std::floor(hu_pts[0])), hi_d = std::min(32767.0, std::ceil(hu_pts[m - 1]));
    const int64_t entries = lo_d <= hi_d ? (int64_t)(hi_d - lo_d) + 1 : 0;
    const int lut_blocks = 2 * sms;
    if (entries > 0 && entries <= kLutMax && (m > 2 || out_dtype == DIFFUS_BF16) && 4 * entries * lut_blocks <= n) {
        if (lut_smem_optin()) return DIFFUS_E_LAUNCH;
        const bool v16 = ((uintptr_t)hu) % 16 == 0 && ((uintptr_t)z_out) % 16 == 0;
        k_hu_lut<<<lut_blocks, kLutThreads, (size_t)entries * sizeof(float), (cudaStream_t)stream>>>(
            hu, n, t, (int)lo_d, (int)hi_d, out_dtype == DIFFUS_F32 ? (float *)z_out : nullptr,
            out_dtype == DIFFUS_BF16 ? (unsigned short *)z_out : nullptr, v16 ? 1 : 0);
        return launch_status();
    }
    // 16-byte loads (8 voxels) and, for FP32, 16-byte stores when aligned
    const bool vec = ((uintptr_t)hu) % 16 == 0 && (out_dtype != DIFFUS_F32 || ((uintptr_t)z_out) % 16 == 0);
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n / 8 + 255) / 256, (int64_t)sms * 16));
    k_hu_to_z<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(
        hu, n, t, out_dtype == DIFFUS_F32 ? (float *)z_out : nullptr,
        out_dtype == DIFFUS_BF16 ? (unsigned short *)z_out : nullptr, vec ? 1 : 0);
    return launch_status();
}
