// Ray setup, forward march and lateral blur kernels.
#pragma once

#include "march.cuh"

namespace dfs {

// A fan and the volume's placement as the ray setup needs them: the steps of
// depth and beam angle and the reciprocal spacings come from the host, because
// an FP64 division is some forty instructions on a pipe that takes 16 clocks
// for each (147 K rays: 53 us with the divisions, 33 us; a frame's setup 7.0 and
// 6.2 us).
struct FanDev {
    int n_rays, S;
    double half_fov, dth, ds;
};

inline FanDev make_fan(int n_rays, int S, double fov, double depth)
{
    return {n_rays, S, n_rays > 1 ? 0.5 * fov : 0.0, n_rays > 1 ? fov / (double)(n_rays - 1) : 0.0, depth / (double)S};
}

struct VolPlace {
    double isx, isy, isz, ox, oy, oz;
};

// Rotation R = Rz Ry Rx of ZYX Euler angles and its three partial
// derivatives, in double precision (pose angles are float inputs), from the
// angles' sines and cosines.  Every product and sum of the geometry is
// rounded as written (explicit intrinsics), so that every kernel that sets
// rays up gets the same positions bit for bit.
__device__ __forceinline__ double mul3(double a, double b, double c) { return __dmul_rn(__dmul_rn(a, b), c); }
__device__ __forceinline__ double mul3_add(double a, double b, double c, double d, double e)
{
    return __fma_rn(__dmul_rn(a, b), c, __dmul_rn(d, e));   // abc + de
}

__device__ __forceinline__ void rotation_zyx(const double sn[3], const double cs[3], double R[3][3], double dR[3][3][3])
{
    const double sx = sn[0], sy = sn[1], sz = sn[2], cx = cs[0], cy = cs[1], cz = cs[2];
    // R = Rz Ry Rx expanded
    R[0][0] = __dmul_rn(cz, cy); R[0][1] = mul3_add(cz, sy, sx, -sz, cx); R[0][2] = mul3_add(cz, sy, cx, sz, sx);
    R[1][0] = __dmul_rn(sz, cy); R[1][1] = mul3_add(sz, sy, sx, cz, cx);  R[1][2] = mul3_add(sz, sy, cx, -cz, sx);
    R[2][0] = -sy;               R[2][1] = __dmul_rn(cy, sx);             R[2][2] = __dmul_rn(cy, cx);
    // d/drx: differentiate the Rx factor
    dR[0][0][0] = 0; dR[0][0][1] = R[0][2]; dR[0][0][2] = -R[0][1];
    dR[0][1][0] = 0; dR[0][1][1] = R[1][2]; dR[0][1][2] = -R[1][1];
    dR[0][2][0] = 0; dR[0][2][1] = R[2][2]; dR[0][2][2] = -R[2][1];
    // d/dry
    dR[1][0][0] = __dmul_rn(-cz, sy); dR[1][0][1] = mul3(cz, cy, sx);     dR[1][0][2] = mul3(cz, cy, cx);
    dR[1][1][0] = __dmul_rn(-sz, sy); dR[1][1][1] = mul3(sz, cy, sx);     dR[1][1][2] = mul3(sz, cy, cx);
    dR[1][2][0] = -cy;                dR[1][2][1] = __dmul_rn(-sy, sx);   dR[1][2][2] = __dmul_rn(-sy, cx);
    // d/drz
    dR[2][0][0] = -R[1][0]; dR[2][0][1] = -R[1][1]; dR[2][0][2] = -R[1][2];
    dR[2][1][0] = R[0][0];  dR[2][1][1] = R[0][1];  dR[2][1][2] = R[0][2];
    dR[2][2][0] = 0;        dR[2][2][1] = 0;        dR[2][2][2] = 0;
}

// Fixed-point (2^-32 voxel) position and step.  No sample X0 + k DX, k = 0..S,
// may leave 64 bits, because everything after the setup counts on a line that
// is monotone along each axis: positions are clamped to 2^30 voxels, a fan is
// at most 2^29 voxels long, and the step of a pose that is not finite (NaN
// reaches here from the device, for example from a diverged optimiser) is 0,
// where the conversion would give the lowest integer, whose multiples wrap.
// Such a pose still shows in rg.v, and so in its gradient.
__host__ __device__ __forceinline__ long long round_fixed(double x)
{
#ifdef __CUDA_ARCH__
    return __double2ll_rn(__dmul_rn(x, 4294967296.0));
#else
    return llrint(x * 4294967296.0);
#endif
}

__host__ __device__ __forceinline__ long long to_fixed(double x)
{
    const double lim = 1073741824.0;   // 2^30 voxels: far outside any volume
    return round_fixed(fmin(fmax(x, -lim), lim));   // NaN: -lim
}

__host__ __device__ __forceinline__ long long step_fixed(double dx) { return dx == dx ? round_fixed(dx) : 0; }

// What the rays of one pose need from it (Section 2.4): columns 0 and 2 of
// R and of each dR/dr_q (a fan direction d = (sin th, 0, cos th) has no
// y component) and the translation, in FP64.  One thread per pose computes
// them, so the per-ray setup has a single sincos.
struct PoseFrame {
    double Rc[3][2];
    double dRc[3][3][2];
    double t[3];
};

__device__ __forceinline__ void pose_frame(const float *__restrict__ pose6, const double sn[3], const double cs[3],
                                           PoseFrame &f)
{
    double R[3][3], dR[3][3][3];
    rotation_zyx(sn, cs, R, dR);
    for (int i = 0; i < 3; i++) {
        f.Rc[i][0] = R[i][0];
        f.Rc[i][1] = R[i][2];
        for (int q = 0; q < 3; q++) {
            f.dRc[q][i][0] = dR[q][i][0];
            f.dRc[q][i][1] = dR[q][i][2];
        }
        f.t[i] = (double)pose6[i];
    }
}

static __global__ void k_pose_frames(const float *__restrict__ poses, int P, PoseFrame *__restrict__ frames)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    PoseFrame f;
    double sn[3], cs[3];
    for (int a = 0; a < 3; a++) sincos((double)poses[6 * (size_t)p + 3 + a], &sn[a], &cs[a]);
    pose_frame(poses + 6 * (size_t)p, sn, cs, f);
    frames[p] = f;
}

// FP64 voxel coordinates of sample 0 of ray `ray` and the step between
// samples (Section 2.4): sample k lies at x0 + k dx = (t + (k + 1/2) ds u -
// origin) / spacing (times the FP64 reciprocal).  st, ct: sin and cos of the beam angle.
__device__ __forceinline__ void beam_sincos(int ray, const FanDev &fan, double &st, double &ct)
{
    sincos(__fma_rn((double)ray, fan.dth, -fan.half_fov), &st, &ct);
}

// One axis of the line: Rc, t: the pose frame's row of that axis.
__device__ __forceinline__ void axis_line(const double Rc[2], double t, double ds, double isp, double org, double st,
                                          double ct, double &x0, double &dx)
{
    const double u = __fma_rn(Rc[0], st, __dmul_rn(Rc[1], ct));
    x0 = __dmul_rn(__dsub_rn(__fma_rn(__dmul_rn(0.5, ds), u, t), org), isp);
    dx = __dmul_rn(__dmul_rn(ds, u), isp);
}

__device__ __forceinline__ void ray_line(const PoseFrame &f, int ray, const FanDev &fan, const VolPlace &vp,
                                         double x0[3], double dx[3], double &st, double &ct)
{
    beam_sincos(ray, fan, st, ct);
    const double isp[3] = {vp.isx, vp.isy, vp.isz}, org[3] = {vp.ox, vp.oy, vp.oz};
    for (int i = 0; i < 3; i++) axis_line(f.Rc[i], f.t[i], fan.ds, isp[i], org[i], st, ct, x0[i], dx[i]);
}

__device__ __forceinline__ float dir_derivative(const double dRc[2], double st, double ct)
{
    return (float)__fma_rn(dRc[0], st, __dmul_rn(dRc[1], ct));
}

// Geometry of ray `ray` of pose `pose_idx` (Section 2.4): FP64 direction and
// fixed-point positions, exactly t + (k + 1/2) ds u in voxel coordinates.
__device__ __forceinline__ void setup_ray(const PoseFrame &f, int pose_idx, int ray, const FanDev &fan,
                                          const VolPlace &vp, RayGeo &out)
{
    double x0[3], dx[3], st, ct;
    ray_line(f, ray, fan, vp, x0, dx, st, ct);
    for (int i = 0; i < 3; i++) {
        out.X0[i] = to_fixed(x0[i]);
        out.DX[i] = step_fixed(dx[i]);
    }
    for (int q = 0; q < 3; q++)
        for (int i = 0; i < 3; i++) out.v[q][i] = dir_derivative(f.dRc[q][i], st, ct);
    out.pose = pose_idx;
    out.ray = ray;
    out.S = fan.S;
    out.ds = (float)fan.ds;
}

// Setup of one pose's rays in one launch: the pose frame, the ray table and
// (rows not null) the offsets that the backward's kernels read.  FP64 runs at
// two operations per clock and SM, so a warp's FP64 instruction takes 16 clocks
// whatever its lanes do: a block takes ten rays with one lane per ray and
// axis while a second warp works out the pose frame.  Frame kernel, ray kernel and offset kernel took 6.5 + 8.5 +
// 2 us for a frame; this one 7.0 us.  Above kSetupFrameRays rays the blocks'
// repeated pose frames cost more than the separate kernel.
constexpr int kSetupRays = 10;
constexpr int kSetupFrameRays = 4096;

struct RowOffsets {
    long long *row, *gz, *ck;
    int *ray0;
    int row_ld;
};

__device__ __forceinline__ void write_offsets(const RowOffsets &o, int j, int n, int S)
{
    o.row[j] = (long long)j * o.row_ld;
    o.gz[j] = (long long)j * gz_stride(S) + kGzLead;
    o.ck[j] = (long long)j * ((S + kSeg - 1) / kSeg);
    if (j == 0) {
        o.ray0[0] = 0;
        o.ray0[1] = n;
    }
}

static __global__ void __launch_bounds__(64) k_setup_frame(const float *__restrict__ pose6, FanDev fan, VolPlace vp,
                                                           PoseFrame *__restrict__ frame, RayGeo *__restrict__ geo,
                                                           RowOffsets off)
{
    __shared__ PoseFrame f;
    __shared__ double sn[3], cs[3];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int j = blockIdx.x * kSetupRays + lane / 3, a = lane % 3;
    const bool on = lane < 3 * kSetupRays && j < fan.n_rays;
    double st = 0.0, ct = 1.0;
    if (w == 1) {
        if (lane < 3) sincos((double)pose6[3 + lane], &sn[lane], &cs[lane]);
        __syncwarp();
        if (lane == 0) {
            pose_frame(pose6, sn, cs, f);
            if (blockIdx.x == 0) *frame = f;
        }
    } else if (on) {
        beam_sincos(j, fan, st, ct);
    }
    __syncthreads();
    if (w == 1 || !on) return;
    double x0, dx;
    axis_line(f.Rc[a], f.t[a], fan.ds, a == 0 ? vp.isx : (a == 1 ? vp.isy : vp.isz), a == 0 ? vp.ox : (a == 1 ? vp.oy : vp.oz),
              st, ct, x0, dx);
    RayGeo &g = geo[j];
    g.X0[a] = to_fixed(x0);
    g.DX[a] = step_fixed(dx);
    for (int q = 0; q < 3; q++) g.v[q][a] = dir_derivative(f.dRc[q][a], st, ct);
    if (a == 0) {
        g.pose = 0;
        g.ray = j;
        g.S = fan.S;
        g.ds = (float)fan.ds;
        if (off.row) write_offsets(off, j, fan.n_rays, fan.S);
    }
}

static __global__ void k_ray_setup(const PoseFrame *__restrict__ frame, FanDev fan, VolPlace vp,
                                   RayGeo *__restrict__ geo, RowOffsets off)
{
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= fan.n_rays) return;
    RayGeo rg;
    setup_ray(*frame, 0, j, fan, vp, rg);
    geo[j] = rg;
    if (off.row) write_offsets(off, j, fan.n_rays, fan.S);
}

inline void launch_setup(const float *pose, const FanDev &fd, const VolPlace &vp, PoseFrame *frame, RayGeo *geo,
                         const RowOffsets &off, cudaStream_t s)
{
    if (fd.n_rays <= kSetupFrameRays) {
        k_setup_frame<<<(fd.n_rays + kSetupRays - 1) / kSetupRays, 64, 0, s>>>(pose, fd, vp, frame, geo, off);
    } else {
        k_pose_frames<<<1, 32, 0, s>>>(pose, 1, frame);
        k_ray_setup<<<(fd.n_rays + 127) / 128, 128, 0, s>>>(frame, fd, vp, geo, off);
    }
}

// Per-pose sum of per-ray pose terms in FP64, one block per pose and one warp
// per component: lanes stride over the pose's rays, then a fixed shuffle tree
// (the same order for a frame and a batch).
static __global__ void __launch_bounds__(192) k_pose_reduce(const double *__restrict__ part,
                                                            const int *__restrict__ ray0,
                                                            float *__restrict__ grad_pose)
{
    const int p = blockIdx.x, q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = ray0[p + 1];
    double s = 0.0;
#pragma unroll 8
    for (int j = ray0[p] + lane; j < b; j += 32) s += part[6 * (size_t)j + q];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) grad_pose[6 * p + q] = (float)s;
}

// One warp per ray, kWarpsFwd warps per CTA.
constexpr int kWarpsFwd = 4;
// Resident warps per SM of the refined pass's kernels: 16 hold it at 128
// registers with no spills (measured on the 512^3 BF16 workload: refined
// forward+backward 11.39 ms with 8 warps per SM at 222 registers, 10.84 with
// 12 at 168, 10.69 with 16 at 126).
constexpr int kRefineWarpsPerSM = 16;

// Where the FP32 pass records the rays that need the refined pass (all null
// when refinement is off): per ray (segments to refine, first ill-posed depth
// of the FP32 pass), the list of such rays, its length and the refined
// pass's ticket counter.
struct RefineSel {
    int2 *rinfo;
    int *rlist;
    unsigned *rcount;
    unsigned *ticket;
};

template <typename T, int MODE, bool TRACK>
__global__ void __launch_bounds__(kWarpsFwd * 32) k_march_fwd(const T *__restrict__ vol, MarchArgs A,
                                                              const RayGeo *__restrict__ geo, int n_rays,
                                                              float *__restrict__ out, int *__restrict__ valid,
                                                              uint32_t *__restrict__ status, RefineSel sel)
{
    __shared__ float2 buf[kWarpsFwd][kSegPad];
    const int w = threadIdx.x >> 5;
    const int j = blockIdx.x * kWarpsFwd + w;
    if (j >= n_rays) return;
    RayGeo rg = geo[j];
    RayOut o{out + (size_t)j * rg.S, valid ? valid + j : nullptr, status, nullptr, nullptr, nullptr, nullptr,
             sel.rinfo ? sel.rinfo + j : nullptr, sel.rlist, sel.rcount, j, false};
    march_fwd_ray<T, MODE, TRACK, true, false>(vol, A, rg, o, buf[w]);
}

// One block per ray, up to kMultiWarps of its segments side by side: for fans
// too small to fill the GPU with one warp per ray, whose time is one ray's
// chain of segments (256 rays x 1024 rows: 24 us with one warp per ray, 9.4
// us with four).  The rows are the same bits (march_fwd_multi).
constexpr int kMultiWarps = 8;
constexpr int kMultiRays = 2432;     // 16 warps per SM: beyond, one warp per ray fills the GPU

template <typename T, int MODE, bool TRACK>
__global__ void __launch_bounds__(kMultiWarps * 32) k_march_fwd_multi(const T *__restrict__ vol, MarchArgs A,
                                                                     const RayGeo *__restrict__ geo,
                                                                     float *__restrict__ out, int *__restrict__ valid,
                                                                     uint32_t *__restrict__ status, RefineSel sel)
{
    __shared__ float2 buf[kMultiWarps][kSegPad];
    __shared__ MultiSmem<kMultiWarps> ms;
    const int j = blockIdx.x;
    const RayGeo rg = geo[j];
    RayOut o{out + (size_t)j * rg.S, valid ? valid + j : nullptr, status, nullptr, nullptr, nullptr, nullptr,
             sel.rinfo ? sel.rinfo + j : nullptr, sel.rlist, sel.rcount, j, false};
    march_fwd_multi<T, MODE, TRACK>(vol, A, rg, o, buf[threadIdx.x >> 5], ms);
}

// The refined pass of one ray that the FP32 pass listed: its FP64 line from
// the pose frame, then the refined march over the segments it recorded.
template <typename T, bool STREAM>
__device__ __forceinline__ void refine_ray(const T *__restrict__ vol, const MarchArgs &A, const RayGeo &rg,
                                           const PoseFrame &f, const FanDev &fan, const VolPlace &vp,
                                           const RayOut &out, int2 info, float *buf, float2 *dbuf)
{
    RayLine64 line;
    double st, ct;
    ray_line(f, rg.ray, fan, vp, line.x0, line.dx, st, ct);
    march_refine_ray<T, STREAM>(vol, A, rg, out, buf, dbuf, line, info);
}

// Refined pass of one pose: each warp takes listed rays from the ticket
// counter until the list (whose length the FP32 pass left in *rcount) is done.
template <typename T>
__global__ void __launch_bounds__(kWarpsFwd * 32, kRefineWarpsPerSM / kWarpsFwd) k_march_refine(const T *__restrict__ vol, MarchArgs A,
                                                                    const RayGeo *__restrict__ geo,
                                                                    const PoseFrame *__restrict__ frame, FanDev fan,
                                                                    VolPlace vp, float *__restrict__ out,
                                                                    int *__restrict__ valid,
                                                                    uint32_t *__restrict__ status, RefineSel sel)
{
    __shared__ float buf[kWarpsFwd][kSegPad];
    __shared__ float2 dbuf[kWarpsFwd][kSegPad];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned n = *sel.rcount;
    const PoseFrame f = *frame;
    for (;;) {
        unsigned q = 0;
        if (lane == 0) q = atomicAdd(sel.ticket, 1u);
        q = __shfl_sync(0xffffffffu, q, 0);
        if (q >= n) break;
        const int j = sel.rlist[q];
        const RayGeo rg = geo[j];
        RayOut o{out + (size_t)j * rg.S, valid ? valid + j : nullptr, status, nullptr, nullptr, nullptr, nullptr,
                 nullptr, nullptr, nullptr, j, false};
        refine_ray<T, false>(vol, A, rg, f, fan, vp, o, sel.rinfo[j], buf[w], dbuf[w]);
        __syncwarp();
    }
}

// ------------------------------------------------------------------ blur

constexpr int kBlurRows = 32;    // depth rows per strip (one per lane)
constexpr int kBlurStep = 8;     // rays entering the sliding window per step
constexpr int kBlurWarps = 4;    // strips (warps) per CTA

struct BlurArgs {
    float sigma0, sigma1;
    int W;
    int gain;              // depth-gain reading: the output row k carries a^(2(k+1))
};

// Gaussian weight of lateral offset m at echo row k (sigma in rays).
__device__ __forceinline__ float blur_w(const BlurArgs &b, int m, int k, float invS)
{
    float sig = fmaf(b.sigma1, (float)(k + 1) * invS, b.sigma0);
    if (!(sig > 0.0f)) return m == 0 ? 1.0f : 0.0f;
    float ex = -(float)(m * m) / (2.0f * sig * sig);
    return expf(ex);
}

// Lateral blur of one pose image (Section 2.4), or its transpose, on one
// strip of 32 echo rows [k0, k0 + 32) (one row per lane), output rays
// [j0, j1) of the n rays.
// in/out: [n] rows of S at strides si and so.
// Forward:   out[j] = sum_m w_m in[j+m] / N_j        (valid j+m)
// Transpose: out[j] = sum_m w_m in[j+m] / N_{j+m}    (valid j+m)
// with N_j = sum of w_m over the valid j+m.  The warp sweeps the rays once:
// every input element is read once, kBlurStep rows at a time into a
// register window of kBlurStep + 2W rows, and every output is written once,
// each access a coalesced 128-byte row segment (a ray range other than the
// whole fan also reads its 2W halo rays).  WT >= 0 is the half-width
// known at compile time; WT < 0 is the general path for wide kernels, which
// reads the window through the cache instead.
template <bool TRANSPOSE, int WT>
__device__ void blur_strip(const float *__restrict__ in, float *__restrict__ out, int n, int S, int si, int so,
                           const BlurArgs &b, int k0, int j0, int j1, float l2_hi, float l2_lo)
{
    const int lane = threadIdx.x & 31;
    const int k = k0 + lane;
    const bool kin = k < S;
    // the depth gain is constant along the strip lane's row and commutes
    // with the lateral blur (and its transpose): applied to the output
    const float gk = (b.gain && kin) ? depth_gain(l2_hi, l2_lo, k) : 1.0f;
    const float invS = 1.0f / (float)S;
    const float *src = in + (kin ? k : 0);
    float *dst = out + (kin ? k : 0);
    if (WT >= 0) {
        constexpr int WW = WT >= 0 ? WT : 0;
        constexpr int B = kBlurStep;
        float w[WW + 1];
#pragma unroll
        for (int m = 0; m <= WW; m++) w[m] = kin ? blur_w(b, m, k, invS) : (m == 0 ? 1.0f : 0.0f);
        float full = w[0];
#pragma unroll
        for (int m = 1; m <= WW; m++) full += 2.0f * w[m];
        const float rfull = 1.0f / full;
        auto rnorm = [&](int j) -> float {          // 1 / N_j
            if (j >= WW && j < n - WW) return rfull;
            float N = 0.0f;
#pragma unroll
            for (int m = -WW; m <= WW; m++)
                if (j + m >= 0 && j + m < n) N += w[m < 0 ? -m : m];
            return 1.0f / N;
        };
        auto ld = [&](int j) -> float {
            if (!kin || j < 0 || j >= n) return 0.0f;
            float x = __ldg(src + (size_t)j * si);
            if (TRANSPOSE) x *= rnorm(j);
            return x;
        };
        float win[B + 2 * WW];
#pragma unroll
        for (int t = 0; t < 2 * WW; t++) win[t] = ld(j0 + t - WW);
        for (int jb = j0; jb < j1; jb += B) {
            // a block whose rays all have the full window inside the fan (the
            // same for every lane): no edge guards and the interior norm;
            // the other lanes' rows of this block are read at row 0 (valid
            // memory) and not written; running pointers, because input and
            // output have their own strides (512 poses: blur 297 -> 295 us,
            // transpose 285 -> 267 us against an offset per row)
            if (jb >= WW && jb + B + 2 * WW <= n && jb + B <= j1) {
                const float *p = src + (size_t)(jb + WW) * si;
                float *q = dst + (size_t)jb * so;
#pragma unroll
                for (int t = 0; t < B; t++) {
                    const float x = __ldg(p);
                    p += si;
                    win[2 * WW + t] = TRANSPOSE ? x * rfull : x;
                }
#pragma unroll
                for (int i = 0; i < B; i++) {
                    float acc = w[0] * win[i + WW];
#pragma unroll
                    for (int m = 1; m <= WW; m++) acc = fmaf(w[m], win[i + WW - m] + win[i + WW + m], acc);
                    if (!TRANSPOSE) acc *= rfull;
                    if (kin) *q = acc * gk;
                    q += so;
                }
#pragma unroll
                for (int t = 0; t < 2 * WW; t++) win[t] = win[t + B];
                continue;
            }
            float nx[B];
#pragma unroll
            for (int t = 0; t < B; t++) nx[t] = (kin && jb + WW + t < n) ? __ldg(src + (size_t)(jb + WW + t) * si) : 0.0f;
#pragma unroll
            for (int t = 0; t < B; t++)
                win[2 * WW + t] = (TRANSPOSE && jb + WW + t < n) ? nx[t] * rnorm(jb + WW + t) : nx[t];
#pragma unroll
            for (int i = 0; i < B; i++) {
                const int j = jb + i;
                float acc = w[0] * win[i + WW];
#pragma unroll
                for (int m = 1; m <= WW; m++) acc = fmaf(w[m], win[i + WW - m] + win[i + WW + m], acc);
                if (kin && j < j1) {
                    if (!TRANSPOSE) acc *= rnorm(j);
                    dst[(size_t)j * so] = acc * gk;
                }
            }
#pragma unroll
            for (int t = 0; t < 2 * WW; t++) win[t] = win[t + B];
        }
        return;
    }
    if (!kin) return;
    const int W = b.W;
    auto wt = [&](int m) { return blur_w(b, m < 0 ? -m : m, k, invS); };
    auto N_of = [&](int j) {
        float N = 0.0f;
        for (int m = -W; m <= W; m++)
            if (j + m >= 0 && j + m < n) N += wt(m);
        return N;
    };
    auto ld = [&](int j) -> float {
        if (j < 0 || j >= n) return 0.0f;
        float x = __ldg(src + (size_t)j * si);
        if (TRANSPOSE) x *= 1.0f / N_of(j);
        return x;
    };
    for (int j = j0; j < j1; j++) {
        float acc = wt(0) * ld(j);
        for (int m = 1; m <= W; m++) acc = fmaf(wt(m), ld(j - m) + ld(j + m), acc);
        if (!TRANSPOSE) acc *= 1.0f / N_of(j);
        dst[(size_t)j * so] = acc * gk;
    }
}

// Single-pose blur: one warp per strip and range of kBlurSegRays rays (one
// pose alone is too small a grid for whole-fan strips).
constexpr int kBlurSegRays = 64;
// Rays per warp: fewer for small images, which are bound by one warp's sweep
// (64 rays x 256 rows: 14.6 us with 64 rays a warp, 5.6 us with 8), as long as the
// image does not fill the GPU's 608 schedulers; a range also reads 2W halo rays.
inline int blur_seg_rays(int strips, int n)
{
    int seg = kBlurSegRays;
    while (seg > kBlurStep && (int64_t)strips * ((n + seg - 1) / seg) < 608) seg /= 2;
    return seg;
}

template <bool TRANSPOSE, int WT>
__global__ void __launch_bounds__(kBlurWarps * 32) k_blur(const float *__restrict__ in, float *__restrict__ out,
                                                          int n, int S, int si, int so, int seg, BlurArgs b, float l2_hi,
                                                          float l2_lo)
{
    const int strip = blockIdx.x * kBlurWarps + (threadIdx.x >> 5);
    if (strip * kBlurRows >= S) return;
    const int j0 = blockIdx.y * seg;
    blur_strip<TRANSPOSE, WT>(in, out, n, S, si, so, b, strip * kBlurRows, j0, min(n, j0 + seg), l2_hi, l2_lo);
}

}  // namespace dfs
