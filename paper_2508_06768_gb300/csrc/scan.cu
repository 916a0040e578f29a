// Scan conversion of polar B-mode images to the fan-shaped display grid
// (Section 2.4, Fig. 3) and its adjoint.
//
// diffus_scan_plan (host, FP64) computes, once per fan and display grid,
// every display pixel's bilinear tap into the polar image (ray j0, row k0,
// fractions fv, fu; outside the fan: j0 = -1) and the transpose of that
// map as a CSR list per polar pixel (display pixel, weight) in pixel order.
// The forward kernel gathers 4 polar values per display pixel; the adjoint
// kernel gathers, per polar pixel, the weighted display gradients of its
// list, so it needs no atomics and its sums have a fixed order.  Both read
// their tap or list once for all images of a call.
#include <cmath>
#include <cstring>
#include <vector>

#include "host.hpp"

using namespace dfs;

namespace {

constexpr uint32_t kScanMagic = 0x44465343u;   // "DFSC"

template <typename T>
const T *at(const void *base, int64_t off) { return (const T *)((const char *)base + off); }

struct ScanTap {
    int32_t j0, k0;
    float fv, fu;
};

struct ScanEnt {
    uint32_t pixel;
    float w;
};

struct ScanHeader {
    uint32_t magic;
    int32_t n, S, W, H;
    int32_t pad;
    int64_t n_ent;
    int64_t off_map, off_rowptr, off_ent, bytes;
};

struct ScanGeom {
    int n, S, W, H;
    double fov, ds, x0, x1, z0, z1;
};

// Bilinear tap of display pixel (ix, iz); false outside the fan.
bool scan_tap(const ScanGeom &g, int ix, int iz, ScanTap &t, double &fv, double &fu)
{
    const double x = g.x0 + ((double)ix + 0.5) * (g.x1 - g.x0) / (double)g.W;
    const double z = g.z0 + ((double)iz + 0.5) * (g.z1 - g.z0) / (double)g.H;
    const double v = (std::atan2(x, z) + 0.5 * g.fov) * (double)(g.n - 1) / g.fov;   // fractional ray
    const double u = std::sqrt(x * x + z * z) / g.ds - 1.0;                          // fractional echo row
    if (!(v >= 0.0 && v <= (double)(g.n - 1) && u >= 0.0 && u <= (double)(g.S - 1))) return false;
    int j = (int)std::floor(v), k = (int)std::floor(u);
    j = j > g.n - 2 ? g.n - 2 : j;
    k = k > g.S - 2 ? g.S - 2 : k;
    fv = v - (double)j;
    fu = u - (double)k;
    t = ScanTap{j, k, (float)fv, (float)fu};
    return true;
}

int scan_geom(const diffus_fan *fan, const diffus_scan_grid *grid, ScanGeom &g)
{
    if (!fan || !grid) return DIFFUS_E_NULL;
    if (fan->n_rays < 2 || fan->n_samples < 2 || !(fan->fov_rad > 0.0) || !(fan->depth_mm > 0.0) ||
        !std::isfinite(fan->fov_rad) || !std::isfinite(fan->depth_mm))
        return DIFFUS_E_DIMS;
    if (grid->width < 1 || grid->height < 1 || (int64_t)grid->width * grid->height > (int64_t)1 << 30 ||
        !std::isfinite(grid->x0) || !std::isfinite(grid->x1) || !std::isfinite(grid->z0) ||
        !std::isfinite(grid->z1) || !(grid->x1 > grid->x0) || !(grid->z1 > grid->z0))
        return DIFFUS_E_PARAM;
    if ((int64_t)fan->n_rays * fan->n_samples >= (int64_t)1 << 31) return DIFFUS_E_DIMS;
    g = ScanGeom{fan->n_rays, fan->n_samples, grid->width, grid->height, fan->fov_rad,
                 fan->depth_mm / (double)fan->n_samples, grid->x0, grid->x1, grid->z0, grid->z1};
    return DIFFUS_OK;
}

int64_t scan_entries(const ScanGeom &g)
{
    int64_t e = 0;
    ScanTap t;
    double fv, fu;
    for (int iz = 0; iz < g.H; iz++)
        for (int ix = 0; ix < g.W; ix++)
            if (scan_tap(g, ix, iz, t, fv, fu)) e += 4;
    return e;
}

ScanHeader scan_layout(const ScanGeom &g, int64_t n_ent)
{
    ScanHeader h{};
    h.magic = kScanMagic;
    h.n = g.n;
    h.S = g.S;
    h.W = g.W;
    h.H = g.H;
    h.n_ent = n_ent;
    size_t o = align256(sizeof(ScanHeader));
    h.off_map = (int64_t)o;
    o = align256(o + sizeof(ScanTap) * (size_t)g.W * g.H);
    h.off_rowptr = (int64_t)o;
    o = align256(o + sizeof(uint32_t) * ((size_t)g.n * g.S + 1));
    h.off_ent = (int64_t)o;
    o = align256(o + sizeof(ScanEnt) * (size_t)n_ent);
    h.bytes = (int64_t)o;
    return h;
}

// Both kernels gather from the other side's image, whose lines run along its
// own x axis, so a warp takes a compact 2D patch rather than 32 neighbours of
// one line: the patch's taps then share lines on the other side.  What bounds
// them is the number of lines per load (L1 wavefronts), then the streams to
// HBM; a few images of a small display are bound by one thread's chain.
// 64 images of 256 x 1024 and a 1024 x 1024 display: forward 143 us with
// 32 x 1 pixels per warp, 105 us (3.4 TB/s) with 8 x 4; adjoint 531 us with 1 ray
// x 32 rows and 4 images per pass over the lists, 335 us with 4 x 8 and 8 images,
// 215 us with the image groups side by side instead of in turn, 198 us with 8
// rays x 4 rows.
constexpr int kScanTile = 256;                   // threads per block: 8 warps of 8 x 4 pixels, or of 4 rows x 8 rays
constexpr int kScanImgs = 8;                     // images per pass over the lists (adjoint)

// One thread per display pixel: the tap is read once and applied to the
// images of the block's group (blockIdx.z, GROUPED; else all), U images' taps in
// flight together.  A block is 2^cols warps wide and 8 / 2^cols high; tile0: the
// grid's first tile along its y axis.  U and the resident blocks MINB trade loads
// in flight against warps: one image of 256 x 1024 to 1024 x 1024 takes 5.0 us
// with 4 and 6, 4.65 with 2 and 8; 64 images 105 us with 4 and 5, 108 with 2 and 8.
template <int U, int MINB, bool GROUPED>
__global__ void __launch_bounds__(kScanTile, MINB)
    k_scan_fwd(const float *__restrict__ img, const ScanTap *__restrict__ map, int S, int64_t img_stride, int W, int H,
               int64_t npix, int cols, int tile0, int count, int group, float *__restrict__ out)
{
    constexpr bool kDown = U == 2;               // grid x runs down the display
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int wx = w & ((1 << cols) - 1), wy = w >> cols;
    const int gx = blockIdx.x, gy = blockIdx.y + tile0;
    const int ix = (((kDown ? gy : gx) << cols) + wx) * 8 + (lane & 7);
    const int iz = ((kDown ? gx : gy) * (8 >> cols) + wy) * 4 + (lane >> 3);
    if (ix >= W || iz >= H) return;
    const int64_t p = (int64_t)iz * W + ix;
    const ScanTap t = map[p];
    if (GROUPED) {
        const int c0 = blockIdx.z * group;
        img += (int64_t)c0 * img_stride;
        out += (int64_t)c0 * npix;
        count = min(count - c0, group);
    }
    out += p;
    if (t.j0 < 0) {
#pragma unroll 1
        for (; count > 0; count--, out += npix) *out = 0.0f;
        return;
    }
    const float a = (1.0f - t.fv) * (1.0f - t.fu), b = t.fv * (1.0f - t.fu);
    const float cc = (1.0f - t.fv) * t.fu, d = t.fv * t.fu;
    img += (int64_t)t.j0 * S + t.k0;
    for (; count >= U; count -= U) {
        float v[U][4];
#pragma unroll
        for (int u = 0; u < U; u++, img += img_stride) {
            v[u][0] = __ldg(img);
            v[u][1] = __ldg(img + S);
            v[u][2] = __ldg(img + 1);
            v[u][3] = __ldg(img + S + 1);
        }
#pragma unroll
        for (int u = 0; u < U; u++, out += npix)
            *out = fmaf(d, v[u][3], fmaf(cc, v[u][2], fmaf(b, v[u][1], a * v[u][0])));
    }
#pragma unroll 1
    for (; count > 0; count--, img += img_stride, out += npix)
        *out = fmaf(d, __ldg(img + S + 1), fmaf(cc, __ldg(img + 1), fmaf(b, __ldg(img + S), a * __ldg(img))));
}

// One thread per polar pixel: its list is read once for N gradients at a time,
// each summed in the list's fixed order.
template <int N>
__device__ __forceinline__ void scan_bwd_pass(const float *__restrict__ g, const ScanEnt *__restrict__ ent, uint32_t e0,
                                              uint32_t e1, int64_t npix, int64_t nq, float *__restrict__ out)
{
    float s[N];
#pragma unroll
    for (int u = 0; u < N; u++) s[u] = 0.0f;
    uint32_t e = e0;
    for (; e + 2 <= e1; e += 2) {          // two entries' loads in flight
        const ScanEnt x = ent[e], y = ent[e + 1];
        float gx[N], gy[N];
#pragma unroll
        for (int u = 0; u < N; u++) {
            gx[u] = __ldg(g + (int64_t)u * npix + x.pixel);
            gy[u] = __ldg(g + (int64_t)u * npix + y.pixel);
        }
#pragma unroll
        for (int u = 0; u < N; u++) s[u] = fmaf(y.w, gy[u], fmaf(x.w, gx[u], s[u]));
    }
    if (e < e1) {
        const ScanEnt x = ent[e];
#pragma unroll
        for (int u = 0; u < N; u++) s[u] = fmaf(x.w, __ldg(g + (int64_t)u * npix + x.pixel), s[u]);
    }
#pragma unroll
    for (int u = 0; u < N; u++) out[(int64_t)u * nq] = s[u];
}

__global__ void __launch_bounds__(kScanTile)
    k_scan_bwd(const float *__restrict__ gout, const uint32_t *__restrict__ rowptr, const ScanEnt *__restrict__ ent, int n,
               int S, int tiles_x, int64_t npix, int count, float *__restrict__ gimg)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = (blockIdx.x % tiles_x) * 32 + w * 4 + (lane & 3);
    const int j = (blockIdx.x / tiles_x) * 8 + (lane >> 2);
    if (k >= S || j >= n) return;
    const int64_t nq = (int64_t)n * S, q = (int64_t)j * S + k;
    const uint32_t e0 = rowptr[q], e1 = rowptr[q + 1];
    // one group of kScanImgs images per block row, what is left over in pairs
    int c = blockIdx.y * kScanImgs;
    const float *g = gout + (int64_t)c * npix;
    float *o = gimg + (int64_t)c * nq + q;
    const int m = min(kScanImgs, count - c);
    if (m == kScanImgs) {
        scan_bwd_pass<kScanImgs>(g, ent, e0, e1, npix, nq, o);
        return;
    }
    c = 0;
    for (; c + 2 <= m; c += 2) scan_bwd_pass<2>(g + (int64_t)c * npix, ent, e0, e1, npix, nq, o + (int64_t)c * nq);
    if (c < m) scan_bwd_pass<1>(g + (int64_t)c * npix, ent, e0, e1, npix, nq, o + (int64_t)c * nq);
}

// The same pass with no more than two entries' loads in flight, which lets every
// group size keep a pass of its own in one kernel's registers.
template <int N>
__device__ __forceinline__ void scan_bwd_rolled(const float *__restrict__ g, const ScanEnt *__restrict__ ent, uint32_t e0,
                                                uint32_t e1, int64_t npix, int64_t nq, float *__restrict__ out)
{
    float s[N];
#pragma unroll
    for (int u = 0; u < N; u++) s[u] = 0.0f;
#pragma unroll 1
    for (uint32_t e = e0; e + 2 <= e1; e += 2) {
        const ScanEnt x = ent[e], y = ent[e + 1];
        float gx[N], gy[N];
#pragma unroll
        for (int u = 0; u < N; u++) {
            gx[u] = __ldg(g + (int64_t)u * npix + x.pixel);
            gy[u] = __ldg(g + (int64_t)u * npix + y.pixel);
        }
#pragma unroll
        for (int u = 0; u < N; u++) s[u] = fmaf(y.w, gy[u], fmaf(x.w, gx[u], s[u]));
    }
    if ((e1 - e0) & 1) {
        const ScanEnt x = ent[e1 - 1];
#pragma unroll
        for (int u = 0; u < N; u++) s[u] = fmaf(x.w, __ldg(g + (int64_t)u * npix + x.pixel), s[u]);
    }
#pragma unroll
    for (int u = 0; u < N; u++) out[(int64_t)u * nq] = s[u];
}

// Calls of fewer than two full groups: one pass over the list whatever the
// group's size, where the pairs above read it up to four times.  64 rays x 256
// rows and a 1024 x 1024 display: three images 88.8 us in pairs, 67.6; seven 184
// and 131 us; three of 256 x 1024 22.6 and 17.8 us.  With two full groups and
// more the pairs are a small part, and the kernel above, whose loop over a full
// group the compiler schedules with fewer loads in flight, keeps more of a small
// display in L1 (30 images of 64 x 256: 387 us, 475 with one pass per group).
__global__ void __launch_bounds__(kScanTile, 6)
    k_scan_bwd_few(const float *__restrict__ gout, const uint32_t *__restrict__ rowptr, const ScanEnt *__restrict__ ent,
                   int n, int S, int tiles_x, int64_t npix, int count, float *__restrict__ gimg)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = (blockIdx.x % tiles_x) * 32 + w * 4 + (lane & 3);
    const int j = (blockIdx.x / tiles_x) * 8 + (lane >> 2);
    if (k >= S || j >= n) return;
    const int64_t nq = (int64_t)n * S, q = (int64_t)j * S + k;
    const uint32_t e0 = rowptr[q], e1 = rowptr[q + 1];
    const int c = blockIdx.y * kScanImgs;
    const float *g = gout + (int64_t)c * npix;
    float *o = gimg + (int64_t)c * nq + q;
    switch (min(kScanImgs, count - c)) {
    case 1: scan_bwd_pass<1>(g, ent, e0, e1, npix, nq, o); break;
    case 2: scan_bwd_pass<2>(g, ent, e0, e1, npix, nq, o); break;
    case 3: scan_bwd_rolled<3>(g, ent, e0, e1, npix, nq, o); break;
    case 4: scan_bwd_rolled<4>(g, ent, e0, e1, npix, nq, o); break;
    case 5: scan_bwd_rolled<5>(g, ent, e0, e1, npix, nq, o); break;
    case 6: scan_bwd_rolled<6>(g, ent, e0, e1, npix, nq, o); break;
    case 7: scan_bwd_rolled<7>(g, ent, e0, e1, npix, nq, o); break;
    default: scan_bwd_rolled<kScanImgs>(g, ent, e0, e1, npix, nq, o); break;
    }
}

int check_scan_plan(const void *plan_host, const void *plan_dev)
{
    if (!plan_host || !plan_dev) return DIFFUS_E_NULL;
    if (((uintptr_t)plan_dev) % 256) return DIFFUS_E_ALIGN;
    const ScanHeader &h = *(const ScanHeader *)plan_host;
    if (h.magic != kScanMagic) return DIFFUS_E_PLAN;
    return DIFFUS_OK;
}

}  // namespace

extern "C" size_t diffus_scan_plan_bytes(const diffus_fan *fan, const diffus_scan_grid *grid)
{
    ScanGeom g;
    if (scan_geom(fan, grid, g)) return 0;
    return (size_t)scan_layout(g, scan_entries(g)).bytes;
}

extern "C" int diffus_scan_plan(const diffus_fan *fan, const diffus_scan_grid *grid, void *plan_host,
                                size_t plan_bytes)
{
    NvtxRange nvtx_range("diffus_scan_plan");
    ScanGeom g;
    int rc = scan_geom(fan, grid, g);
    if (rc) return rc;
    if (!plan_host) return DIFFUS_E_NULL;
    const ScanHeader h = scan_layout(g, scan_entries(g));
    if (plan_bytes < (size_t)h.bytes) return DIFFUS_E_WORKSPACE;
    char *base = (char *)plan_host;
    std::memset(base, 0, (size_t)h.bytes);
    std::memcpy(base, &h, sizeof h);
    ScanTap *map = (ScanTap *)(base + h.off_map);
    uint32_t *rowptr = (uint32_t *)(base + h.off_rowptr);
    ScanEnt *ent = (ScanEnt *)(base + h.off_ent);
    const size_t nq = (size_t)g.n * g.S;
    std::vector<double> wts;
    // taps, and the number of list entries of every polar pixel
    std::vector<uint32_t> cnt(nq + 1, 0);
    for (int iz = 0; iz < g.H; iz++)
        for (int ix = 0; ix < g.W; ix++) {
            ScanTap t;
            double fv, fu;
            const size_t p = (size_t)iz * g.W + ix;
            if (!scan_tap(g, ix, iz, t, fv, fu)) {
                map[p] = ScanTap{-1, -1, 0.0f, 0.0f};
                continue;
            }
            map[p] = t;
            const size_t q = (size_t)t.j0 * g.S + t.k0;
            cnt[q]++;
            cnt[q + g.S]++;
            cnt[q + 1]++;
            cnt[q + g.S + 1]++;
        }
    rowptr[0] = 0;
    for (size_t q = 0; q < nq; q++) rowptr[q + 1] = rowptr[q] + cnt[q];
    std::vector<uint32_t> fill(rowptr, rowptr + nq);
    // transpose in display-pixel order, weights from the FP64 fractions
    for (int iz = 0; iz < g.H; iz++)
        for (int ix = 0; ix < g.W; ix++) {
            ScanTap t;
            double fv, fu;
            if (!scan_tap(g, ix, iz, t, fv, fu)) continue;
            const uint32_t p = (uint32_t)((size_t)iz * g.W + ix);
            const size_t q = (size_t)t.j0 * g.S + t.k0;
            ent[fill[q]++] = ScanEnt{p, (float)((1.0 - fv) * (1.0 - fu))};
            ent[fill[q + g.S]++] = ScanEnt{p, (float)(fv * (1.0 - fu))};
            ent[fill[q + 1]++] = ScanEnt{p, (float)((1.0 - fv) * fu)};
            ent[fill[q + g.S + 1]++] = ScanEnt{p, (float)(fv * fu)};
        }
    return DIFFUS_OK;
}

extern "C" int diffus_scan_convert(const float *images, int32_t count, const void *plan_host, const void *plan_dev,
                                   float *out, diffus_stream_t stream)
{
    NvtxRange nvtx_range("diffus_scan_convert");
    int rc = check_scan_plan(plan_host, plan_dev);
    if (rc) return rc;
    if (!images || !out) return DIFFUS_E_NULL;
    if (count < 1 || count > 65535) return DIFFUS_E_PARAM;
    if (((uintptr_t)images) % 4 || ((uintptr_t)out) % 4) return DIFFUS_E_ALIGN;
    const ScanHeader &h = *(const ScanHeader *)plan_host;
    int cols = 2;                          // fewer warp columns for a display narrower than four
    while (cols > 0 && (4 << cols) >= h.W) cols--;
    const int tx = (h.W + (8 << cols) - 1) / (8 << cols), ty = (h.H + (32 >> cols) - 1) / (32 >> cols);
    // a display of fewer than four tiles per SM takes its images in groups side
    // by side (64 images of 64 x 256 to 256 x 256: 16.7 us in turn, 10.2; at 512 x
    // 512, seven tiles per SM, eight images take 5.5 us in turn, 6.1 in two groups)
    int group = count;
    while (group >= 8 && (int64_t)tx * ty * ((count + group - 1) / group) < 608) group = (group + 1) / 2;
    // up to three images never fill a step of four
    const bool few = count <= 3;
    auto kernel = few ? k_scan_fwd<2, 8, false> : group < count ? k_scan_fwd<4, 5, true> : k_scan_fwd<4, 5, false>;
    const int gx = few ? ty : tx, gy = few ? tx : ty;
    for (int t0 = 0; t0 < gy; t0 += 65535) {   // the grid's y axis has 65535 places
        const dim3 grid((unsigned)gx, (unsigned)(gy - t0 < 65535 ? gy - t0 : 65535), (unsigned)((count + group - 1) / group));
        kernel<<<grid, kScanTile, 0, (cudaStream_t)stream>>>(images, at<ScanTap>(plan_dev, h.off_map), h.S,
                                                             (int64_t)h.n * h.S, h.W, h.H, (int64_t)h.W * h.H, cols, t0,
                                                             count, group, out);
    }
    return launch_status();
}

extern "C" int diffus_scan_convert_bwd(const float *grad_out, int32_t count, const void *plan_host,
                                       const void *plan_dev, float *grad_images, diffus_stream_t stream)
{
    NvtxRange nvtx_range("diffus_scan_convert_bwd");
    int rc = check_scan_plan(plan_host, plan_dev);
    if (rc) return rc;
    if (!grad_out || !grad_images) return DIFFUS_E_NULL;
    if (count < 1 || count > 65535) return DIFFUS_E_PARAM;
    if (((uintptr_t)grad_out) % 4 || ((uintptr_t)grad_images) % 4) return DIFFUS_E_ALIGN;
    const ScanHeader &h = *(const ScanHeader *)plan_host;
    const int tx = (h.S + 31) / 32, ty = (h.n + 7) / 8;
    const dim3 bgrid((unsigned)((int64_t)tx * ty), (unsigned)((count + kScanImgs - 1) / kScanImgs));
    const bool few = count < 2 * kScanImgs && count != kScanImgs;   // see k_scan_bwd_few
    auto kernel = few ? k_scan_bwd_few : k_scan_bwd;
    kernel<<<bgrid, kScanTile, 0, (cudaStream_t)stream>>>(grad_out, at<uint32_t>(plan_dev, h.off_rowptr),
                                                          at<ScanEnt>(plan_dev, h.off_ent), h.n, h.S, tx,
                                                          (int64_t)h.W * h.H, count, grad_images);
    return launch_status();
}
