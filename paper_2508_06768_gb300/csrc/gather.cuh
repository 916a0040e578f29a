// Atomic-free, deterministic gather of the volume gradient.
//
// dL/dvol[v] = sum over samples s of dL/dZ_s * w_v(p_s), the transpose of
// trilinear sampling.  Work is organised by brick of 8^3 cells:
//
//  1. runs:   every ray walks the bricks its (clamped) cells pass through, a
//             3D DDA on the exact fixed-point line; clamping is monotone
//             along a ray, so each brick is one run [k0, k1] of samples.
//  2. sort:   the runs, written at fixed slots (run i of ray r at slot
//             i * n_rays + r), are put in order of brick, then slot: by a
//             stable radix sort, or, for a frame or a few, by placing each
//             in its brick's range and counting the smaller slots there.
//             Either way every brick's runs appear in slot order whatever
//             the launch schedule.
//  3. units:  each brick's runs are cut into units of at most unit_runs() runs
//             (hot bricks crossed by many poses spread over many CTAs).
//  4. gather: one warp per unit accumulates its samples into the 9^3 voxels
//             the brick's cells touch, in a shared-memory copy of its own.
//             Each lane walks one run, one cell at a time, summing moments
//             of dL/dZ; cell records on equal cells are combined in lane
//             order and written one corner at a time, so no two lanes
//             update a voxel at once.  The copy is the unit's partial.
//  5. reduce: each voxel sums the partials of the units of the (up to 8)
//             bricks whose cells touch it, in a fixed order.
//
// The same cell moments give the pose gradient (Section 2.5): inside a cell
// the derivative of the trilinear form along each axis is a quadratic in the
// sample index, so sum_k dL/dZ_k dZ/dx_a(k) and its depth-weighted twin
// follow from the moments and the cell's 8 corners.  Each lane sums them over
// its run and writes them at the run's slot; a per-ray pass adds a ray's runs
// in slot order.  The adjoint march then samples values only.
//
// No floating-point atomics are used and every sum has a fixed order, so the
// gradient is bitwise reproducible.
#pragma once

#include "common.cuh"

namespace dfs {

constexpr int kBrick = 8;
constexpr int kBrickV = kBrick + 1;            // voxels touched by a brick's cells, per axis
constexpr int kBrickVox = kBrickV * kBrickV * kBrickV;
constexpr int kGatherWarps = 4;
// Runs per unit.  A warp walks a unit's runs 32 at a time, so a unit of n
// runs is n/32 run walks in series (about 20 us each); more units cost more
// partials (729 floats each).  Large problems fill the GPU with units of 256;
// below, units shrink to one run per lane.  The cut-offs are plain ones: with
// about four slots per run each allows some 8000 units, a little more than two
// per resident warp (152 SMs x 24).  Measured with 256 and with 32: a 251-ray
// frame's unit kernel 182 and 43 us, nine small frames' 132 and 45 us; 512 frames
// stay at 256.
__host__ __device__ inline int unit_runs(size_t slots)
{
    return slots <= (1u << 20) ? 32 : slots <= (1u << 21) ? 64 : slots <= (1u << 22) ? 128 : 256;
}

struct GatherArgs {
    int nx, ny, nz;
    int nbx, nby, nbz;                // bricks of cells per axis (cells 0..n-2)
};

// Samples k0 .. k0+len-1 of one ray lie in cells of one brick: where the run
// starts, and for each axis the samples before its first crossing of a cell
// face (kNextBits bits each, at most kNextMax).
struct alignas(16) Run {
    long long X, Y, Z;
    int ray, k0, len;
    uint32_t next;
    uint32_t pad[2];
};
static_assert(sizeof(Run) == 48, "Run layout");
constexpr int kNextBits = 10;
constexpr int kNextMax = (1 << kNextBits) - 1;

// What every run of a ray needs to step from cell to cell.  Along an axis with
// step e = |d| (2^-32 voxel) the samples between two crossings are q or q + 1,
// q = floor(2^32 / e): a crossing leaves the position less than e inside the
// new cell, so with r = 2^32 - q e the next one comes after q + (rem < r)
// samples, rem the position's fraction counted in the direction of travel.  v is
// d / 2^32 as a float (the slope of the cell weights).
struct alignas(16) RayStep {
    long long d[3], g_off;   // step per axis; offset of the ray's first dL/dZ value
    uint2 qr[3];
    float v[3], pad[3];
};
static_assert(sizeof(RayStep) == 80, "RayStep layout");

__host__ __device__ __forceinline__ uint2 cell_steps(long long d)
{
    const unsigned long long e = (unsigned long long)(d < 0 ? -d : d);
    if (e <= 1) return make_uint2(0xffffffffu, 0u);      // (never within a run)
    if (e >> 32) return make_uint2(1u, 0u);              // a crossing at every sample
    const uint32_t e32 = (uint32_t)e, q = 0xffffffffu / e32, r = 0xffffffffu - q * e32;   // 2^32 = q e + r + 1
    return r + 1 == e32 ? make_uint2(q + 1, 0u) : make_uint2(q, r + 1);
}

// A 64-bit fixed-point quantity as a float, from two 32-bit conversions
// (high word x 2^32 + low word): within about an ulp.  The direct 64-bit
// integer conversion runs on the FP64 pipe, which is narrow on this part;
// every use here is an estimate that exact integer tests correct, or the
// weight slope of a cell record.
__host__ __device__ __forceinline__ float ll_to_float(long long x)
{
    return fmaf((float)(int)(x >> 32), 4294967296.0f, (float)(unsigned)(x & 0xffffffffll));
}

// An estimate of a / b (every use is corrected with exact integer tests).
__host__ __device__ __forceinline__ float quotient_estimate(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}

// First k in [0, kmax+1] with X0 + k DX >= L for DX > 0, or kmax+1 if no
// k <= kmax qualifies.  Exact in fixed point: the float estimate is off by
// at most a step or two and is corrected with integer tests.
__host__ __device__ __forceinline__ long long first_at_or_above(long long X0, long long DX, long long L, long long kmax)
{
    if (X0 >= L) return 0;
    if (X0 + (kmax + 1) * DX < L) return kmax + 1;
    float est = ceilf(quotient_estimate(ll_to_float(L - X0), ll_to_float(DX)));
    est = fminf(fmaxf(est, 0.0f), (float)(int)(kmax + 1));   // kmax < 2^31: 32-bit conversions
    long long k = (long long)(int)est;
    while (k > 0 && X0 + (k - 1) * DX >= L) k--;
    while (k <= kmax && X0 + k * DX < L) k++;
    return k;
}

// k at which the brick index of one axis changes next, for a ray whose
// brick index on that axis is b (kmax + 1 when it never does).
__host__ __device__ __forceinline__ long long next_change(long long X0, long long DX, int b, int n, long long kmax)
{
    if (DX > 0) {
        int c = (b + 1) * kBrick;               // first cell of the next brick
        if (c > n - 2) return kmax + 1;
        return first_at_or_above(X0, DX, (long long)c << 32, kmax);
    }
    if (DX < 0) {
        if (b == 0) return kmax + 1;
        // cell < 8b  <=>  X < 8b * 2^32  <=>  -X >= -(8b * 2^32) + 1
        long long L = -(((long long)(b * kBrick)) << 32) + 1;
        return first_at_or_above(-X0, -DX, L, kmax);
    }
    return kmax + 1;
}

__host__ __device__ __forceinline__ int cell_of(long long X, int n)
{
    int hi = (int)(X >> 32);
    return X < 0 ? 0 : (hi > n - 2 ? n - 2 : hi);
}

// A ray's brick crossings, for the run pass that solves them independently: the
// brick index of an axis is monotone along the ray, so axis a is crossed
// off[a+1] - off[a] times, as entries off[a] .. off[a+1]-1 of the ray's list.
// A ray crosses at most cap - 1 <= kRunMax times (runs_per_ray); one that did
// not keep to that has no entries (fits = false), because a list cut short
// would put the missing bricks' samples into other bricks' runs.
constexpr int kRunMax = 255;

struct Cuts {
    int b0[3], off[4];
    bool fits;
};

__host__ __device__ __forceinline__ Cuts ray_cuts(const long long X0[3], const long long DX[3], int S, const int n[3])
{
    Cuts c;
    c.off[0] = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        c.b0[a] = cell_of(X0[a], n[a]) / kBrick;
        const int b1 = cell_of(X0[a] + (long long)S * DX[a], n[a]) / kBrick;
        c.off[a + 1] = c.off[a] + abs(b1 - c.b0[a]);
    }
    c.fits = c.off[3] <= kRunMax;
    if (!c.fits) c.off[1] = c.off[2] = c.off[3] = 0;
    return c;
}

__host__ __device__ __forceinline__ int cut_axis(const Cuts &c, int e) { return e < c.off[1] ? 0 : (e < c.off[2] ? 1 : 2); }

// The sample that crosses at entry e.
__host__ __device__ __forceinline__ int cut_sample(const Cuts &c, int e, const long long X0[3], const long long DX[3],
                                                   int S)
{
    const int a = cut_axis(c, e);
    const int j = e - (a == 0 ? 0 : (a == 1 ? c.off[1] : c.off[2]));
    const long long x = a == 0 ? X0[0] : (a == 1 ? X0[1] : X0[2]);
    const long long d = a == 0 ? DX[0] : (a == 1 ? DX[1] : DX[2]);
    const int b = a == 0 ? c.b0[0] : (a == 1 ? c.b0[1] : c.b0[2]);
    if (d > 0) return (int)first_at_or_above(x, d, (long long)((b + j + 1) * kBrick) << 32, S);
    // cell < 8c  <=>  -X >= -(8c << 32) + 1
    return (int)first_at_or_above(-x, -d, -((long long)((b - j) * kBrick) << 32) + 1, S);
}

__host__ __device__ __forceinline__ int count_below(const int *k, int n, int v, bool or_equal)
{
    int lo = 0;
    while (n > 0) {
        const int h = n >> 1;
        const int m = k[lo + h];
        if (m < v || (or_equal && m == v)) {
            lo += h + 1;
            n -= h + 1;
        } else {
            n = h;
        }
    }
    return lo;
}

// Entry e's place in the merged order of all m entries (equal samples: lower
// axis first).
__host__ __device__ __forceinline__ int cut_rank(const Cuts &c, const int *k, int m, int e)
{
    const int a = cut_axis(c, e), v = k[e];
    int pos = e - (a == 0 ? 0 : (a == 1 ? c.off[1] : c.off[2]));
    if (a != 0) pos += count_below(k, c.off[1], v, true);
    if (a != 1) pos += count_below(k + c.off[1], c.off[2] - c.off[1], v, a == 2);
    if (a != 2) pos += count_below(k + c.off[2], m - c.off[2], v, false);
    return pos;
}

// Samples [k0, k1) of run i of the ray's cnt runs (start: the first sample of
// runs 1 .. cnt-1).  A run ends where the next one starts, whether or not that
// one has a slot.
__host__ __device__ __forceinline__ void run_span(const int *start, int i, int cnt, int S, int &k0, int &k1)
{
    k0 = i ? start[i - 1] : 0;
    k1 = i + 1 < cnt ? start[i] : S + 1;
}

template <bool POSE>
struct GatherSmem {
    float acc[kGatherWarps][kBrickVox];
    float vox[POSE ? kGatherWarps : 1][POSE ? kBrickVox : 1];   // the brick's volume values (pose terms)
    uint2 qr[kGatherWarps][3][32];                               // the lane's ray: cell steps and
    float slope[kGatherWarps][3][32];                            // weight slopes
};

// Adds one closed cell record per flagged lane into the warp's accumulator.
// Records on the same cell are grouped with a warp match and added into the
// group's lowest lane in lane order (base: the cell's first voxel in the
// accumulator); the group leaders, all on distinct
// cells, then write one corner at a time: for a fixed corner offset
// distinct cells hit distinct voxels.
__device__ __forceinline__ void flush_records(bool fl, int base, float (&fv)[8], float *acc, int lane,
                                              unsigned lt)
{
    const int key = fl ? base : 1024 + lane;
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    const bool leader = (grp & lt) == 0;
    unsigned rest = (fl && leader) ? (grp & (grp - 1u)) : 0u;   // other members, lane order
    if (__any_sync(0xffffffffu, rest != 0u)) {
        const int rounds = (int)__reduce_max_sync(0xffffffffu, (unsigned)__popc(rest));
        for (int t = 0; t < rounds; t++) {
            const int src = rest ? __ffs(rest) - 1 : lane;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const float o = __shfl_sync(0xffffffffu, fv[q], src);
                if (rest) fv[q] += o;
            }
            rest &= rest - 1u;
        }
    }
    const bool writes = fl && leader;
#pragma unroll
    for (int q = 0; q < 8; q++) {
        if (writes) {
            const int off = ((q >> 2) * kBrickV + ((q >> 1) & 1)) * kBrickV + (q & 1);
            acc[base + off] += fv[q];
        }
        __syncwarp();
    }
}

constexpr int kGCellCap = 32;  // samples of one cell record at most (bounds the moment orders)

// One axis of a run position inside its current cell: the cell index i, and
// the trilinear weight of the upper corner as u + v k for the next samples
// k = 0, 1, ... (exact in the clamped regions, where v = 0), plus the number
// of samples before the cell or the clamping changes (at most cap).
// Boundaries are found exactly on the fixed-point line: the float estimate
// of ceil(num / den) is corrected with integer tests.
__host__ __device__ __forceinline__ int ceil_div_fixed(long long num, long long den, int cap)
{
    // smallest k >= 1 with k den >= num (num >= 1, den >= 1), at most cap
    float est = ceilf(quotient_estimate(ll_to_float(num), ll_to_float(den)));
    long long k = est < 1.0f ? 1 : (est > (float)cap ? cap : (long long)(int)est);
    while (k > 1 && (k - 1) * den >= num) k--;
    while (k < cap && k * den < num) k++;
    return (int)k;
}

// Cell index i and upper-corner weight u + v k of one axis at position X
// (exact in the clamped regions, where v = 0); vd = d / 2^32.
__host__ __device__ __forceinline__ void axis_cell(long long X, float vd, int n, int &i, float &u, float &v)
{
    const int hi = (int)(X >> 32);
    i = hi;
    u = frac23((unsigned)X);
    v = vd;
    if (hi < 0) {
        i = 0;
        u = 0.0f;
        v = 0.0f;
    } else if (hi >= n - 1) {
        i = n - 2;
        u = 1.0f;
        v = 0.0f;
    }
}

// dX / 2^32 as a float.
__host__ __device__ __forceinline__ float slope_of(long long dX)
{
    return fmaf((float)(unsigned)(dX & 0xffffffffll), 2.3283064365386963e-10f, (float)(int)(dX >> 32));
}

// Samples from X (inclusive) before the axis's cell or its clamping changes
// (at most cap): the next crossing of a cell face, of 0 from below or of
// n-1 from above.  A sample exactly at coordinate 0 forms a record of its
// own: there the sampler's gradient along the axis is zero (the coordinate
// is not strictly inside the volume), so every record is either wholly
// strictly inside or wholly not, along each axis.
__host__ __device__ __forceinline__ int axis_steps(long long X, long long dX, int n, int cap)
{
    const long long top = (long long)(n - 1) << 32;
    if (X < 0) return dX > 0 ? ceil_div_fixed(-X, dX, cap) : cap;
    if (X >= top) return dX < 0 ? ceil_div_fixed(X - top + 1, -dX, cap) : cap;
    if (X == 0 && dX != 0) return 1;
    const long long c = X >> 32;
    if (dX > 0) return ceil_div_fixed(((c + 1) << 32) - X, dX, cap);
    if (dX < 0) return ceil_div_fixed(X - (c << 32) + (c == 0 ? 0 : 1), -dX, cap);
    return cap;
}

// The derivative along one axis of the trilinear form, over a cell record,
// as a quadratic p0 + p1 k + p2 k^2 in the record's sample index k.  D[i][j]
// are the corner differences along the axis at the other two axes' corners
// i (weight u + v k of corner 1) and j (weight w + t k of corner 1).
__device__ __forceinline__ void axis_poly(float D00, float D10, float D01, float D11, float u, float v, float w,
                                          float t, float &p0, float &p1, float &p2)
{
    const float h0 = D10 - D00, h1 = D11 - D01;
    const float e00 = fmaf(h0, u, D00), e01 = h0 * v;    // j = 0: e00 + e01 k
    const float e10 = fmaf(h1, u, D01), e11 = h1 * v;    // j = 1
    const float f0 = e10 - e00, f1 = e11 - e01;
    p0 = fmaf(f0, w, e00);
    p1 = fmaf(f1, w, fmaf(f0, t, e01));
    p2 = f1 * t;
}

constexpr int kGStepCap = 1 << 24;   // "no crossing within the run"

// axis_steps at a position that a crossing of this axis has just reached: in
// an inner cell the count comes from (q, r); next to the volume's faces, in the
// clamped regions and for steps so small that a run's first count was cut at
// kNextMax, from axis_steps (512 frames: 173 M warp instructions per 34 M
// samples with that division at every crossing, 142 M).
__host__ __device__ __forceinline__ int next_steps(long long X, long long dX, int n, uint2 qr)
{
    const int hi = (int)(X >> 32);
    if ((unsigned)(hi - 1) < (unsigned)(n - 2) && qr.x < (unsigned)(kNextMax - 1)) {
        const unsigned rem = (unsigned)X ^ (unsigned)((int)(dX >> 32) >> 31);
        return (int)qr.x + (rem < qr.y);
    }
    return axis_steps(X, dX, n, kGStepCap);
}

// The same at any position.  With t the distance to the last position of the
// cell in the direction of travel (a 32-bit number), the next crossing comes
// after floor(t / e) + 1 samples; inv = 1 / e estimates the quotient (below
// kNextMax, so off by one at most) and an exact product corrects it.
__host__ __device__ __forceinline__ int first_steps1(long long X, long long dX, uint32_t q, float inv, int n)
{
    const int hi = (int)(X >> 32);
    if ((unsigned)(hi - 1) < (unsigned)(n - 2) && q < (unsigned)(kNextMax - 1)) {
        const bool neg = dX < 0;
        const unsigned t = neg ? (unsigned)X : ~(unsigned)X;
        const unsigned long long e = (unsigned long long)(neg ? -dX : dX);
        if (e >> 32) return 1;
        unsigned k = (unsigned)((float)t * inv);
        const long long r = (long long)t - (long long)((unsigned long long)k * (unsigned)e);
        if (r < 0)
            k--;
        else if (r >= (long long)e)
            k++;
        return (int)k + 1;
    }
    return axis_steps(X, dX, n, kNextMax);
}

// A ray's steps as its runs' first counts need them.
struct FirstSteps {
    uint32_t q[3];
    float inv[3];
};

__host__ __device__ __forceinline__ FirstSteps first_steps_of(const long long d[3])
{
    FirstSteps f;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        f.q[a] = cell_steps(d[a]).x;
        f.inv[a] = 1.0f / fmaxf(fabsf(ll_to_float(d[a])), 1.0f);
    }
    return f;
}

// The three first counts of a run, packed.
__host__ __device__ __forceinline__ uint32_t first_steps(long long X, long long Y, long long Z, const long long d[3],
                                                const FirstSteps &f, int nx, int ny, int nz)
{
    return (uint32_t)first_steps1(X, d[0], f.q[0], f.inv[0], nx) |
           ((uint32_t)first_steps1(Y, d[1], f.q[1], f.inv[1], ny) << kNextBits) |
           ((uint32_t)first_steps1(Z, d[2], f.q[2], f.inv[2], nz) << (2 * kNextBits));
}

// Pose-gradient sums of one run, written at the run's slot: component q
// (T_x, T_y, T_z, U_x, U_y, U_z) at rpart[q * slots + slot], with
// T_a = sum_k dL/dZ_k dZ/dx_a(k) and U_a = sum_k dL/dZ_k (k + 1/2) dZ/dx_a(k)
// in voxel-index units (k along the ray).
struct PoseOut {
    float *rpart;
    size_t slots;
};

// Gather the runs [q0, q1) of one brick into this warp's 9^3 accumulator.  Each lane walks one run, one cell at a
// time.  Inside a cell the upper-corner weights along each axis are linear
// in the sample index k (u + v k), so each of the cell's 8 trilinear corner
// sums sum_k g_k w_x(k) w_y(k) w_z(k) is a fixed combination of the four
// moments sum_k g_k k^j (j = 0..3): the sample loop only accumulates the
// moments, and the corner sums are formed once per cell.  The warp then
// flushes the step's cell records together.  A lane whose run ends takes
// the next run in order, so every decision depends only on the data and
// the sums have a fixed order.  With POSE the lane also sums the run's
// pose-gradient terms from the same moments and the cell's corner values.
template <bool POSE>
__device__ __forceinline__ void gather_runs(const Run *__restrict__ runs, const RayStep *__restrict__ steps,
                                            const uint32_t *__restrict__ order,
                                            uint32_t q0, uint32_t q1, const float *__restrict__ gzbuf,
                                            const GatherArgs &G, GatherSmem<POSE> &sm, int w, const PoseOut &po)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    float *acc = sm.acc[w];
    const float *vox = sm.vox[POSE ? w : 0];
    long long X = 0, Y = 0, Z = 0, dX = 0, dY = 0, dZ = 0;
    const float *g = gzbuf;
    int left = 0;                 // samples left in the lane's run
    int cx = 0, cy = 0, cz = 0;   // samples left before each axis's next crossing
    int len = 0;                  // samples of the lane's current cell
    uint32_t slot = 0;            // the run's slot (pose output)
    int kc = 0;                   // index along the ray of the next sample
    float ps[6] = {};             // pose-gradient sums of the run
    uint2(*qr)[32] = sm.qr[w];
    float(*slope)[32] = sm.slope[w];
    uint32_t next = q0;           // next unassigned run (warp-uniform)
    // the first samples of the lane's next cell, loaded while the current
    // cell's corner sums and flush run (the cell's other samples are loaded
    // in its moment loop), and no others (each lane reads its own line, so a
    // load costs several L1 wavefronts: 49 M per 34 M samples with all eight
    // loaded, 42 M).
    constexpr int kPre = 8;
    float pre_g[kPre] = {};
    auto enter_cell = [&] {
        len = min(min(cx, cy), min(cz, min(left, kGCellCap)));
#pragma unroll
        for (int q = 0; q < kPre; q++) pre_g[q] = q < len ? __ldg(g + q) : 0.0f;
    };
    // lane i holds the index of run next + i, loaded one refill ahead
    uint32_t pre = next + lane < q1 ? order[next + lane] : 0u;
    for (;;) {
        // refill idle lanes in lane order
        const bool idle = left == 0;
        const unsigned idles = __ballot_sync(0xffffffffu, idle);
        if (idles && next < q1) {
            const int src = __popc(idles & lt);
            const uint32_t idx = __shfl_sync(0xffffffffu, pre, src);
            if (idle && next + src < q1) {
                const Run run = runs[idx];
                const RayStep &rs = steps[run.ray];
                X = run.X;
                Y = run.Y;
                Z = run.Z;
                dX = rs.d[0];
                dY = rs.d[1];
                dZ = rs.d[2];
#pragma unroll
                for (int q = 0; q < 3; q++) {
                    qr[q][lane] = rs.qr[q];
                    slope[q][lane] = rs.v[q];
                }
                g = gzbuf + rs.g_off + run.k0;
                left = run.len;
                cx = (int)(run.next & kNextMax);
                cy = (int)((run.next >> kNextBits) & kNextMax);
                cz = (int)(run.next >> (2 * kNextBits));
                enter_cell();
                if (POSE) {
                    slot = idx;
                    kc = run.k0;
#pragma unroll
                    for (int q = 0; q < 6; q++) ps[q] = 0.0f;
                }
            }
            next += __popc(idles);
            pre = next + lane < q1 ? order[next + lane] : 0u;
        }
        if (!__any_sync(0xffffffffu, left > 0)) break;
        const bool has = left > 0;
        // the lane's current cell
        int ix, iy, iz;
        float ux, vx, uy, vy, uz, vz;
        axis_cell(X, slope[0][lane], G.nx, ix, ux, vx);
        axis_cell(Y, slope[1][lane], G.ny, iy, uy, vy);
        axis_cell(Z, slope[2][lane], G.nz, iz, uz, vz);
        if (!has) len = 0;
        // moments of dL/dZ over the cell's samples
        float M0 = 0.0f, M1 = 0.0f, M2 = 0.0f, M3 = 0.0f;
        const int kmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
        auto moment = [&](float gk, int k) {
            const float kf = (float)k, k2 = kf * kf;
            M0 += gk;
            M1 = fmaf(gk, kf, M1);
            M2 = fmaf(gk, k2, M2);
            M3 = fmaf(gk, k2 * kf, M3);   // k < 32: the powers are exact
        };
#pragma unroll
        for (int k = 0; k < kPre; k++)
            if (k < len) moment(pre_g[k], k);
#pragma unroll 4
        for (int k = kPre; k < kmax; k++)
            if (k < len) moment(__ldg(g + k), k);
        // corner sums: yz products as quadratics in k, then the x factors
        float v[8];
        {
            const float ay[2] = {1.0f - uy, uy}, by[2] = {-vy, vy};
            const float az[2] = {1.0f - uz, uz}, bz[2] = {-vz, vz};
            const float ax0 = 1.0f - ux, bx0 = -vx;
#pragma unroll
            for (int zz = 0; zz < 2; zz++)
#pragma unroll
                for (int yy = 0; yy < 2; yy++) {
                    const float q0c = ay[yy] * az[zz];
                    const float q1c = fmaf(ay[yy], bz[zz], by[yy] * az[zz]);
                    const float q2c = by[yy] * bz[zz];
                    const float A = fmaf(q2c, M2, fmaf(q1c, M1, q0c * M0));
                    const float B = fmaf(q2c, M3, fmaf(q1c, M2, q0c * M1));
                    v[(zz << 2) | (yy << 1)] = fmaf(bx0, B, ax0 * A);
                    v[(zz << 2) | (yy << 1) | 1] = fmaf(vx, B, ux * A);
                }
        }
        // the cell's first voxel in the brick's arrays, from the low bits of
        // the cell, so that no cell index reaches past them
        const int base = ((iz & (kBrick - 1)) * kBrickV + (iy & (kBrick - 1))) * kBrickV + (ix & (kBrick - 1));
        if (POSE && has) {
            // the cell's 8 corner values, from the brick copy in shared memory
            float c[8];
#pragma unroll
            for (int q = 0; q < 8; q++) c[q] = vox[base + ((q >> 2) * kBrickV + ((q >> 1) & 1)) * kBrickV + (q & 1)];
            // per axis: sum_k g_k dZ/dx_a(k) = p0 M0 + p1 M1 + p2 M2 and the
            // k-weighted sum p0 M1 + p1 M2 + p2 M3, zero where the coordinate
            // is not strictly inside (0, n-1)
            float p[3][3];
            axis_poly(c[1] - c[0], c[3] - c[2], c[5] - c[4], c[7] - c[6], uy, vy, uz, vz, p[0][0], p[0][1], p[0][2]);
            axis_poly(c[2] - c[0], c[3] - c[1], c[6] - c[4], c[7] - c[5], ux, vx, uz, vz, p[1][0], p[1][1], p[1][2]);
            axis_poly(c[4] - c[0], c[5] - c[1], c[6] - c[2], c[7] - c[3], ux, vx, uy, vy, p[2][0], p[2][1], p[2][2]);
            const bool in[3] = {X > 0 && (int)(X >> 32) < G.nx - 1, Y > 0 && (int)(Y >> 32) < G.ny - 1,
                                Z > 0 && (int)(Z >> 32) < G.nz - 1};
            const float kh = (float)kc + 0.5f;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const float Ta = fmaf(p[a][2], M2, fmaf(p[a][1], M1, p[a][0] * M0));
                const float Wa = fmaf(p[a][2], M3, fmaf(p[a][1], M2, p[a][0] * M1));
                if (in[a]) {
                    ps[a] += Ta;
                    ps[3 + a] += fmaf(kh, Ta, Wa);
                }
            }
        }
        if (has) {
            X += (long long)len * dX;
            Y += (long long)len * dY;
            Z += (long long)len * dZ;
            g += len;
            left -= len;
            cx -= len;
            cy -= len;
            cz -= len;
            if (POSE) kc += len;
            if (left > 0) {
                // only an axis that crossed is counted again
                if (cx == 0) cx = next_steps(X, dX, G.nx, qr[0][lane]);
                if (cy == 0) cy = next_steps(Y, dY, G.ny, qr[1][lane]);
                if (cz == 0) cz = next_steps(Z, dZ, G.nz, qr[2][lane]);
                enter_cell();
            } else if (POSE) {
#pragma unroll
                for (int q = 0; q < 6; q++) po.rpart[(size_t)q * po.slots + slot] = ps[q];
            }
        }
        flush_records(has, base, v, acc, lane, lt);
    }
}

}  // namespace dfs
