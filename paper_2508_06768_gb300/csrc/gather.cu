// Volume-gradient gather: brick runs, stable radix sort, units, reduction.
// See gather.cuh for the algorithm.
#include "gather.cuh"
#include "host.hpp"

namespace dfs {

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;                 // items per thread per tile
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kScanChunk = 4096;

// ------------------------------------------------------------------ runs

// The run's 40 bytes in use.
__device__ __forceinline__ void store_run(Run *dst, const Run &r)
{
    longlong2 *p = reinterpret_cast<longlong2 *>(dst);
    p[0] = make_longlong2(r.X, r.Y);
    p[1] = make_longlong2(r.Z, (long long)(unsigned)r.ray | ((long long)r.k0 << 32));
    reinterpret_cast<uint2 *>(dst)[4] = make_uint2((uint32_t)r.len, r.next);
}

__device__ __forceinline__ void store_steps(RayStep *dst, const long long d[3], long long g_off)
{
    RayStep s;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        s.d[a] = d[a];
        s.qr[a] = cell_steps(d[a]);
        s.v[a] = slope_of(d[a]);
        s.pad[a] = 0.0f;
    }
    s.g_off = g_off;
    *dst = s;
}

// One thread per ray: many rays, or rays of more than kRunMax brick changes.
// 72 registers hold 24 warps per SM, which takes 147 K rays in about one wave
// (512 frames: 195 us at 90 registers, 168 us).
__global__ void __launch_bounds__(128, 6) k_ray_runs(const RayGeo *__restrict__ geo, const long long *__restrict__ gz_off, int n_rays,
                           GatherArgs G, int cap, Run *__restrict__ runs, RayStep *__restrict__ steps,
                           uint32_t *__restrict__ keys, int *__restrict__ nrun, uint32_t *__restrict__ bcount,
                           unsigned long long *__restrict__ brick_work, uint32_t *__restrict__ status)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rays) return;
    const RayGeo rg = geo[r];
    const long long S = rg.S;
    const int n[3] = {G.nx, G.ny, G.nz};
    int b[3];
    long long nxt[3];
    for (int a = 0; a < 3; a++) {
        b[a] = cell_of(rg.X0[a], n[a]) / kBrick;
        nxt[a] = next_change(rg.X0[a], rg.DX[a], b[a], n[a], S);
    }
    const FirstSteps fs = first_steps_of(rg.DX);
    long long k = 0;
    int cnt = 0;
    // slot of run i of ray r: i * n_rays + r (consecutive rays write consecutive slots)
    while (k <= S) {
        long long kn = nxt[0];
        kn = nxt[1] < kn ? nxt[1] : kn;
        kn = nxt[2] < kn ? nxt[2] : kn;
        long long k1 = kn - 1 < S ? kn - 1 : S;
        if (cnt < cap) {
            const uint32_t brick = (uint32_t)((b[2] * G.nby + b[1]) * G.nbx + b[0]);
            Run run;
            run.X = rg.X0[0] + k * rg.DX[0];
            run.Y = rg.X0[1] + k * rg.DX[1];
            run.Z = rg.X0[2] + k * rg.DX[2];
            run.ray = r;
            run.len = (int)(k1 - k + 1);
            run.k0 = (int)k;
            run.next = first_steps(run.X, run.Y, run.Z, rg.DX, fs, G.nx, G.ny, G.nz);
            const size_t slot = (size_t)cnt * n_rays + r;
            store_run(runs + slot, run);
            keys[slot] = brick;
            {   // lanes on the same brick add once, through their lowest lane
                // (integer sums, so the order does not matter)
                const unsigned act = __activemask();
                const unsigned grp = __match_any_sync(act, brick);
                unsigned long long sum = 0;
                for (unsigned m = grp; m; m &= m - 1)
                    sum += (unsigned long long)__shfl_sync(grp, run.len, __ffs(m) - 1);
                if ((int)(threadIdx.x & 31) == __ffs(grp) - 1) {
                    atomicAdd(brick_work + brick, sum);
                    atomicAdd(bcount + brick, (uint32_t)__popc(grp));
                }
            }
            cnt++;
        } else if (status) {
            atomicOr(status + 2, (uint32_t)DIFFUS_STATUS_QUEUE);
        }
        k = kn;
        if (k > S) break;
        for (int a = 0; a < 3; a++) {
            if (nxt[a] == kn) {
                long long X = rg.X0[a] + k * rg.DX[a];
                b[a] = cell_of(X, n[a]) / kBrick;
                nxt[a] = next_change(rg.X0[a], rg.DX[a], b[a], n[a], S);
                if (nxt[a] <= k) nxt[a] = k + 1;   // guard: never stall
            }
        }
    }
    nrun[r] = cnt;
    store_steps(steps + r, rg.DX, gz_off[r]);
}

// The same runs with one warp per ray, for rays of at most kRunMax brick
// changes.  The brick index of an axis is monotone along the ray, so its
// changes can be found independently: lanes solve one crossing each, the three
// axes' ordered lists are merged by rank, and equal crossings (a sample that
// enters a new brick on two axes) become one.  One thread per ray walks up to
// 80 dependent steps of 64-bit arithmetic, which is latency-bound for a frame
// of a few hundred rays: 48 us for 251, 5.4 us here.  With many rays the walk
// is hidden and its aggregated counter updates win: 147 K rays 168 us, 227 us
// here; the two lines cross near kRunWarpRays rays.
//
// bcount receives the runs of each brick.  ARRIVE keeps each run's arrival
// number in its brick (any order; ranked by slot afterwards), else brick_work
// receives the samples of each brick for the unit order.
constexpr int kRunWarps = 8;
constexpr int kRunWarpRays = 50000;

template <bool ARRIVE>
__global__ void __launch_bounds__(kRunWarps * 32)
    k_ray_runs_warp(const RayGeo *__restrict__ geo, const long long *__restrict__ gz_off, int n_rays, GatherArgs G,
                    int cap, Run *__restrict__ runs, RayStep *__restrict__ steps, uint32_t *__restrict__ keys,
                    int *__restrict__ nrun, uint32_t *__restrict__ bcount, uint32_t *__restrict__ arrival,
                    unsigned long long *__restrict__ brick_work, uint32_t *__restrict__ status)
{
    __shared__ int sk[kRunWarps][kRunMax + 1], sm[kRunWarps][kRunMax + 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int r = blockIdx.x * kRunWarps + w;
    if (r >= n_rays) return;
    const RayGeo rg = geo[r];
    const int S = rg.S;
    const int n[3] = {G.nx, G.ny, G.nz};
    const Cuts c = ray_cuts(rg.X0, rg.DX, S, n);
    const int m = c.off[3];                     // <= kRunMax
    int *k = sk[w], *start = sm[w];
    for (int e = lane; e < m; e += 32) k[e] = cut_sample(c, e, rg.X0, rg.DX, S);
    __syncwarp();
    int *order = start;                         // merged, with repeats
    for (int e = lane; e < m; e += 32) order[cut_rank(c, k, m, e)] = k[e];
    __syncwarp();
    // distinct crossings: the first sample of every run after the first
    int cnt = c.fits ? 1 : 0;
    for (int e0 = 0; e0 < m; e0 += 32) {
        const int e = e0 + lane;
        const int v = e < m ? order[e] : 0;
        const bool first = e < m && (e == 0 || order[e - 1] != v);
        const unsigned bal = __ballot_sync(0xffffffffu, first);
        if (first) k[cnt - 1 + __popc(bal & ((1u << lane) - 1u))] = v;   // k[i]: start of run i + 1
        cnt += __popc(bal);
    }
    __syncwarp();
    // as in k_ray_runs, samples beyond the last slot are dropped and reported
    const int kept = min(cnt, cap);
    if ((kept < cnt || !c.fits) && status && lane == 0) atomicOr(status + 2, (uint32_t)DIFFUS_STATUS_QUEUE);
    const FirstSteps fs = first_steps_of(rg.DX);
    for (int i = lane; i < kept; i += 32) {
        int ka, kb;
        run_span(k, i, cnt, S, ka, kb);
        Run run;
        run.X = rg.X0[0] + (long long)ka * rg.DX[0];
        run.Y = rg.X0[1] + (long long)ka * rg.DX[1];
        run.Z = rg.X0[2] + (long long)ka * rg.DX[2];
        run.ray = r;
        run.len = kb - ka;
        run.k0 = ka;
        run.next = first_steps(run.X, run.Y, run.Z, rg.DX, fs, G.nx, G.ny, G.nz);
        const uint32_t brick = (uint32_t)(((cell_of(run.Z, n[2]) / kBrick) * G.nby + cell_of(run.Y, n[1]) / kBrick) * G.nbx +
                                          cell_of(run.X, n[0]) / kBrick);
        const size_t slot = (size_t)i * n_rays + r;
        store_run(runs + slot, run);
        keys[slot] = brick;
        if (ARRIVE) {
            arrival[slot] = atomicAdd(bcount + brick, 1u);
        } else {
            atomicAdd(bcount + brick, 1u);
            atomicAdd(brick_work + brick, (unsigned long long)run.len);
        }
    }
    if (lane == 0) {
        nrun[r] = kept;
        store_steps(steps + r, rg.DX, gz_off[r]);
    }
}

// ------------------------------------------------------------ exclusive scan

__global__ void k_chunk_sums(const uint32_t *__restrict__ in, size_t n, uint32_t *__restrict__ sums)
{
    __shared__ uint32_t red[32];
    const size_t b0 = (size_t)blockIdx.x * kScanChunk;
    uint32_t s = 0;
    for (int i = threadIdx.x; i < kScanChunk; i += blockDim.x)
        if (b0 + i < n) s += in[b0 + i];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0;
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (threadIdx.x == 0) sums[blockIdx.x] = v;
    }
}

// single block: exclusive scan of m values in place, total to *total
__global__ void k_scan_sums(uint32_t *__restrict__ sums, int m, uint32_t *__restrict__ total)
{
    __shared__ uint32_t buf[1024];
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < m; base += 1024) {
        int i = base + threadIdx.x;
        uint32_t v = i < m ? sums[i] : 0;
        buf[threadIdx.x] = v;
        __syncthreads();
        for (int off = 1; off < 1024; off <<= 1) {
            uint32_t t = threadIdx.x >= off ? buf[threadIdx.x - off] : 0;
            __syncthreads();
            buf[threadIdx.x] += t;
            __syncthreads();
        }
        uint32_t incl = buf[threadIdx.x];
        if (i < m) sums[i] = carry + incl - v;
        __syncthreads();
        if (threadIdx.x == 1023) carry += incl;
        __syncthreads();
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void k_chunk_scan(const uint32_t *__restrict__ in, size_t n, const uint32_t *__restrict__ sums,
                             uint32_t *__restrict__ out)
{
    __shared__ uint32_t buf[1024];
    __shared__ uint32_t carry;
    const size_t b0 = (size_t)blockIdx.x * kScanChunk;
    if (threadIdx.x == 0) carry = sums[blockIdx.x];
    __syncthreads();
    for (int base = 0; base < kScanChunk; base += 1024) {
        size_t i = b0 + base + threadIdx.x;
        uint32_t v = i < n ? in[i] : 0;
        buf[threadIdx.x] = v;
        __syncthreads();
        for (int off = 1; off < 1024; off <<= 1) {
            uint32_t t = threadIdx.x >= off ? buf[threadIdx.x - off] : 0;
            __syncthreads();
            buf[threadIdx.x] += t;
            __syncthreads();
        }
        uint32_t incl = buf[threadIdx.x];
        if (i < n) out[i] = carry + incl - v;
        __syncthreads();
        if (threadIdx.x == 1023) carry += incl;
        __syncthreads();
    }
}

// ------------------------------------------------------- stable radix sort

// The first pass reads the slots (n = all of them; kNoRun marks a slot without
// a run) and drops the empty ones, about three in four; the later passes run
// over the *n_used runs that are left (512 frames: histograms 30 + 28 us and
// scatters 68 + 67 us with every slot in both passes, 14 + 9.5 and 44 + 29 us).
constexpr uint32_t kNoRun = 0xffffffffu;

template <bool FIRST>
__global__ void __launch_bounds__(kSortThreads) k_digit_hist(const uint32_t *__restrict__ keys, size_t slots,
                                                             const uint32_t *__restrict__ n_used, int shift, int nblk,
                                                             uint32_t *__restrict__ hist)
{
    __shared__ uint32_t cnt[256];
    const size_t n = FIRST ? slots : (size_t)*n_used;
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const size_t b0 = (size_t)blockIdx.x * kSortTile;
    if (b0 < n) {
        uint32_t key[kSortItems];
#pragma unroll
        for (int s = 0; s < kSortItems; s++) {
            const size_t i = b0 + (size_t)s * kSortThreads + threadIdx.x;
            key[s] = i < n ? keys[i] : kNoRun;
        }
#pragma unroll
        for (int s = 0; s < kSortItems; s++) {
            // neighbouring slots are the same run of neighbouring rays and
            // mostly lie in one brick: one shared add per distinct digit
            const uint32_t d = key[s] != kNoRun ? ((key[s] >> shift) & 255u) : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            if (d < 256u && (peers & ((1u << (threadIdx.x & 31)) - 1u)) == 0)
                atomicAdd(&cnt[d], (uint32_t)__popc(peers));   // integer counts: order-free
        }
    }
    __syncthreads();
    hist[(size_t)threadIdx.x * nblk + blockIdx.x] = cnt[threadIdx.x];
}

// Stable scatter: an item's position is its digit's offset for this tile,
// plus the items of the same digit earlier in the tile (earlier sub-tiles,
// earlier warps, lower lanes).  FIRST: the values are the slot numbers.
template <bool FIRST>
__global__ void __launch_bounds__(kSortThreads) k_digit_scatter(const uint32_t *__restrict__ kin,
                                                                const uint32_t *__restrict__ vin, size_t slots,
                                                                const uint32_t *__restrict__ n_used, int shift,
                                                                int nblk, const uint32_t *__restrict__ offs,
                                                                uint32_t *__restrict__ kout,
                                                                uint32_t *__restrict__ vout)
{
    constexpr int W = kSortThreads / 32;
    __shared__ uint32_t run[256];
    __shared__ uint32_t wcnt[W][257];
    const size_t n = FIRST ? slots : (size_t)*n_used;
    const size_t b0 = (size_t)blockIdx.x * kSortTile;
    if (b0 >= n) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    run[threadIdx.x] = offs[(size_t)threadIdx.x * nblk + blockIdx.x];
    for (int q = 0; q < W; q++) wcnt[q][threadIdx.x] = 0;
    if (threadIdx.x == 0)
        for (int q = 0; q < W; q++) wcnt[q][256] = 0;
    __syncthreads();
    for (int s = 0; s < kSortItems; s++) {
        const size_t i = b0 + (size_t)s * kSortThreads + threadIdx.x;
        const uint32_t key = i < n ? kin[i] : kNoRun;
        const bool valid = key != kNoRun;
        if (FIRST && !__syncthreads_or(valid)) continue;   // a stretch of empty slots
        const uint32_t val = FIRST ? (uint32_t)i : (valid ? vin[i] : 0u);
        const uint32_t d = valid ? ((key >> shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int wrank = __popc(peers & ((1u << lane) - 1u));
        if (wrank == 0) wcnt[w][d] = __popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t pos = run[d] + (uint32_t)wrank;
            for (int q = 0; q < w; q++) pos += wcnt[q][d];
            kout[pos] = key;
            vout[pos] = val;
        }
        __syncthreads();
        uint32_t add = 0;
        for (int q = 0; q < W; q++) {
            add += wcnt[q][threadIdx.x];
            wcnt[q][threadIdx.x] = 0;
        }
        run[threadIdx.x] += add;
        if (threadIdx.x == 0)
            for (int q = 0; q < W; q++) wcnt[q][256] = 0;
        __syncthreads();
    }
}

// --------------------------------------------------------------- units

// Per brick, from its run count: its runs [bstart, bend) in sorted order and
// its units ustart .. ustart + ucount - 1 (with the unit -> brick table).  A
// block owns 1024 bricks and adds up the counts before its own by itself, so
// the two prefix sums take one launch and no block waits for another; beyond
// kPlanDirect bricks (a quarter of a MB of counts from L2 per block) it adds up
// per-block sums that k_brick_sums wrote first.
constexpr int kPlanThreads = 1024;
constexpr int kPlanDirect = 65536;

__device__ __forceinline__ unsigned long long block_sum2(unsigned long long v, unsigned long long *red)
{
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long t = red[threadIdx.x & 31];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    __syncthreads();
    return t;
}

// Runs (high word) and units (low word) of a brick with c runs; unit is a
// power of two.
__device__ __forceinline__ unsigned long long runs_units(uint32_t c, int unit)
{
    return ((unsigned long long)c << 32) | ((c + (uint32_t)unit - 1) >> (31 - __clz(unit)));
}

__global__ void __launch_bounds__(kPlanThreads)
    k_brick_sums(const uint32_t *__restrict__ bcount, int nb, int unit, unsigned long long *__restrict__ sums)
{
    __shared__ unsigned long long red[32];
    const int b = blockIdx.x * kPlanThreads + threadIdx.x;
    const unsigned long long t = block_sum2(runs_units(b < nb ? bcount[b] : 0u, unit), red);
    if (threadIdx.x == 0) sums[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kPlanThreads)
    k_brick_plan(const uint32_t *__restrict__ bcount, const unsigned long long *__restrict__ sums, int nb, int unit,
                 uint32_t *__restrict__ bstart, uint32_t *__restrict__ bend, uint32_t *__restrict__ ucount,
                 uint32_t *__restrict__ ustart, uint32_t *__restrict__ unit_brick, uint32_t *__restrict__ n_units,
                 uint32_t *__restrict__ n_runs)
{
    __shared__ unsigned long long red[32], wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b0 = blockIdx.x * kPlanThreads, b = b0 + threadIdx.x;
    unsigned long long before = 0;
    if (sums) {
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += kPlanThreads) before += sums[i];
    } else {
        for (int i = threadIdx.x * 4; i < b0; i += kPlanThreads * 4) {
            const uint4 c = *reinterpret_cast<const uint4 *>(bcount + i);
            before += (runs_units(c.x, unit) + runs_units(c.y, unit)) + (runs_units(c.z, unit) + runs_units(c.w, unit));
        }
    }
    before = block_sum2(before, red);
    const uint32_t c = b < nb ? bcount[b] : 0u;
    const unsigned long long v = runs_units(c, unit);
    unsigned long long x = v;
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    unsigned long long base = before;
    for (int q = 0; q < w; q++) base += wsum[q];
    const unsigned long long ex = base + x - v;
    if (b < nb) {
        const uint32_t r0 = (uint32_t)(ex >> 32), u0 = (uint32_t)ex, nu = (uint32_t)v;
        bstart[b] = r0;
        bend[b] = r0 + c;
        ustart[b] = u0;
        ucount[b] = nu;
        for (uint32_t i = 0; i < nu; i++) unit_brick[u0 + i] = (uint32_t)b;
    }
    if (b == nb - 1) {
        *n_units = (uint32_t)(ex + v);
        *n_runs = (uint32_t)((ex + v) >> 32);
    }
}

// Small problems (a frame, a few frames) are sorted by place and rank instead
// of the radix passes: every run goes to its arrival place in its brick's
// range, then each counts the runs of its brick with a smaller slot.  The
// result is the same order (by brick, then slot); the work is the sum of the
// squared brick counts.  Two launches of 3 to 7 us for a frame, where two radix
// passes of five launches took 50 us.  Grid y: run number along the ray.
__global__ void k_place_runs(const uint32_t *__restrict__ keys, const uint32_t *__restrict__ arrival,
                             const int *__restrict__ nrun, int n_rays, const uint32_t *__restrict__ bstart,
                             uint2 *__restrict__ list)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rays || (int)blockIdx.y >= nrun[r]) return;
    const uint32_t slot = blockIdx.y * (uint32_t)n_rays + (uint32_t)r;
    const uint32_t b = keys[slot];
    list[bstart[b] + arrival[slot]] = make_uint2(slot, b);
}

__global__ void k_rank_runs(const uint2 *__restrict__ list, const uint32_t *__restrict__ n_runs,
                            const uint32_t *__restrict__ bstart, const uint32_t *__restrict__ bend,
                            uint32_t *__restrict__ sorted)
{
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= *n_runs) return;
    const uint2 me = list[p];
    const uint32_t q0 = bstart[me.y], q1 = bend[me.y];
    uint32_t rank = 0;
#pragma unroll 8
    for (uint32_t q = q0; q < q1; q++) rank += list[q].x < me.x;
    sorted[q0 + rank] = me.x;
}

// Work class of each unit, one thread per unit: its share of its brick's
// samples (a unit of m of the brick's n runs gets m/n of them), binned as
// class = 31 - floor(log2(samples)), largest first; with a histogram of
// the classes.
__global__ void k_unit_work(const unsigned long long *__restrict__ brick_work, const uint32_t *__restrict__ bstart,
                            const uint32_t *__restrict__ bend, const uint32_t *__restrict__ ustart,
                            const uint32_t *__restrict__ unit_brick, const uint32_t *__restrict__ n_units,
                            int unit, uint32_t *__restrict__ uclass, uint32_t *__restrict__ class_count)
{
    const uint32_t total = *n_units;
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x) {
        const int b = (int)unit_brick[u];
        const uint32_t n = bend[b] - bstart[b];
        const uint32_t r0 = (u - ustart[b]) * (uint32_t)unit;
        const uint32_t m = min((uint32_t)unit, n - r0);
        const unsigned long long w = brick_work[b] * m / n;
        const uint32_t c = (uint32_t)__clzll(w | 1ull) - 32u;   // 31 - floor(log2(w)) for w < 2^32
        const uint32_t cc = c > 31u ? 0u : c;                    // w >= 2^32 (not reached): largest class
        uclass[u] = cc;
        atomicAdd(class_count + cc, 1u);   // integer counts: order-free
    }
}

// Exclusive scan of the 32 class counts into cursors (one warp).
__global__ void k_class_cursors(uint32_t *__restrict__ class_count)
{
    const int lane = threadIdx.x;
    const uint32_t c = class_count[lane];
    uint32_t x = c;
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    class_count[lane] = x - c;
}

// The units in order of their work class, largest first.  The order inside
// a class is whatever the atomics give: it decides only which warp takes a
// unit when, never a result (every unit writes its own partial).
__global__ void k_unit_order(const uint32_t *__restrict__ uclass, const uint32_t *__restrict__ n_units,
                             uint32_t *__restrict__ cursor, uint32_t *__restrict__ order)
{
    const uint32_t total = *n_units;
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < total; u += gridDim.x * blockDim.x)
        order[atomicAdd(cursor + uclass[u], 1u)] = u;
}

// Resident blocks per SM of the unit kernel: 6 at 80 registers, where the form
// with pose terms keeps 12 bytes on the stack.  Measured on the 512-pose batch:
// 5 (96 registers) 1056 us, 6 986, 7 (72 registers, spills in the cell loop) 1270.
constexpr int kGatherCtas = 6;

// One warp per unit, units handed out by a ticket queue: the warp gathers
// the unit's runs into its own 9^3 accumulator and writes the unit's
// partial (with POSE, also each run's pose-gradient sums).  Warps are
// independent, so a CTA has no block barriers.
template <typename T, bool POSE>
__global__ void __launch_bounds__(kGatherWarps * 32, kGatherCtas)
    k_gather_units(const float *__restrict__ gz, const Run *__restrict__ runs, const RayStep *__restrict__ steps,
                   const uint32_t *__restrict__ sorted_vals,
                   const uint32_t *__restrict__ bstart, const uint32_t *__restrict__ bend,
                   const uint32_t *__restrict__ ustart, const uint32_t *__restrict__ unit_brick,
                   const uint32_t *__restrict__ n_units, GatherArgs G, int unit, float *__restrict__ upart,
                   uint32_t *__restrict__ queue, const uint32_t *__restrict__ order, const T *__restrict__ vol,
                   PoseOut po)
{
    __shared__ GatherSmem<POSE> sm;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t total = *n_units;
    float *acc = sm.acc[w];
    for (;;) {
        uint32_t u = 0;
        if (lane == 0) u = atomicAdd(queue, 1u);
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= total) break;
        if (order) u = order[u];   // longest-first
        const int b = (int)unit_brick[u];
        const uint32_t part = u - ustart[b];
        const uint32_t r0 = bstart[b] + part * (uint32_t)unit;
        uint32_t r1 = r0 + (uint32_t)unit;
        r1 = r1 < bend[b] ? r1 : bend[b];
        for (int i = lane; i < kBrickVox; i += 32) acc[i] = 0.0f;
        if (POSE) {
            const int bx0 = (b % G.nbx) * kBrick, by0 = ((b / G.nbx) % G.nby) * kBrick, bz0 = (b / (G.nbx * G.nby)) * kBrick;
            // the 9^3 voxels the brick's cells touch (clamped at the far faces,
            // where no cell of the brick reaches)
            const unsigned sy = (unsigned)G.nx, sz = (unsigned)G.nx * (unsigned)G.ny;
#pragma unroll 8
            for (int i = lane; i < kBrickVox; i += 32) {   // eight loads in flight per lane
                const int lx = i % kBrickV, ly = (i / kBrickV) % kBrickV, lz = i / (kBrickV * kBrickV);
                const unsigned x = (unsigned)min(bx0 + lx, G.nx - 1), y = (unsigned)min(by0 + ly, G.ny - 1),
                               z = (unsigned)min(bz0 + lz, G.nz - 1);
                sm.vox[w][i] = ldv(vol, z * sz + y * sy + x);
            }
        }
        __syncwarp();
        gather_runs<POSE>(runs, steps, sorted_vals, r0, r1, gz, G, sm, w, po);
        __syncwarp();
        float *out = upart + (size_t)u * kBrickVox;
        for (int i = lane; i < kBrickVox; i += 32) out[i] = acc[i];
        __syncwarp();
    }
}

// The bricks whose cells touch voxel v along one axis, with v's index
// inside each brick's 9 voxels: first the brick of cell v-1 when v is on its
// far face (or v is the last voxel), then the brick of cell v.  Returns how
// many (1 or 2); the entries are (b0, l0) and (b1, l1), scalars so that
// they stay in registers.
struct AxisBricks {
    int n, b0, l0, b1, l1;
};

__device__ __forceinline__ AxisBricks voxel_bricks(int v, int n)
{
    const int own = v >> 3;                  // brick of cell v (when v <= n-2)
    const int low = (v - 1) >> 3;            // brick of cell v-1 (when v >= 1)
    const bool has_own = v <= n - 2;
    const bool has_low = v >= 1 && !(has_own && low == own);
    AxisBricks a;
    a.n = (int)has_low + (int)has_own;
    a.b0 = has_low ? low : own;
    a.l0 = v - a.b0 * kBrick;
    a.b1 = own;
    a.l1 = v - own * kBrick;
    return a;
}

// Each voxel: sum over the bricks whose cells touch it (z outer, then y,
// then x; on each axis the lower brick first), units in order.  A thread owns
// kRedVox consecutive voxels of one brick along x (voxel 0 of a brick also
// belongs to the brick below), so the brick tables are read once for all of
// them and a row away from every ray (most of a volume around one frame) is
// one 16-byte store: bound by the volume's write there, by the partials' reads
// where many frames meet.  A 251-ray frame in 256 x 256 x 192: one voxel per
// thread 54 us, four 28, and 256-thread blocks over several rows 15.7 us; 512
// frames in 256^3: 97 us, now 43.
// Blocks cover blockDim.x * 4 voxels of blockDim.y rows of one slice.
constexpr int kRedVox = 4;

__global__ void k_voxel_reduce(const float *__restrict__ upart, const uint32_t *__restrict__ ustart,
                               const uint32_t *__restrict__ ucount, GatherArgs G, float *__restrict__ grad_vol, bool vec)
{
    const int vx = (blockIdx.x * blockDim.x + threadIdx.x) * kRedVox;
    const int vy = blockIdx.y * blockDim.y + threadIdx.y, vz = blockIdx.z;
    if (vx >= G.nx || vy >= G.ny) return;
    const AxisBricks ay = voxel_bricks(vy, G.ny), az = voxel_bricks(vz, G.nz);
    const int own = vx >> 3, l = vx & 7;
    const bool has_own = own * kBrick <= G.nx - 2;   // the brick has cells (else vx is its only voxel)
    const bool has_low = vx >= 1 && l == 0;  // voxel vx is the far face of the brick below
    float s[kRedVox] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int iz = 0; iz < 2; iz++) {
        if (iz >= az.n) break;
        const int bz = iz ? az.b1 : az.b0, lz = iz ? az.l1 : az.l0;
#pragma unroll
        for (int iy = 0; iy < 2; iy++) {
            if (iy >= ay.n) break;
            const int by = iy ? ay.b1 : ay.b0, ly = iy ? ay.l1 : ay.l0;
            const int row = (bz * G.nby + by) * G.nbx, li = (lz * kBrickV + ly) * kBrickV;
            if (has_low) {
                const int b = row + own - 1;
                const uint32_t u0 = ustart[b], n = ucount[b];
                const float *p = upart + (size_t)u0 * kBrickVox + li + kBrick;
                for (uint32_t u = 0; u < n; u++, p += kBrickVox) s[0] += *p;
            }
            if (has_own) {
                const int b = row + own;
                const uint32_t u0 = ustart[b], n = ucount[b];
                const float *p = upart + (size_t)u0 * kBrickVox + li + l;
#pragma unroll 4
                for (uint32_t u = 0; u < n; u++, p += kBrickVox) {
#pragma unroll
                    for (int q = 0; q < kRedVox; q++) s[q] += p[q];   // l + q <= 7: inside the brick's 9
                }
            }
        }
    }
    float *out = grad_vol + ((size_t)vz * G.ny + vy) * G.nx + vx;
    if (vec) {
        *reinterpret_cast<float4 *>(out) = make_float4(s[0], s[1], s[2], s[3]);
    } else {
#pragma unroll
        for (int q = 0; q < kRedVox; q++)
            if (vx + q < G.nx) out[q] = s[q];
    }
}

// Pose-gradient terms of each ray from its runs' sums, added in slot order
// (run order along the ray) in compensated FP32 (Knuth's two-sum; FP64
// arithmetic is slow on this part): the translation part sum_k dL/dZ_k
// grad Z(p_k) (per mm) and the rotation part sum_k dL/dZ_k s_k grad Z(p_k)
// projected on the ray's direction derivatives, s_k = (k + 1/2) ds.  A block
// takes 32 rays, one warp per component, so a ray's chain of loads is one
// component's, eight in flight (251 rays: 18 us with one thread per ray for all
// six, 7 us; 147 K rays: 48 us, 36 us).
__global__ void __launch_bounds__(192) k_ray_pose(const float *__restrict__ rpart, size_t slots,
                                                  const int *__restrict__ nrun, const RayGeo *__restrict__ geo,
                                                  int n_rays, float isx, float isy, float isz,
                                                  double *__restrict__ pose_part)
{
    __shared__ double sum6[6][32];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int r = blockIdx.x * 32 + lane;
    const int cnt = r < n_rays ? nrun[r] : 0;
    const float *p = rpart + (size_t)q * slots + r;
    float sum = 0.0f, err = 0.0f;
    constexpr int kB = 8;
    for (int i0 = 0; i0 < cnt; i0 += kB) {
        float x[kB];
#pragma unroll
        for (int b = 0; b < kB; b++) x[b] = i0 + b < cnt ? p[(size_t)(i0 + b) * n_rays] : 0.0f;
#pragma unroll
        for (int b = 0; b < kB; b++) {
            const float t = __fadd_rn(sum, x[b]);
            const float z = __fsub_rn(t, sum);
            const float e = __fadd_rn(__fsub_rn(sum, __fsub_rn(t, z)), __fsub_rn(x[b], z));
            err = __fadd_rn(err, e);
            sum = t;
        }
    }
    sum6[q][lane] = (double)sum + (double)err;
    __syncthreads();
    if (r >= n_rays || q >= 3) return;
    // warp a: translation component a and rotation component a
    const int a = q;
    const double is[3] = {(double)isx, (double)isy, (double)isz};
    const RayGeo &rg = geo[r];
    const double ds = (double)rg.ds;
    double *out = pose_part + 6 * (size_t)r;
    out[a] = __dmul_rn(sum6[a][lane], is[a]);
    double u[3];
#pragma unroll
    for (int i = 0; i < 3; i++) u[i] = __dmul_rn(sum6[3 + i][lane], __dmul_rn(is[i], ds));
    out[3 + a] = __fma_rn(u[2], (double)rg.v[a][2], __fma_rn(u[1], (double)rg.v[a][1], __dmul_rn(u[0], (double)rg.v[a][0])));
}

int sort_bits(int nb)
{
    int bits = 1;
    while ((1u << bits) < (uint32_t)nb) bits++;
    return bits;
}

// Place and rank instead of the radix passes: up to 32 K slots (12 launches and
// about 50 us less for a frame; ranking grows with the runs per brick), unless
// a few bricks hold so many runs that ranking is dearer.
bool sort_by_rank(size_t slots, size_t nb) { return slots <= 32768 && slots * slots <= nb << 26; }

}  // namespace

GatherArgs make_gather_args(const diffus_volume_desc *vd)
{
    GatherArgs G;
    G.nx = vd->nx; G.ny = vd->ny; G.nz = vd->nz;
    G.nbx = (vd->nx - 2) / kBrick + 1;
    G.nby = (vd->ny - 2) / kBrick + 1;
    G.nbz = (vd->nz - 2) / kBrick + 1;
    return G;
}

// Upper bound on the brick runs of one ray: the brick index is monotone on
// every axis and moves at most ceil(S ds / (8 s_a)) + 1 bricks on axis a.
int runs_per_ray(const diffus_volume_desc *vd, double max_path_mm)
{
    GatherArgs G = make_gather_args(vd);
    int nb[3] = {G.nbx, G.nby, G.nbz};
    double sp[3] = {vd->sx, vd->sy, vd->sz};
    int cap = 1;
    for (int a = 0; a < 3; a++) {
        double m = ceil(max_path_mm / (kBrick * sp[a])) + 1.0;
        cap += (int)fmin((double)(nb[a] - 1), m);
    }
    return cap;
}

struct GatherLayout {
    Run *runs;
    RayStep *steps;
    uint32_t *keys[2], *vals[2];    // radix passes; by rank: keys[1] arrivals, vals[0..1] the placed list
    uint32_t *hist, *sums, *misc;   // misc: [0] units total, [1] runs in use
    uint32_t *bstart, *bend, *ucount, *ustart, *unit_brick;
    uint32_t *uclass, *uorder;             // unit work classes, the longest-first order
    // zeroed by one memset: 64 counters (0..31 unit classes, 32 unit queue),
    // runs of each brick, samples of each brick's runs
    uint32_t *zero, *bcount;
    unsigned long long *bwork, *bsums;
    float *upart;
    float *rpart;   // per-run pose-gradient sums, 6 x slots
    int *nrun;      // runs of each ray
    size_t bytes;
};

static GatherLayout gather_layout(void *ws, const diffus_volume_desc *vd, long long n_rays, int cap)
{
    Carve c(ws);
    GatherLayout L;
    GatherArgs G = make_gather_args(vd);
    size_t nb = (size_t)G.nbx * G.nby * G.nbz;
    size_t slots = (size_t)n_rays * cap;
    size_t nblk = (slots + kSortTile - 1) / kSortTile;
    size_t nhist = 256 * nblk;
    size_t nsums = (nhist + kScanChunk - 1) / kScanChunk;
    size_t max_units = slots / unit_runs(slots) + nb;
    L.runs = c.take<Run>(slots);
    L.steps = c.take<RayStep>((size_t)n_rays);
    L.keys[0] = c.take<uint32_t>(slots);
    L.keys[1] = c.take<uint32_t>(slots);
    L.vals[0] = c.take<uint32_t>(2 * slots);
    L.vals[1] = L.vals[0] ? L.vals[0] + slots : nullptr;
    L.hist = c.take<uint32_t>(nhist);
    L.sums = c.take<uint32_t>(nsums + 1);
    L.misc = c.take<uint32_t>(4);
    L.bstart = c.take<uint32_t>(nb);
    L.bend = c.take<uint32_t>(nb);
    L.ucount = c.take<uint32_t>(nb);
    L.ustart = c.take<uint32_t>(nb);
    L.unit_brick = c.take<uint32_t>(max_units);
    L.uclass = c.take<uint32_t>(max_units);
    L.uorder = c.take<uint32_t>(max_units);
    L.zero = c.take<uint32_t>(64);
    L.bcount = c.take<uint32_t>(nb);
    L.bwork = c.take<unsigned long long>(nb);
    L.bsums = c.take<unsigned long long>((nb + kPlanThreads - 1) / kPlanThreads);
    L.upart = c.take<float>(max_units * kBrickVox);
    L.rpart = c.take<float>(6 * slots);
    L.nrun = c.take<int>((size_t)n_rays);
    L.bytes = c.used;
    return L;
}

size_t gather_workspace_bytes(const diffus_volume_desc *vd, long long n_rays, double max_path_mm)
{
    return gather_layout(nullptr, vd, n_rays, runs_per_ray(vd, max_path_mm)).bytes;
}

static void launch_scan(const uint32_t *in, uint32_t *out, size_t n, uint32_t *sums, uint32_t *total, cudaStream_t s)
{
    int nch = (int)((n + kScanChunk - 1) / kScanChunk);
    k_chunk_sums<<<nch, 256, 0, s>>>(in, n, sums);
    k_scan_sums<<<1, 1024, 0, s>>>(sums, nch, total);
    k_chunk_scan<<<nch, 1024, 0, s>>>(in, n, sums, out);
}

template <typename T, bool POSE>
static void launch_units(const float *gz, const GatherLayout &L, const uint32_t *sorted, const uint32_t *order, const GatherArgs &G, const void *vol,
                         const PoseOut &po, int unit, int grid, cudaStream_t s)
{
    k_gather_units<T, POSE><<<grid, kGatherWarps * 32, 0, s>>>(gz, L.runs, L.steps, sorted, L.bstart, L.bend, L.ustart,
                                                             L.unit_brick, L.misc + 0, G, unit, L.upart, L.zero + 32,
                                                             order, (const T *)vol, po);
}

int launch_gather(const diffus_volume_desc *vd, const void *vol, const RayGeo *geo, long long n_rays,
                  double max_path_mm, const float *gz, const long long *gz_off, void *ws, uint32_t *status,
                  float *grad_vol, double *pose_part, int ctas_per_sm, cudaStream_t s, const GatherMarks &marks)
{
    const GatherArgs G = make_gather_args(vd);
    const int nb = G.nbx * G.nby * G.nbz;
    const int cap = runs_per_ray(vd, max_path_mm);
    GatherLayout L = gather_layout(ws, vd, n_rays, cap);
    const size_t slots = (size_t)n_rays * cap;
    const int unit = unit_runs(slots);
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);

    const bool by_rank = cap - 1 <= kRunMax && sort_by_rank(slots, (size_t)nb);
    const size_t zbytes = (by_rank ? (char *)(L.bcount + nb) : (char *)(L.bwork + nb)) - (char *)L.zero;
    if (cudaMemsetAsync(L.zero, 0, zbytes, s) != cudaSuccess) return DIFFUS_E_LAUNCH;
    const int wgrid = (int)((n_rays + kRunWarps - 1) / kRunWarps);
    const int pgrid = (nb + kPlanThreads - 1) / kPlanThreads;
    const uint32_t *sorted, *order = nullptr;
    auto brick_plan = [&] {
        if (nb > kPlanDirect) k_brick_sums<<<pgrid, kPlanThreads, 0, s>>>(L.bcount, nb, unit, L.bsums);
        k_brick_plan<<<pgrid, kPlanThreads, 0, s>>>(L.bcount, nb > kPlanDirect ? L.bsums : nullptr, nb, unit, L.bstart,
                                                    L.bend, L.ucount, L.ustart, L.unit_brick, L.misc + 0, L.misc + 1);
    };
    if (by_rank) {
        k_ray_runs_warp<true><<<wgrid, kRunWarps * 32, 0, s>>>(geo, gz_off, (int)n_rays, G, cap, L.runs, L.steps, L.keys[0],
                                                              L.nrun, L.bcount, L.keys[1], nullptr, status);
        brick_plan();
        uint2 *list = reinterpret_cast<uint2 *>(L.vals[0]);
        k_place_runs<<<dim3((unsigned)((n_rays + 127) / 128), (unsigned)cap), 128, 0, s>>>(
            L.keys[0], L.keys[1], L.nrun, (int)n_rays, L.bstart, list);
        // the ranked order replaces the arrivals, which the list has absorbed
        k_rank_runs<<<(unsigned)((slots + 127) / 128), 128, 0, s>>>(list, L.misc + 1, L.bstart, L.bend, L.keys[1]);
        sorted = L.keys[1];
    } else {
        if (cudaMemsetAsync(L.keys[0], 0xff, sizeof(uint32_t) * slots, s) != cudaSuccess) return DIFFUS_E_LAUNCH;
        if (cap - 1 <= kRunMax && n_rays <= kRunWarpRays)
            k_ray_runs_warp<false><<<wgrid, kRunWarps * 32, 0, s>>>(geo, gz_off, (int)n_rays, G, cap, L.runs, L.steps,
                                                                   L.keys[0], L.nrun, L.bcount, nullptr, L.bwork,
                                                                   status);
        else
            k_ray_runs<<<(unsigned)((n_rays + 127) / 128), 128, 0, s>>>(geo, gz_off, (int)n_rays, G, cap, L.runs, L.steps,
                                                                       L.keys[0], L.nrun, L.bcount, L.bwork, status);
        brick_plan();
        // stable LSD radix sort by brick
        const int bits = sort_bits(nb);
        const int nblk = (int)((slots + kSortTile - 1) / kSortTile);
        int cur = 0;
        for (int shift = 0; shift < bits; shift += 8) {
            if (shift == 0)
                k_digit_hist<true><<<nblk, kSortThreads, 0, s>>>(L.keys[cur], slots, L.misc + 1, shift, nblk, L.hist);
            else
                k_digit_hist<false><<<nblk, kSortThreads, 0, s>>>(L.keys[cur], slots, L.misc + 1, shift, nblk, L.hist);
            launch_scan(L.hist, L.hist, (size_t)256 * nblk, L.sums, nullptr, s);
            if (shift == 0)
                k_digit_scatter<true><<<nblk, kSortThreads, 0, s>>>(L.keys[cur], L.vals[cur], slots, L.misc + 1, shift,
                                                                    nblk, L.hist, L.keys[cur ^ 1], L.vals[cur ^ 1]);
            else
                k_digit_scatter<false><<<nblk, kSortThreads, 0, s>>>(L.keys[cur], L.vals[cur], slots, L.misc + 1,
                                                                     shift, nblk, L.hist, L.keys[cur ^ 1],
                                                                     L.vals[cur ^ 1]);
            cur ^= 1;
        }
        sorted = L.vals[cur];
        // longest-first unit order (by classes of work), so that no long unit starts last
        k_unit_work<<<sms, 256, 0, s>>>(L.bwork, L.bstart, L.bend, L.ustart, L.unit_brick, L.misc + 0, unit, L.uclass,
                                        L.zero);
        k_class_cursors<<<1, 32, 0, s>>>(L.zero);
        k_unit_order<<<sms * 4, 256, 0, s>>>(L.uclass, L.misc + 0, L.zero, L.uorder);
        order = L.uorder;
    }
    record_mark(marks.units, marks.external, s);
    const int grid = sms * ctas_per_sm;
    const PoseOut po{L.rpart, slots};
    if (!pose_part)
        launch_units<float, false>(gz, L, sorted, order, G, vol, po, unit, grid, s);
    else if (vd->dtype == DIFFUS_F32)
        launch_units<float, true>(gz, L, sorted, order, G, vol, po, unit, grid, s);
    else
        launch_units<unsigned short, true>(gz, L, sorted, order, G, vol, po, unit, grid, s);
    record_mark(marks.reduce, marks.external, s);
    const bool rvec = vd->nx % kRedVox == 0 && (uintptr_t)grad_vol % 16 == 0;
    int rx = 4;
    while (rx < 64 && rx * kRedVox < vd->nx) rx *= 2;
    const dim3 rblk((unsigned)rx, (unsigned)(256 / rx));
    const dim3 rgrid((unsigned)((vd->nx + rx * kRedVox - 1) / (rx * kRedVox)),
                     (unsigned)((vd->ny + rblk.y - 1) / rblk.y), (unsigned)vd->nz);
    k_voxel_reduce<<<rgrid, rblk, 0, s>>>(L.upart, L.ustart, L.ucount, G, grad_vol, rvec);
    if (pose_part)
        k_ray_pose<<<(unsigned)((n_rays + 31) / 32), 192, 0, s>>>(
            L.rpart, slots, L.nrun, geo, (int)n_rays, (float)(1.0 / vd->sx), (float)(1.0 / vd->sy),
            (float)(1.0 / vd->sz), pose_part);
    return launch_status();
}

}  // namespace dfs
