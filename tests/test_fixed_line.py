"""The fixed-point line of a ray and the counts that walk it from cell to cell
and from brick to brick (csrc/gather.cuh), compiled for the host: every sample
of every run lies in the run's brick and in the cell its record names, for
poses of any value a device buffer can hold."""
import os
import subprocess

import pytest

from paper_2508_06768_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include "host.hpp"
#include "gather.cuh"
using namespace dfs;

static int fails = 0;
#define CHECK(c, ...) do { if (!(c)) { if (fails++ < 5) { printf(__VA_ARGS__); printf("\n"); } } } while (0)

static long long at(long long X0, long long DX, long long k)   // wraps as the kernels' registers do
{
    return (long long)((unsigned long long)X0 + (unsigned long long)k * (unsigned long long)DX);
}

// One axis of one ray: runs by next_change, cells by first_steps1 and next_steps.
static void walk(double x0, double dx, int n, int S)
{
    const long long X0 = to_fixed(x0), DX = step_fixed(dx);
    const uint2 qr = cell_steps(DX);
    const long long d3[3] = {DX, DX, DX};
    const FirstSteps fs = first_steps_of(d3);
    int b = cell_of(X0, n) / kBrick;
    for (long long k = 0; k <= S;) {
        const long long kn = next_change(X0, DX, b, n, S);
        CHECK(kn > k, "no progress: x0 %g dx %g n %d S %d at %lld", x0, dx, n, S, k);
        if (kn <= k) return;
        int left = (int)((kn - 1 < S ? kn - 1 : S) - k + 1);
        long long X = at(X0, DX, k), kk = k;
        int c = first_steps1(X, DX, fs.q[0], fs.inv[0], n);
        CHECK(c >= 1 && c <= kNextMax, "first count %d", c);
        while (left > 0) {
            const int len = std::min(c, std::min(left, kGCellCap));
            int i;
            float u, v;
            axis_cell(X, slope_of(DX), n, i, u, v);
            CHECK(i >= b * kBrick && i < (b + 1) * kBrick && i <= n - 2,
                  "x0 %g dx %g n %d S %d: sample %lld in cell %d, its run in brick %d", x0, dx, n, S, kk, i, b);
            if (len < 1) return;
            for (int q = 0; q < len; q++) {
                const long long Y = at(X0, DX, kk + q);
                CHECK(cell_of(Y, n) == i, "x0 %g dx %g n %d S %d: sample %lld in cell %d, its record in %d", x0, dx, n,
                      S, kk + q, cell_of(Y, n), i);
            }
            X = at(X, DX, len);
            kk += len;
            left -= len;
            c -= len;
            if (left > 0 && c == 0) c = next_steps(X, DX, n, qr);
            if (fails > 5) return;
        }
        k = kn;
        if (k <= S) b = cell_of(at(X0, DX, k), n) / kBrick;
    }
}

int main()
{
    const double nan = std::nan(""), inf = INFINITY;
    const int sizes[] = {2, 3, 9, 10, 17, 64, 400}, rows[] = {1, 2, 31, 1022, 1023, 1024, 1055, 4200};
    const double bad[] = {nan, -nan, inf, -inf, 1e300, -1e300, 1e9, -3e9};
    srand(1);
    auto uni = [] { return rand() / (double)RAND_MAX; };
    for (int n : sizes)
        for (int S : rows) {
            // the longest step that the entry points take: 2^29 voxels over the fan
            const double lim = 536870912.0 / S;
            for (double x0 : bad)
                for (double dx : {nan, -nan, 0.0, 0.3, -0.3, 1e-9, -1e-9, 9.0, lim, -lim}) walk(x0, dx, n, S);
            for (double dx : {nan, -nan, lim, -lim, 0.0, 0x1p-32, -0x1p-32})
                for (double x0 : {0.0, 3.25, n - 1.0, n - 1.5, -0.5}) walk(x0, dx, n, S);
            for (int q = 0; q < 60; q++) {
                const double span = uni() < 0.5 ? n : 0.05 * n;
                double dx = (uni() - 0.5) * 4.0 * span / S, x0 = uni() * 1.4 * n - 0.2 * n;
                if (q % 4 == 1) x0 = std::floor(x0);
                if (q % 4 == 2) dx = std::ldexp(1.0, -(int)(uni() * 12)) * (q % 8 == 2 ? 1 : -1);
                walk(x0, dx, n, S);
            }
        }
    // a spacing whose reciprocal is not finite still gives a step
    diffus_volume_desc vd{8, 8, 8, DIFFUS_F32, 1e-310, 5e-324, 1.0, 0.0, 0.0, 0.0};
    const VolPlace vp = make_place(&vd);
    for (double s : {vp.isx, vp.isy, vp.isz})
        for (double u : {0.0, 1e-310, 5e-320}) CHECK(std::isfinite(u * s), "step %g x %g", u, s);
    printf("%d faults\n", fails);
    return fails ? 1 : 0;
}
"""


@pytest.fixture(scope="module")
def host_program(tmp_path_factory):
    """Compiles a source against the kernels' headers and returns its path."""
    def compile_(source):
        d = tmp_path_factory.mktemp("host")
        (d / "t.cu").write_text(source)
        subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-I", B.INCLUDE, "-I", B.CSRC,
                        "-o", str(d / "t"), str(d / "t.cu")], check=True, capture_output=True, text=True)
        return os.path.join(str(d), "t")
    return compile_


def test_cells_and_bricks_of_a_line(host_program):
    r = subprocess.run([host_program(SOURCE)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


RUNS = r"""
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <vector>
#include "host.hpp"
#include "gather.cuh"
using namespace dfs;

static int fails = 0;
#define CHECK(c, ...) do { if (!(c)) { if (fails++ < 5) { printf(__VA_ARGS__); printf("\n"); } } } while (0)

static int brick_at(const long long X0[3], const long long DX[3], const int n[3], int k)
{
    int b = 0;
    for (int a = 2; a >= 0; a--) b = b * 8192 + cell_of(X0[a] + k * DX[a], n[a]) / kBrick;
    return b;
}

// The runs of one ray as the warp-per-ray pass forms them, with room for cap.
static void runs_of(const long long X0[3], const long long DX[3], const int n[3], int S, int cap)
{
    std::vector<int> want{0};             // first sample of every run
    for (int k = 1; k <= S; k++)
        if (brick_at(X0, DX, n, k) != brick_at(X0, DX, n, k - 1)) want.push_back(k);
    const Cuts c = ray_cuts(X0, DX, S, n);
    const int m = c.off[3];
    CHECK(c.off[1] >= 0 && c.off[2] >= c.off[1] && m >= c.off[2] && m <= kRunMax, "entries %d %d %d", c.off[1], c.off[2], m);
    if (m > kRunMax || c.off[2] > kRunMax || c.off[1] > kRunMax) return;   // what follows would leave the lists
    if (!c.fits) {                        // no entry, no run: the pass reports the ray
        CHECK(m == 0 && (int)want.size() > 1, "%d entries of a ray that does not fit", m);
        return;
    }
    std::vector<int> k(m), start(m, -1);
    for (int e = 0; e < m; e++) k[e] = cut_sample(c, e, X0, DX, S);
    for (int e = 0; e < m; e++) {
        const int p = cut_rank(c, k.data(), m, e);
        CHECK(p >= 0 && p < m && start[p] == -1, "entry %d at place %d of %d", e, p, m);
        if (p >= 0 && p < m) start[p] = k[e];
    }
    int cnt = 1;
    for (int e = 0; e < m; e++)
        if (e == 0 || start[e] != start[e - 1]) k[cnt++ - 1] = start[e];
    CHECK(cnt == (int)want.size(), "%d runs, %d expected", cnt, (int)want.size());
    const int kept = std::min(cnt, cap);
    for (int i = 0; i < kept && !fails; i++) {
        int a, b;
        run_span(k.data(), i, cnt, S, a, b);
        CHECK(a == want[i] && b == (i + 1 < cnt ? want[i + 1] : S + 1), "run %d of %d (room for %d): %d..%d", i, cnt, cap,
              a, b);
    }
}

int main()
{
    srand(2);
    auto uni = [] { return rand() / (double)RAND_MAX; };
    const int shapes[][3] = {{44, 41, 37}, {2, 2, 2}, {9, 17, 64}, {700, 700, 600}, {2000, 2000, 16}, {16, 2000, 2000},
                             {65535, 16, 16}, {16, 16, 65535}};
    for (auto &n : shapes)
        for (int q = 0; q < 200; q++) {
            const int S = q % 5 == 0 ? 1 + (int)(uni() * 8) : 1 + (int)(uni() * 3000);
            long long X0[3], DX[3];
            for (int a = 0; a < 3; a++) {
                const double p = (uni() * 1.2 - 0.1) * n[a], e = (uni() * 1.2 - 0.1) * n[a];
                X0[a] = to_fixed(q % 3 ? p : std::floor(p));
                DX[a] = step_fixed(q % 7 == 0 && a ? 1.0 * (a == 1 ? 1 : -1) : (e - p) / S);
            }
            for (int cap : {256, 256, 40, 7, 2, 1}) runs_of(X0, DX, n, S, cap);
        }
    printf("%d faults\n", fails);
    return fails ? 1 : 0;
}
"""


def test_runs_of_a_ray_with_more_crossings_than_room(host_program):
    # a ray of more runs than slots, or of more crossings than the pass has
    # entries, loses the samples beyond; none lands in another brick's run
    r = subprocess.run([host_program(RUNS)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
