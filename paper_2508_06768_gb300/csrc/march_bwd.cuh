// Adjoint of the warp-per-ray march (reverse mode of Sections 2.3-2.4).
//
// For L = sum_i ge_i e_i with ge_i = speckle_i * dL/dy_i, the adjoint of the
// bottom-row state (b_i, D_i) obeys
//     lambda_i = de_i/db_i ge_i + lambda_{i+1} M_i^T,   mu_i = de_i/dD_i ge_i + mu_{i+1} delta_i,
// an affine recurrence run from the end of the ray.  Each lane owns 8
// interfaces of a 256-interface segment; the lanes' affine maps are combined
// by a warp suffix scan, so the reverse sweep is as parallel as the forward
// one.  Per-ray recomputation replaces stored march state: a forward sweep
// keeps only the scan carry at each segment start (16 bytes per segment),
// then segments are revisited from the last to the first.
//
// Outputs per ray: dL/dZ_k for the S+1 samples (for the volume gather) and,
// with POSE, the ray's contribution to dL/dpose (FP64 sums of per-segment
// FP32 sums).  Without POSE the march samples values only; the brick gather
// then forms the pose gradient from dL/dZ and the cells' corners.
#pragma once

#include "march.cuh"

namespace dfs {

constexpr int kBwdPad = 289;   // smem_idx(256) + 1

template <bool POSE, bool STORED = false>
struct BwdSmem {
    static constexpr int kZ = STORED ? 1 : kBwdPad;
    float4 eg[kSeg];                  // echo partials of interface lane*8+t at [t*32 + lane] (both reverse passes)
    float zr[kZ], dz[kZ];             // samples base .. base+256 (zref + dz form; not STORED)
    float gx[POSE ? kBwdPad : 1], gy[POSE ? kBwdPad : 1], gz[POSE ? kBwdPad : 1];   // dZ/dp (POSE)
    double acc[POSE ? 6 : 1];         // the ray's pose-gradient sums (lane 0)
};

// Echo of one interface and its partial derivatives with respect to the
// state (b0, b1, D) and to x = m01 (see march.cuh for e).
struct EchoGrad {
    float gb0, gb1, gD, gx;
};

__device__ __forceinline__ EchoGrad echo_grad(float b0, float b1, float D, float x, float ge)
{
    if (ge == 0.0f) return {0.0f, 0.0f, 0.0f, 0.0f};   // masked rows (e.g. past a pole) add nothing
    float q = fmaf(b0, x, b1);
    float iq = frcp(q), ib1 = frcp(b1);
    float e = x * D * ib1 * iq;
    EchoGrad g;
    g.gb0 = -ge * e * x * iq;
    g.gb1 = -ge * e * (ib1 + iq);
    g.gD = ge * x * ib1 * iq;
    g.gx = ge * D * iq * iq;
    return g;
}

// have_ckpt: the forward march of the same call already wrote the segment
// carries into ckpt, so the recording sweep is skipped.
// mrow: speckle factors written by the forward of the same call (nullable;
// recomputed from Philox when absent).
// STORED (requires have_ckpt, not POSE): the forward of the same call kept,
// per sample k, zref + dz in zrow and r_{k-1} in rrow, so the march reads them
// instead of resampling the volume (the same values bit for bit), each lane
// its own chunk in 16-byte loads.
// gy_vec: gy_row is an internal row (aligned, row_stride long); mrow always is.
// gz_row, zrow and rrow lie kGzLead floats into an aligned block of
// gz_stride(S).  Only the gather reads dL/dZ, so POSE (which runs without one)
// does not write it.
//
// MULTI (not STORED; mm is the block's): all warps of the block march one ray,
// a segment each, side by side up to the true reverse pass, which runs in turn
// from the last segment to the first and hands the adjoint on through shared
// memory: the same arithmetic in the same order, for fans too small to fill
// the GPU with one warp per ray.
//
// Past the ray's end r and the adjoint sources are 0, so the passes need no
// row tests; only the Z1-role term of interface S, which would reach sample
// S, is dropped explicitly.
struct BwdMulti {
    float4 q[32];            // segment totals (first sweep)
    float d[32];
    float lam0, lam1, mu, carry;   // adjoint at the end of the segment whose turn it is
};

template <typename T, int MODE, bool POSE, bool STORED = false, bool MULTI = false>
__device__ void march_bwd_ray(const T *__restrict__ vol, const MarchArgs &A, const RayGeo &rg,
                              const float *__restrict__ gy_row, float *__restrict__ gz_row,
                              double *__restrict__ pose_part, float4 *__restrict__ ckpt, BwdSmem<POSE, STORED> &sm,
                              bool gy_vec, bool have_ckpt = false, const float *__restrict__ mrow = nullptr,
                              const float *__restrict__ zrow = nullptr, const float *__restrict__ rrow = nullptr,
                              BwdMulti *mm = nullptr, double *macc = nullptr)
{
    static_assert(!(STORED && MULTI), "the batched march takes one ray per warp");
    static_assert(!(STORED && POSE), "the pose terms of the march need the sampled gradient");
    // The batched call (STORED) streams gigabytes of one-pass rows: evict-
    // first loads and stores keep them from displacing reused L2 lines.  The
    // small single-pose rows stay ordinary.
    auto ld_once = [](const float *p) { return STORED ? __ldcs(p) : __ldg(p); };
    const int lane = threadIdx.x & 31;
    const int S = rg.S;
    const float a2 = A.a2;
    const int nseg = (S + kSeg - 1) / kSeg;

    const int w = MULTI ? (int)(threadIdx.x >> 5) : 0, nw = MULTI ? (int)(blockDim.x >> 5) : 1;

    // ---------------- sweep 1: forward, record the carry at segment starts
    // (the last segment's totals reach no carry)
    if (!STORED && !have_ckpt) {
        float czr, cdz;
        if (!MULTI) sample_z<T, false>(vol, A.g, rg.X0[0], rg.X0[1], rg.X0[2], czr, cdz);
        float bs0 = 0.0f, bs1 = 1.0f, Ds = 1.0f;
        if (lane == 0 && w == 0) ckpt[0] = make_float4(bs0, bs1, Ds, 0.0f);
        for (int s0 = 0; s0 < nseg - 1; s0 += nw) {
            const int s = s0 + w;
            Mat2 Qall;
            float dall;
            if (s < nseg - 1) {
                if (MULTI) {
                    long long X, Y, Z;
                    sample_pos(rg, s * kSeg, X, Y, Z);
                    sample_z<T, false>(vol, A.g, X, Y, Z, czr, cdz);
                }
                float rr[kChunk];
                seg_coefficients<T, false>(vol, A.g, rg, s * kSeg, czr, cdz, reinterpret_cast<float2 *>(sm.eg),
                                           nullptr, rr);
                Mat2 Q, E;
                float dq, de;
                chunk_product<MODE>(rr, a2, Q, dq);
                warp_scan_prefix(Q, dq, E, de, Qall, dall);
                if (MULTI && lane == 0) {
                    mm->q[w] = make_float4(Qall.a, Qall.b, Qall.c, Qall.d);
                    mm->d[w] = dall;
                }
            }
            if (MULTI) __syncthreads();
            for (int v = 0; v < nw && s0 + v < nseg - 1; v++) {
                if (MULTI) {
                    const float4 q = mm->q[v];
                    Qall = {q.x, q.y, q.z, q.w};
                    dall = mm->d[v];
                }
                float n0 = fmaf(bs0, Qall.a, bs1 * Qall.c);
                float n1 = fmaf(bs0, Qall.b, bs1 * Qall.d);
                bs0 = n0;
                bs1 = n1;
                Ds *= dall;
                if (lane == 0 && w == 0) ckpt[s0 + v + 1] = make_float4(bs0, bs1, Ds, 0.0f);
            }
            if (MULTI) __syncthreads();
        }
    }
    if (MULTI) {
        if (threadIdx.x == 0) mm->lam0 = mm->lam1 = mm->mu = mm->carry = 0.0f;
        __syncthreads();
    } else {
        __syncwarp();
    }

    // ---------------- sweep 2: reverse over segments
    float lam0 = 0.0f, lam1 = 0.0f, mus = 0.0f;   // adjoint at the end of the current segment
    float carry_gz1 = 0.0f;                       // dL/dZ of sample base+256 from interface base+256
    float czr = 0.0f, cdz = 0.0f, cg0 = 0.0f, cg1 = 0.0f, cg2 = 0.0f;   // sample base+256
    double *acc = MULTI ? macc : sm.acc;
    if (POSE && lane == 0 && w == 0)
        for (int q = 0; q < 6; q++) acc[q] = 0.0;
    const float ds = rg.ds;

    for (int s0 = nseg - 1; s0 >= 0; s0 -= nw) {
        const bool on = !MULTI || s0 >= w;   // a warp without a segment repeats segment 0 and writes nothing
        const int s = on ? s0 - w : 0;
        const int base = s * kSeg;
        const int i0 = base + lane * kChunk;
        float rr[kChunk];
        if (STORED) {
            load_chunk(rrow + i0 + 1, i0 < S, rr);   // r_{i0+t} is kept with sample i0+t+1, 0 past the ray
        } else {
            // A': samples base .. base+255 (with dZ/dp when POSE); sample base+256 carried
            long long X, Y, Z;
            sample_pos(rg, base + lane, X, Y, Z);
            const long long sX = rg.DX[0] * kWarp, sY = rg.DX[1] * kWarp, sZ = rg.DX[2] * kWarp;
            constexpr int kGroup = POSE ? 1 : kSampleGroup;
#pragma unroll
            for (int t0 = 0; t0 < kChunk; t0 += kGroup) {
                if (base + t0 * kWarp <= S) {   // past the ray a lane samples at a clamped position
#pragma unroll
                    for (int t = t0; t < t0 + kGroup; t++) {
                        float zr, dz, g3[3];
                        sample_z<T, POSE>(vol, A.g, X, Y, Z, zr, dz, g3);
                        X += sX;
                        Y += sY;
                        Z += sZ;
                        int o = smem_idx(t * kWarp + lane);
                        sm.zr[o] = zr; sm.dz[o] = dz;
                        if (POSE) { sm.gx[o] = g3[0]; sm.gy[o] = g3[1]; sm.gz[o] = g3[2]; }
                    }
                }
            }
            if (lane == 0) {
                if ((MULTI || s == nseg - 1) && base + kSeg <= S) {
                    float g3[3];
                    sample_pos(rg, base + kSeg, X, Y, Z);
                    sample_z<T, POSE>(vol, A.g, X, Y, Z, czr, cdz, g3);
                    if (POSE) { cg0 = g3[0]; cg1 = g3[1]; cg2 = g3[2]; }
                }
                int o = smem_idx(kSeg);
                sm.zr[o] = czr; sm.dz[o] = cdz;
                if (POSE) { sm.gx[o] = cg0; sm.gy[o] = cg1; sm.gz[o] = cg2; }
            }
            __syncwarp();
            {   // carry the first sample of this segment to the earlier one
                int o = smem_idx(0);
                czr = sm.zr[o]; cdz = sm.dz[o];
                if (POSE) { cg0 = sm.gx[o]; cg1 = sm.gy[o]; cg2 = sm.gz[o]; }
            }
#pragma unroll
            for (int t = 0; t < kChunk; t++) {
                int o = smem_idx(lane * kChunk + t), o1 = smem_idx(lane * kChunk + t + 1);
                rr[t] = (i0 + t < S) ? refl(sm.zr[o], sm.dz[o], sm.zr[o1], sm.dz[o1]) : 0.0f;
            }
        }
        // adjoint sources of the echo rows
        float m[kChunk];
        if (mrow) {
            load_chunk(mrow + i0, i0 < S, m);
        } else if (!STORED && A.sp.on) {
            chunk_speckle(A.sp, i0, S, rg.ray, A.sp.pose_ctr + (uint32_t)rg.pose, m);
        } else {
#pragma unroll
            for (int t = 0; t < kChunk; t++) m[t] = 1.0f;
        }
        float ge[kChunk];
        if (gy_vec) {
            load_chunk(gy_row + i0, i0 < S, ge);
        } else {
#pragma unroll
            for (int t = 0; t < kChunk; t++) ge[t] = (i0 + t < S) ? ld_once(gy_row + i0 + t) : 0.0f;
        }
#pragma unroll
        for (int t = 0; t < kChunk; t++) ge[t] = (i0 + t < S) ? m[t] * ge[t] : 0.0f;

        // B': the chunk's forward states
        Mat2 Q, E, Qall;
        float dq, de, dall;
        chunk_product<MODE>(rr, a2, Q, dq);
        warp_scan_prefix(Q, dq, E, de, Qall, dall);
        const float4 ck = ckpt[s];
        float b0s[kChunk], b1s[kChunk], Dsv[kChunk];
        {
            float b0 = fmaf(ck.x, E.a, ck.y * E.c);
            float b1 = fmaf(ck.x, E.b, ck.y * E.d);
            float D = ck.z * de;
#pragma unroll
            for (int t = 0; t < kChunk; t++) {
                b0s[t] = b0; b1s[t] = b1; Dsv[t] = D;
                const Xfer x = xfer_t<MODE>(rr[t], a2);
                float nb0 = fmaf(b0, x.m00, b1 * x.m10);
                b1 = fmaf(b0, x.m01, b1);
                b0 = nb0;
                D *= x.delta;
            }
        }

        // C': local reverse pass with zero adjoint at the chunk end; the
        // echo partials are kept for the true pass
        float c0 = 0.0f, c1 = 0.0f, dloc = 0.0f;
#pragma unroll
        for (int t = kChunk - 1; t >= 0; t--) {
            const Xfer x = xfer_t<MODE>(rr[t], a2);
            EchoGrad g = echo_grad(b0s[t], b1s[t], Dsv[t], x.m01, ge[t]);
            sm.eg[t * kWarp + lane] = make_float4(g.gb0, g.gb1, g.gD, g.gx);
            // explicit adds: the partials are not fused here either, as
            // in the true pass, which reads them back
            float n0 = __fadd_rn(g.gb0, fmaf(c0, x.m00, c1 * x.m01));
            float n1 = __fadd_rn(g.gb1, fmaf(c0, x.m10, c1));
            dloc = fmaf(dloc, x.delta, g.gD);
            c0 = n0;
            c1 = n1;
        }
        // impedances of samples i0+1 .. i0+8 (and of i0), on their way during the scan
        float zz[kChunk], z_first = 0.0f;
        if (STORED) {
            load_chunk(zrow + i0 + 1, i0 < S, zz);
            if (lane == 0) z_first = __ldcs(zrow + base);
        }
        // D': warp suffix scan of the affine maps (lambda -> c + lambda Q^T, mu -> d + mu dq)
        Mat2 Pm = Q;          // chunk product (warp_scan_prefix took Q by value)
        float pal = dq;
        float pc0 = c0, pc1 = c1, pd = dloc;
#pragma unroll
        for (int off = 1; off < kWarp; off <<= 1) {
            Mat2 Po = {__shfl_down_sync(0xffffffffu, Pm.a, off), __shfl_down_sync(0xffffffffu, Pm.b, off),
                       __shfl_down_sync(0xffffffffu, Pm.c, off), __shfl_down_sync(0xffffffffu, Pm.d, off)};
            float o0 = __shfl_down_sync(0xffffffffu, pc0, off);
            float o1 = __shfl_down_sync(0xffffffffu, pc1, off);
            float oal = __shfl_down_sync(0xffffffffu, pal, off);
            float od = __shfl_down_sync(0xffffffffu, pd, off);
            if (lane + off < kWarp) {
                // self o other: c + c_o P^T, P P_o ; d + d_o al, al al_o
                float n0 = pc0 + fmaf(o0, Pm.a, o1 * Pm.b);
                float n1 = pc1 + fmaf(o0, Pm.c, o1 * Pm.d);
                pc0 = n0;
                pc1 = n1;
                pd = fmaf(od, pal, pd);
                Pm = mat_mul(Pm, Po);
                pal *= oal;
            }
        }
        for (int turn = 0; turn < nw; turn++) {
            if (MULTI) {
                __syncthreads();
                if (turn != w || !on) continue;
                lam0 = mm->lam0;
                lam1 = mm->lam1;
                mus = mm->mu;
                carry_gz1 = mm->carry;
            }
            // adjoint at this lane's chunk end = G_{lane+1}(lambda_seg)
            float le0, le1, lmu;
            {
                Mat2 Po = {__shfl_down_sync(0xffffffffu, Pm.a, 1), __shfl_down_sync(0xffffffffu, Pm.b, 1),
                           __shfl_down_sync(0xffffffffu, Pm.c, 1), __shfl_down_sync(0xffffffffu, Pm.d, 1)};
                float o0 = __shfl_down_sync(0xffffffffu, pc0, 1);
                float o1 = __shfl_down_sync(0xffffffffu, pc1, 1);
                float oal = __shfl_down_sync(0xffffffffu, pal, 1);
                float od = __shfl_down_sync(0xffffffffu, pd, 1);
                if (lane == kWarp - 1) {
                    le0 = lam0; le1 = lam1; lmu = mus;
                } else {
                    le0 = o0 + fmaf(lam0, Po.a, lam1 * Po.b);
                    le1 = o1 + fmaf(lam0, Po.c, lam1 * Po.d);
                    lmu = fmaf(mus, oal, od);
                }
            }

            // E': true reverse pass: parameter adjoints -> dL/dr -> dL/dZ.
            // dL/dZ of sample i0+t+1 (t < 7) is complete once interfaces t and
            // t+1 are done, so it is finalised inside the loop; sample i0+8 also
            // needs the next lane's interface and is finalised after it.
            float a[6] = {0, 0, 0, 0, 0, 0};
            float c_next = 0.0f;     // Z1-role contribution of interface t+1 to sample i0+t+1
            float n_last = 0.0f;     // Z2-role contribution of interface i0+7 to sample i0+8
            float c_first = 0.0f;    // Z1-role contribution of interface i0 to sample i0
            float G[kChunk];         // dL/dZ of samples i0+1 .. i0+8
            auto add_pose = [&](int k, int o, float g) {
                if (!POSE) return;
                const float gx = sm.gx[o], gyv = sm.gy[o], gzv = sm.gz[o];
                const float sk = ((float)k + 0.5f) * ds;
                a[0] = fmaf(g, gx, a[0]);
                a[1] = fmaf(g, gyv, a[1]);
                a[2] = fmaf(g, gzv, a[2]);
                a[3] = fmaf(g * sk, gx, a[3]);
                a[4] = fmaf(g * sk, gyv, a[4]);
                a[5] = fmaf(g * sk, gzv, a[5]);
            };
            if (STORED) {
                const float zl = __shfl_up_sync(0xffffffffu, zz[kChunk - 1], 1);
                if (lane) z_first = zl;
            }
#pragma unroll
            for (int t = kChunk - 1; t >= 0; t--) {
                const float r = rr[t];
                const Xfer x = xfer_t<MODE>(r, a2);
                float gm00 = b0s[t] * le0, gm10 = b1s[t] * le0, gm01 = b0s[t] * le1;
                float gdel = lmu * Dsv[t];
                const float4 gv = sm.eg[t * kWarp + lane];   // written by this lane in C'
                const EchoGrad g{gv.x, gv.y, gv.z, gv.w};
                float gr;
                if (MODE == DIFFUS_MODE_LITERAL) {
                    float R = fabsf(r);
                    float gR = gm00 * (-4.0f * a2 * R) + (gm01 + g.gx) * a2 - gm10 + gdel * (-2.0f * a2 * R);
                    gr = r > 0.0f ? gR : (r < 0.0f ? -gR : 0.0f);
                } else {
                    gr = (gm01 + g.gx) * a2 + gm10 + gdel * (-2.0f * a2 * r);
                }
                float n0 = g.gb0 + fmaf(le0, x.m00, le1 * x.m01);
                float n1 = g.gb1 + fmaf(le0, x.m10, le1);
                lmu = fmaf(lmu, x.delta, g.gD);
                le0 = n0;
                le1 = n1;
                float z1, z2;
                if (STORED) {
                    z1 = t == 0 ? z_first : zz[t == 0 ? 0 : t - 1];
                    z2 = zz[t];
                } else {
                    const int o1 = smem_idx(lane * kChunk + t), o2 = smem_idx(lane * kChunk + t + 1);
                    z1 = sm.zr[o1] + sm.dz[o1];
                    z2 = sm.zr[o2] + sm.dz[o2];
                }
                const float sz = z1 + z2;
                const float is2 = frcp(sz * sz);
                const float gzc = i0 + t < S ? gr * (-2.0f * z2) * is2 : 0.0f;
                const float gzn = gr * (2.0f * z1) * is2;
                if (t == kChunk - 1) {
                    n_last = gzn;
                } else {
                    const int k = i0 + t + 1;
                    G[t] = c_next + gzn;
                    if (k <= S) add_pose(k, smem_idx(lane * kChunk + t + 1), G[t]);
                }
                c_next = gzc;
                if (t == 0) c_first = gzc;
            }
            // adjoint at the segment start for the earlier segment
            lam0 = __shfl_sync(0xffffffffu, le0, 0);
            lam1 = __shfl_sync(0xffffffffu, le1, 0);
            mus = __shfl_sync(0xffffffffu, lmu, 0);

            // F': sample i0+8 (the next lane's first sample) and sample 0
            {
                float nextc = __shfl_down_sync(0xffffffffu, c_first, 1);
                if (lane == kWarp - 1) nextc = carry_gz1;
                const int k = i0 + kChunk;
                G[kChunk - 1] = n_last + nextc;
                if (k <= S) add_pose(k, smem_idx(lane * kChunk + kChunk), G[kChunk - 1]);
                if (!POSE && i0 < S) {
                    // samples i0+1 .. i0+8 lie on one aligned sector (samples past
                    // S fall into the block's padding)
                    float4 *dst = reinterpret_cast<float4 *>(gz_row + i0 + 1);
                    const float4 lo = make_float4(G[0], G[1], G[2], G[3]), hi = make_float4(G[4], G[5], G[6], G[7]);
                    if (STORED) {
                        __stcs(dst, lo);
                        __stcs(dst + 1, hi);
                    } else {
                        dst[0] = lo;
                        dst[1] = hi;
                    }
                }
            }
            if (s == 0 && lane == 0) {
                if (!POSE) gz_row[0] = c_first;
                add_pose(0, smem_idx(0), c_first);
            }
            carry_gz1 = __shfl_sync(0xffffffffu, c_first, 0);
            if (POSE) {
#pragma unroll
                for (int q = 0; q < 6; q++) {
                    float v = a[q];
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                    if (lane == 0) acc[q] += (double)v;
                }
            }
            if (MULTI && lane == 0) {
                mm->lam0 = lam0;
                mm->lam1 = lam1;
                mm->mu = mus;
                mm->carry = carry_gz1;
            }
        }
        __syncwarp();
    }
    if (MULTI) __syncthreads();
    if (POSE && lane == 0 && w == 0) {
        pose_part[0] = acc[0];
        pose_part[1] = acc[1];
        pose_part[2] = acc[2];
        for (int q = 0; q < 3; q++)
            pose_part[3 + q] = acc[3] * (double)rg.v[q][0] + acc[4] * (double)rg.v[q][1] + acc[5] * (double)rg.v[q][2];
    }
}

}  // namespace dfs
