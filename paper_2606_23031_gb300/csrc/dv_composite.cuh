// Per-segment arithmetic, per-pixel state and set-up of the compositing kernels (dv_composite.cu: tiles
// without actors and the launches; dv_composite_act.cu: tiles that actor boxes cover).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "dv_internal.cuh"

namespace dv {

// One compositing pass: the call's constants and the buffers its kernels read and write.
struct CompositeArgs {
    BatchParams bp;
    const VoxRec* rec;
    const uint32_t* pval;        // record of each tile-sorted pair
    const uint16_t* prect;       // its voxel's pixel rectangle within the tile
    const uint2* tile_range;
    const uint32_t* vis_start;   // first record of every (view, octree)
    const uint32_t* tile_order;  // the launch's tiles, heaviest first
    uint32_t* n_seg;             // forward results kept per pixel
    float* t_final;
    const float *g_rgb, *g_depth, *g_alpha, *g_normal;  // backward: upstream gradients
    float* grad_rec;                                    //   and the records' gradient rows
    unsigned long long* work;                           // forward: work counters
    const int64_t* ex_off;                              // weights export
    uint32_t* ex_vid;
    float* ex_w;
    int n_spread;  // actor launches: the first n_spread tiles have a CTA per 8x4 block (see dv_composite_act.cu)
};

namespace {

constexpr int CT_THREADS = 128;
// per-record gradient slots: 8 densities, 3 colour (+ 3 normal with normals), padded to 16 bytes
template <bool NRM>
struct GradLayout {
    static constexpr int NV = NRM ? 14 : 11;      // values per record
    static constexpr int STRIDE = NRM ? 16 : 12;  // floats per record row
};

// With gradients, lanes that step through records of their own add their values with three 16-byte vector
// atomics; a chunk whose longest lane list is above 1 / LANE_GAIN of its records is visited in lockstep
// instead, where the warp sums a record's values first (2 against 1 and 3 on the 8M-leaf six-camera frame's plain
// tiles: 2,540 us, 2,718, 2,853).
constexpr int LANE_GAIN = 2;

struct PixBase {
    float C0, C1, C2, D, T;
    float Tp;  // transmittance before the last composited segment
    float R;  // residual form of the backward: sum over the composited segments of w (dL/dC . c + dL/dD mid)
    uint32_t n;
    uint32_t tests, boxes;  // work counters: voxel slab tests, actor box tests
    // the ray is composited up to here; -1 once it has stopped (or for a lane without a pixel), so that
    // the clip of a segment alone leaves it out
    float end;
    __device__ __forceinline__ bool done() const { return end < 0.0f; }
    __device__ __forceinline__ void stop() { end = -1.0f; }
};
template <bool NRM>
struct Pix : PixBase {};
template <>
struct Pix<true> : PixBase {
    float N0, N1, N2;  // normal state
};

struct BwdBase {
    // upstream gradient and the forward's results
    float g0, g1, g2, gD, gA;
    float Cf0, Cf1, Cf2, Df, Tend;
    float base;  // dL/dA T_end - (dL/dC . C_final + dL/dD D_final [+ dL/dN . N_final]), for the residual form
};
template <bool NRM>
struct Bwd : BwdBase {};
template <>
struct Bwd<true> : BwdBase {
    float gN0, gN1, gN2, Nf0, Nf1, Nf2;  // normal state: upstream gradient and final value
};

// per-lane writer of the composited segments' (voxel, weight) list (weights export)
struct ExportSink {
    uint32_t* vid;             // [total] voxel index within the view's concatenated octrees
    float* w;                  // [total] T alpha
    const uint32_t* sorted_g;  // record -> view * n_vox + voxel
    int64_t base, voff;        // first slot of this pixel; view * n_vox
    uint32_t n, lim;           // written so far; this pixel's slots
};

// 2^x on the SFU (ex2.approx.ftz: relative error about 2^-22)
__device__ __forceinline__ float ex2_sfu(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// exponential-linear activation: x above 1.1, 1.1 exp(x/1.1 - 1) below (C1 at 1.1).  The exponential
// branch is one SFU power of two, 1.1 exp(x/1.1 - 1) = 2^(x / (1.1 ln 2) + (ln 1.1 - 1) / ln 2), and
// its slope exp(x/1.1 - 1) is the same power divided by 1.1.
__device__ __forceinline__ float explin_low(float x) {
    return ex2_sfu(fmaf(x, 1.3115409462626941f, -1.3051915171390283f));
}

// thr: 1.1, or -infinity for the identity activation (BatchParams::act_thr)
__device__ __forceinline__ float act_fn(float x, float thr) { return x > thr ? x : explin_low(x); }

__device__ __forceinline__ float act_grad(float x, float thr) {
    return x > thr ? 1.0f : explin_low(x) * 0.90909090909090909f;
}

// exp(-x) on the SFU
__device__ __forceinline__ float exp_neg(float x) { return ex2_sfu(x * -1.4426950408889634f); }

__device__ __forceinline__ void rotate(const float* A, const float* x, float* y) {
#pragma unroll
    for (int r = 0; r < 3; ++r) y[r] = fmaf(A[r * 3 + 0], x[0], fmaf(A[r * 3 + 1], x[1], A[r * 3 + 2] * x[2]));
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Inverse ray direction, also split by sign, so that the slab test takes each axis's
// entry and exit plane without a min/max.  |d| is kept at or above 1e-20, so every
// product stays finite: a ray parallel to a slab gets entry and exit times of order
// 1e20 of the right signs instead of infinities (and NaN where inf - inf would meet).
struct InvDir {
    float inv[3];  // 1 / d
    float ip[3];   // 1 / d where d > 0, else 0
    float in[3];   // 1 / d where d < 0, else 0
};

__device__ __forceinline__ InvDir inv_dir(const float* d) {
    InvDir r;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float dk = fabsf(d[k]) < 1e-20f ? copysignf(1e-20f, d[k]) : d[k];
        r.inv[k] = 1.0f / dk;
        r.ip[k] = dk > 0.0f ? r.inv[k] : 0.0f;
        r.in[k] = dk < 0.0f ? r.inv[k] : 0.0f;
    }
    return r;
}

// Ray / voxel slab test.  g = (min corner - ray origin, size): along axis k the ray
// crosses the min plane at g_k / d_k and the max plane at (g_k + size) / d_k; which of
// the two it enters by follows from the sign of d_k.  The x and y axes go through packed two-lane
// multiplies and FMAs (the same roundings as scalar ones, half the instructions).  The ray misses the
// voxel where t1 <= t0; a caller that clips both ends only compares once, after the clip.
__device__ __forceinline__ void slab_cube(const InvDir& v, float4 g, float& t0, float& t1) {
    const float2 ww = make_float2(g.w, g.w);
    const float2 ta = __fmul2_rn(make_float2(g.x, g.y), make_float2(v.inv[0], v.inv[1]));
    const float2 en = __ffma2_rn(ww, make_float2(v.in[0], v.in[1]), ta);
    const float2 ex = __ffma2_rn(ww, make_float2(v.ip[0], v.ip[1]), ta);
    const float tz = g.z * v.inv[2];
    t0 = max3f(en.x, en.y, fmaf(g.w, v.in[2], tz));
    t1 = min3f(ex.x, ex.y, fmaf(g.w, v.ip[2], tz));
}


// optical depth of the segment [t0, t1] through one voxel (da, db: the record's density polynomial);
// optionally d tau / d dens[c] for the raw corner densities
// KS > 0: K known at compile time (KS); KS == 0: K from the launch.  With GRAD and a single sample
// (KS == 1), d tau / d dens[c] = s w_c(x, y, z) is left factored: sxyz receives (s, x, y, z), the
// activation's slope times the step and the sample's voxel coordinates, and dtd is not written.
template <bool GRAD, int KS>
__device__ __forceinline__ float seg_tau(float4 da, float4 db, float is, const float* rel, const float* d, float t0,
                                         float t1, int K_rt, float inv_k_rt, float thr, float* dtd, float* sxyz) {
    const int K = KS > 0 ? KS : K_rt;
    const float inv_k = KS == 1 ? 1.0f : inv_k_rt;
    const float h = (t1 - t0) * inv_k;
    float tau = 0.0f;
    if (GRAD && KS != 1) {
#pragma unroll
        for (int c = 0; c < 8; ++c) dtd[c] = 0.0f;
    }
    for (int k = 0; k < K; ++k) {
        const float t = KS == 1 ? 0.5f * (t0 + t1) : fmaf((float)k + 0.5f, h, t0);
        // voxel-local coordinates of the sample o + t d: (t d - (min - o)) / size
        const float x = __saturatef(fmaf(t, d[0], -rel[0]) * is);
        const float y = __saturatef(fmaf(t, d[1], -rel[1]) * is);
        const float z = __saturatef(fmaf(t, d[2], -rel[2]) * is);
        // the record holds the trilinear field as a polynomial (da = (c0, c3, c1, c5), db = (c2, c6, c4,
        // c7)): rho = (c0 + c1 x) + y (c2 + c4 x) + z ((c3 + c5 x) + y (c6 + c7 x)), the two x-linear
        // pairs and the two y steps taken as packed two-lane FMAs (same roundings as the scalar form)
        const float2 xx = make_float2(x, x);
        const float2 pA = __ffma2_rn(make_float2(da.z, da.w), xx, make_float2(da.x, da.y));
        const float2 pB = __ffma2_rn(make_float2(db.z, db.w), xx, make_float2(db.x, db.y));
        const float2 qq = __ffma2_rn(pB, make_float2(y, y), pA);
        const float rho = fmaf(qq.y, z, qq.x);
        tau += act_fn(rho, thr);
        if (GRAD && KS == 1) {
            sxyz[0] = act_grad(rho, thr) * h;
            sxyz[1] = x;
            sxyz[2] = y;
            sxyz[3] = z;
        } else if (GRAD) {
            const float s = act_grad(rho, thr) * h;
            const float x0 = 1.0f - x, y0 = 1.0f - y, z0 = 1.0f - z;
            dtd[0] = fmaf(s, x0 * y0 * z0, dtd[0]);
            dtd[1] = fmaf(s, x * y0 * z0, dtd[1]);
            dtd[2] = fmaf(s, x0 * y * z0, dtd[2]);
            dtd[3] = fmaf(s, x * y * z0, dtd[3]);
            dtd[4] = fmaf(s, x0 * y0 * z, dtd[4]);
            dtd[5] = fmaf(s, x * y0 * z, dtd[5]);
            dtd[6] = fmaf(s, x0 * y * z, dtd[6]);
            dtd[7] = fmaf(s, x * y * z, dtd[7]);
        }
    }
    return tau * h;
}

// Front-to-back compositing of one segment of optical depth tau; returns its weight T alpha.
template <bool NRM>
__device__ __forceinline__ float composite_step(Pix<NRM>& ps, float tau, float4 col, float4 nv, float t0, float t1) {
    const float e = exp_neg(tau);  // transmittance of the segment
    const float alpha = 1.0f - e;
    const float w = ps.T * alpha;
    const float mid = 0.5f * (t0 + t1);
    ps.C0 = fmaf(w, col.x, ps.C0);
    ps.C1 = fmaf(w, col.y, ps.C1);
    ps.C2 = fmaf(w, col.z, ps.C2);
    ps.D = fmaf(w, mid, ps.D);
    if constexpr (NRM) {
        ps.N0 = fmaf(w, nv.x, ps.N0);
        ps.N1 = fmaf(w, nv.y, ps.N1);
        ps.N2 = fmaf(w, nv.z, ps.N2);
    }
    ps.Tp = ps.T;
    ps.T = ps.T * e;
    ps.n += 1;
    return w;
}

template <bool NRM>
__device__ __forceinline__ void composite_tau(Pix<NRM>& ps, float tau, float4 col, float4 nv, float t0, float t1,
                                              float eps_stop) {
    composite_step<NRM>(ps, tau, col, nv, t0, t1);
    if (ps.T < eps_stop) ps.stop();
}

// d L / d dens[c] of one segment, added into acc[0..7], from gt = d L / d tau
template <int KS>
__device__ __forceinline__ void seg_density_grad(float gt, const float* dtd, const float* sxyz, float* acc) {
    if constexpr (KS == 1) {
        // gt s w_c(x, y, z): the trilinear weights with gt s folded into the y-z products; corners c and
        // c + 1 (x = 0 and 1) are accumulated as one packed two-lane FMA
        const float a = gt * sxyz[0];
        const float x = sxyz[1], y = sxyz[2], z = sxyz[3];
        const float2 xw = make_float2(1.0f - x, x);
        const float2 ay = __fmul2_rn(make_float2(a, a), make_float2(1.0f - y, y));
        const float2 cz0 = __fmul2_rn(ay, make_float2(1.0f - z, 1.0f - z));
        const float2 cz1 = __fmul2_rn(ay, make_float2(z, z));
        float2 r;
        r = __ffma2_rn(xw, make_float2(cz0.x, cz0.x), make_float2(acc[0], acc[1])); acc[0] = r.x; acc[1] = r.y;
        r = __ffma2_rn(xw, make_float2(cz0.y, cz0.y), make_float2(acc[2], acc[3])); acc[2] = r.x; acc[3] = r.y;
        r = __ffma2_rn(xw, make_float2(cz1.x, cz1.x), make_float2(acc[4], acc[5])); acc[4] = r.x; acc[5] = r.y;
        r = __ffma2_rn(xw, make_float2(cz1.y, cz1.y), make_float2(acc[6], acc[7])); acc[6] = r.x; acc[7] = r.y;
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = fmaf(gt, dtd[c], acc[c]);
    }
}

// Composites one segment (with the stop test when STOP); with GRAD also adds
// this segment's gradient into acc[0..10] (8 densities, 3 colour channels).
// RF (backward only): the residual form.  The gradient of tau_k only needs the upstream-weighted
// sums, dL/dtau_k = T_{k+1} s_k - (K - R_k) + dL/dA T_end with s_k = dL/dC . c_k + dL/dD mid_k
// (+ dL/dN . n_k), K the same sum over the final images and R_k = sum_{j <= k} w_j s_j; so the lane
// carries the one scalar R instead of the prefix colour, depth (and normal).
template <bool GRAD, bool STOP, int KS, bool NRM, bool WEX = false, bool RF = false>
__device__ __forceinline__ void add_segment(Pix<NRM>& ps, const Bwd<NRM>& bw, const BatchParams& bp, float4 da, float4 db,
                                            float4 col, float4 nv, const float* rel, const float* d, float t0,
                                            float t1, float* acc, uint32_t r = 0, ExportSink* ex = nullptr) {
    float dtd[8], sxyz[4];
    const float tau = seg_tau<GRAD, KS>(da, db, col.w, rel, d, t0, t1, bp.K, bp.inv_k, bp.act_thr, dtd, sxyz);
    if constexpr (RF) {
        // (without GRAD: an actor's partial in the backward, R only)
        const float e = exp_neg(tau);
        const float w = ps.T * (1.0f - e);
        const float mid = 0.5f * (t0 + t1);
        float s = fmaf(bw.g0, col.x, fmaf(bw.g1, col.y, fmaf(bw.g2, col.z, bw.gD * mid)));
        if constexpr (NRM) s = fmaf(bw.gN0, nv.x, fmaf(bw.gN1, nv.y, fmaf(bw.gN2, nv.z, s)));
        ps.R = fmaf(w, s, ps.R);
        ps.T = ps.T * e;
        ps.n += 1;
        if constexpr (GRAD) {
            const float gt = fmaf(ps.T, s, bw.base + ps.R);
            seg_density_grad<KS>(gt, dtd, sxyz, acc);
            acc[8] = fmaf(bw.g0, w, acc[8]);
            acc[9] = fmaf(bw.g1, w, acc[9]);
            acc[10] = fmaf(bw.g2, w, acc[10]);
            if constexpr (NRM) {
                acc[11] = fmaf(bw.gN0, w, acc[11]);
                acc[12] = fmaf(bw.gN1, w, acc[12]);
                acc[13] = fmaf(bw.gN2, w, acc[13]);
            }
        }
        if (STOP && ps.T < bp.eps_stop) ps.stop();
        return;
    }
    const float w = composite_step<NRM>(ps, tau, col, nv, t0, t1);
    if constexpr (WEX) {
        if (ex->n < ex->lim) {
            ex->vid[ex->base + ex->n] = (uint32_t)((int64_t)ex->sorted_g[r] - ex->voff);
            ex->w[ex->base + ex->n] = w;
        }
        ex->n += 1;
    }
    if (GRAD) {
        const float mid = 0.5f * (t0 + t1);
        const float Tn = ps.T;
        float gt = bw.gA * bw.Tend;
        gt = fmaf(bw.g0, fmaf(Tn, col.x, -(bw.Cf0 - ps.C0)), gt);
        gt = fmaf(bw.g1, fmaf(Tn, col.y, -(bw.Cf1 - ps.C1)), gt);
        gt = fmaf(bw.g2, fmaf(Tn, col.z, -(bw.Cf2 - ps.C2)), gt);
        gt = fmaf(bw.gD, fmaf(Tn, mid, -(bw.Df - ps.D)), gt);
        if constexpr (NRM) {
            gt = fmaf(bw.gN0, fmaf(Tn, nv.x, -(bw.Nf0 - ps.N0)), gt);
            gt = fmaf(bw.gN1, fmaf(Tn, nv.y, -(bw.Nf1 - ps.N1)), gt);
            gt = fmaf(bw.gN2, fmaf(Tn, nv.z, -(bw.Nf2 - ps.N2)), gt);
            acc[11] = fmaf(bw.gN0, w, acc[11]);
            acc[12] = fmaf(bw.gN1, w, acc[12]);
            acc[13] = fmaf(bw.gN2, w, acc[13]);
        }
        seg_density_grad<KS>(gt, dtd, sxyz, acc);
        acc[8] = fmaf(bw.g0, w, acc[8]);
        acc[9] = fmaf(bw.g1, w, acc[9]);
        acc[10] = fmaf(bw.g2, w, acc[10]);
    }
    if (STOP && ps.T < bp.eps_stop) ps.stop();
}

// One backward step in residual form with one sample, for a lane that meets the record at most once
// (a plain tile, or one actor interval): [u0, u1] is the lane's segment, the empty segment [0, 0] for a
// lane that misses or has finished (zero optical depth, weight and gradient, state unchanged).  The
// record's gradient values (8 densities, 3 colour, + 3 normal) are written into acc, not added, so the
// caller clears nothing and the warp runs it without branches once any lane hits.  (The stop rule is tested for
// the misses too, which eps_stop above 1 would stop: one_sample has those.)
template <bool NRM>
__device__ __forceinline__ void bwd_single_step(Pix<NRM>& ps, const Bwd<NRM>& bw, const BatchParams& bp, float4 g,
                                                float4 da, float4 dd, float4 col, float4 nv, const float* d, float u0,
                                                float u1, bool hit, float* acc) {
    const float rel[3] = {g.x, g.y, g.z};
    float sxyz[4];
    const float tau = seg_tau<true, 1>(da, dd, col.w, rel, d, u0, u1, bp.K, bp.inv_k, bp.act_thr, nullptr, sxyz);
    const float e = exp_neg(tau);
    const float w = ps.T * (1.0f - e);
    const float mid = 0.5f * (u0 + u1);
    float sg = fmaf(bw.g0, col.x, fmaf(bw.g1, col.y, fmaf(bw.g2, col.z, bw.gD * mid)));
    if constexpr (NRM) sg = fmaf(bw.gN0, nv.x, fmaf(bw.gN1, nv.y, fmaf(bw.gN2, nv.z, sg)));
    ps.R = fmaf(w, sg, ps.R);
    ps.T = ps.T * e;
    ps.n += hit ? 1u : 0u;
    const float gt = fmaf(ps.T, sg, bw.base + ps.R);
    const float a = gt * sxyz[0];
    const float x = sxyz[1], y = sxyz[2], z = sxyz[3];
    const float2 xw = make_float2(1.0f - x, x);
    const float2 ay = __fmul2_rn(make_float2(a, a), make_float2(1.0f - y, y));
    const float2 cz0 = __fmul2_rn(ay, make_float2(1.0f - z, 1.0f - z));
    const float2 cz1 = __fmul2_rn(ay, make_float2(z, z));
    float2 r;
    r = __fmul2_rn(xw, make_float2(cz0.x, cz0.x));
    acc[0] = r.x;
    acc[1] = r.y;
    r = __fmul2_rn(xw, make_float2(cz0.y, cz0.y));
    acc[2] = r.x;
    acc[3] = r.y;
    r = __fmul2_rn(xw, make_float2(cz1.x, cz1.x));
    acc[4] = r.x;
    acc[5] = r.y;
    r = __fmul2_rn(xw, make_float2(cz1.y, cz1.y));
    acc[6] = r.x;
    acc[7] = r.y;
    acc[8] = bw.g0 * w;
    acc[9] = bw.g1 * w;
    acc[10] = bw.g2 * w;
    if constexpr (NRM) {
        acc[NRM ? 11 : 0] = bw.gN0 * w;
        acc[NRM ? 12 : 0] = bw.gN1 * w;
        acc[NRM ? 13 : 0] = bw.gN2 * w;
    }
    if (ps.T < bp.eps_stop) ps.stop();
}

// Sum of acc[0..NV-1] over the warp, transposed.  Each butterfly level (lane distance 16, 8, 4, 2,
// 1) splits the values the lane still holds into a first half (kept by the lanes without that
// distance's bit) and the rest (kept by the others), exchanging the half it gives up: NV = 11 takes
// 6 + 3 + 2 + 1 + 1 = 13 shuffles (14 values: 15).  Afterwards every value's total sits in exactly
// one lane, which adds it to the record's gradient slot.
template <int N, int D>
__device__ __forceinline__ void fold_level(float* v, int lane, int& idx, int& nreal) {
    if constexpr (D >= 1) {
        constexpr int H = (N + 1) / 2;
        const bool up = lane & D;
        float own[H + 1], got[H + 1];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const float lo = v[i];
            const float hi = (H + i < N) ? v[H + i] : 0.0f;
            own[i] = up ? hi : lo;
            got[i] = __shfl_xor_sync(0xffffffffu, up ? lo : hi, D);
        }
        own[H] = got[H] = 0.0f;
#pragma unroll
        for (int i = 0; i < H; i += 2) {  // packed two-lane additions
            const float2 s = __fadd2_rn(make_float2(own[i], own[i + 1]), make_float2(got[i], got[i + 1]));
            v[i] = s.x;
            if (i + 1 < H) v[i + 1] = s.y;
        }
        idx += up ? H : 0;
        nreal = up ? max(nreal - H, 0) : min(nreal, H);
        fold_level<H, D / 2>(v, lane, idx, nreal);
    }
}

template <int NV>
__device__ __forceinline__ void warp_reduce_add(const float* acc, float* gp) {
    const int lane = threadIdx.x & 31;
    float v[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) v[c] = acc[c];
    int idx = 0, nreal = NV;
    fold_level<NV, 16>(v, lane, idx, nreal);
    if (nreal > 0 && v[0] != 0.0f) atomicAdd(gp + idx, v[0]);
}

// Record of pair q.  Every pair's record is below n_vis unless a sort's bounded wait ran out (the
// call is then reported as timed out); the clamp keeps the reads and gradient atomics in range.
__device__ __forceinline__ uint32_t rec_index(const BatchParams& bp, const uint32_t* __restrict__ pval, uint32_t q) {
    return min(__ldg(pval + q), (uint32_t)(bp.n_vis - 1));
}

// Pixels of the 8x4 block (bx, by) of a tile that a pair's pixel rectangle covers, as lane bits (lane
// l renders pixel (l & 7, l >> 3) of the block).  rc: the rectangle within the tile, x0 | x1 << 4 |
// y0 << 8 | y1 << 12.
__device__ __forceinline__ uint32_t block_pixels(uint32_t rc, int bx, int by) {
    const int x0 = (int)(rc & 15u) - 8 * bx, x1 = (int)((rc >> 4) & 15u) - 8 * bx;
    const int y0 = (int)((rc >> 8) & 15u) - 4 * by, y1 = (int)((rc >> 12) & 15u) - 4 * by;
    const uint32_t xm = (0xffu << max(x0, 0)) & (0xffu >> max(7 - x1, 0));
    const uint32_t ym = (0xfu << max(y0, 0)) & (0xfu >> max(3 - y1, 0));
    return (xm & 0xffu) * (((ym & 0xfu) * 0x00204081u) & 0x01010101u);
}

// One lane's gradient values of record r, added with 16-byte vector atomics (the rows are 16-byte
// aligned and padded to a multiple of four floats).
template <bool NRM>
__device__ __forceinline__ void lane_add(float* grad_rec, uint32_t r, const float* acc) {
    constexpr int NV = GradLayout<NRM>::NV;
    float4* gp = reinterpret_cast<float4*>(grad_rec + (size_t)r * GradLayout<NRM>::STRIDE);
#pragma unroll
    for (int c = 0; c < NV; c += 4)
        atomicAdd(gp + c / 4, make_float4(acc[c], acc[c + 1], c + 2 < NV ? acc[c + 2] : 0.0f, c + 3 < NV ? acc[c + 3] : 0.0f));
}

// Transpose of the 32x32 bit matrix whose row l is lane l's x: afterwards bit j of lane l is bit l of
// what lane j held.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 16; k >= 1; k >>= 1) {
        const uint32_t m = k == 16 ? 0x0000ffffu : k == 8 ? 0x00ff00ffu : k == 4 ? 0x0f0f0f0fu : k == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, k);
        x = (lane & k) ? (x & ~m) | ((y >> k) & m) : (x & m) | ((y << k) & ~m);
    }
    return x;
}

// 16-byte asynchronous global -> shared copy (L2 only), and its group fences
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_one() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// ---------------------------------------------------------------------------
// per-pixel set-up and results, shared by the plain and the actor kernels
// ---------------------------------------------------------------------------

__device__ __forceinline__ int view_of(const BatchParams& bp, int gtile) {
    int lo = 0, hi = bp.n_view - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (bp.tile_base[mid] <= gtile)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// the tile's slice of the pair list, kept inside [0, n_pairs] whatever the range words hold (they
// are only inconsistent after a sort wait that timed out, which the call then reports)
__device__ __forceinline__ uint2 tile_slice(const CompositeArgs& A, int gtile) {
    uint2 rg = __ldg(A.tile_range + gtile);
    rg.y = (uint32_t)min((int64_t)rg.y, A.bp.n_pairs);
    rg.x = min(rg.x, rg.y);
    return rg;
}

// unit ray of pixel (u, v) in the camera frame
__device__ __forceinline__ void pixel_ray(const ViewParams& fp, int u, int v, float* dc) {
    const float x = ((float)u + 0.5f - fp.cx) / fp.fx;
    const float y = ((float)v + 0.5f - fp.cy) / fp.fy;
    const float in = rsqrtf(fmaf(x, x, fmaf(y, y, 1.0f)));
    dc[0] = x * in;
    dc[1] = y * in;
    dc[2] = in;
}

template <bool NRM>
__device__ __forceinline__ void init_pix(Pix<NRM>& p, float end) {
    p.C0 = p.C1 = p.C2 = p.D = 0.0f;
    if constexpr (NRM) p.N0 = p.N1 = p.N2 = 0.0f;
    p.T = p.Tp = 1.0f;
    p.R = 0.0f;
    p.n = 0;
    p.tests = 0;
    p.boxes = 0;
    p.end = end;
}

template <bool BWD, bool NRM>
__device__ __forceinline__ void load_bwd(Bwd<NRM>& bw, const CompositeArgs& A, const ViewParams& fp, int64_t lpix,
                                         int64_t pix, bool valid) {
    if (BWD && valid) {
        bw.g0 = A.g_rgb ? A.g_rgb[pix * 3 + 0] : 0.0f;
        bw.g1 = A.g_rgb ? A.g_rgb[pix * 3 + 1] : 0.0f;
        bw.g2 = A.g_rgb ? A.g_rgb[pix * 3 + 2] : 0.0f;
        bw.gD = A.g_depth ? A.g_depth[pix] : 0.0f;
        bw.gA = A.g_alpha ? A.g_alpha[pix] : 0.0f;
        bw.Cf0 = fp.rgb[lpix * 3 + 0];
        bw.Cf1 = fp.rgb[lpix * 3 + 1];
        bw.Cf2 = fp.rgb[lpix * 3 + 2];
        bw.Df = fp.depth[lpix];
        bw.Tend = A.t_final[pix];
    } else {
        bw.g0 = bw.g1 = bw.g2 = bw.gD = bw.gA = 0.0f;
        bw.Cf0 = bw.Cf1 = bw.Cf2 = bw.Df = bw.Tend = 0.0f;
    }
    if constexpr (NRM) {
        bw.gN0 = bw.gN1 = bw.gN2 = bw.Nf0 = bw.Nf1 = bw.Nf2 = 0.0f;
        if (BWD && valid) {
            bw.gN0 = A.g_normal[pix * 3 + 0];
            bw.gN1 = A.g_normal[pix * 3 + 1];
            bw.gN2 = A.g_normal[pix * 3 + 2];
            bw.Nf0 = fp.normal[lpix * 3 + 0];
            bw.Nf1 = fp.normal[lpix * 3 + 1];
            bw.Nf2 = fp.normal[lpix * 3 + 2];
        }
    }
    bw.base = bw.gA * bw.Tend - fmaf(bw.g0, bw.Cf0, fmaf(bw.g1, bw.Cf1, fmaf(bw.g2, bw.Cf2, bw.gD * bw.Df)));
    if constexpr (NRM) bw.base -= fmaf(bw.gN0, bw.Nf0, fmaf(bw.gN1, bw.Nf1, bw.gN2 * bw.Nf2));
}

__device__ __forceinline__ void init_sink(ExportSink& ex, const CompositeArgs& A, int view, int64_t pix, bool valid) {
    ex.vid = A.ex_vid;
    ex.w = A.ex_w;
    ex.sorted_g = A.bp.sorted_g;
    ex.voff = (int64_t)view * A.bp.n_vox;
    ex.base = valid ? A.ex_off[pix] : 0;
    ex.n = 0;
    ex.lim = valid ? (uint32_t)(A.ex_off[pix + 1] - ex.base) : 0u;
}

template <bool NRM>
__device__ __forceinline__ void store_pix(const Pix<NRM>& ps, const CompositeArgs& A, const ViewParams& fp,
                                          int64_t lpix, int64_t pix) {
    fp.rgb[lpix * 3 + 0] = ps.C0;
    fp.rgb[lpix * 3 + 1] = ps.C1;
    fp.rgb[lpix * 3 + 2] = ps.C2;
    fp.depth[lpix] = ps.D;
    fp.alpha[lpix] = 1.0f - ps.T;
    A.n_seg[pix] = ps.n;
    A.t_final[pix] = ps.T;
    if constexpr (NRM) {
        fp.normal[lpix * 3 + 0] = ps.N0;
        fp.normal[lpix * 3 + 1] = ps.N1;
        fp.normal[lpix * 3 + 2] = ps.N2;
    }
}

// adds the warp's tests, box tests and segments to the call's work counters
__device__ __forceinline__ void add_work(unsigned long long* work, uint32_t tests, uint32_t boxes, uint32_t segs) {
    unsigned long long t = tests, b = boxes, n = segs;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        t += __shfl_down_sync(0xffffffffu, t, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
        n += __shfl_down_sync(0xffffffffu, n, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(work + 0, t);
        atomicAdd(work + 1, b);
        atomicAdd(work + 2, n);
    }
}

}  // namespace

// Whether a pass takes the variants for one sample per segment.  The backward's do not test for a hit before the stop
// rule, which a ray at T = 1 meets without one where eps_stop is above 1; the general ones do.  (The test in the
// step itself: backward of the 1080p frame some 20 us longer.)
inline bool one_sample(const BatchParams& bp, bool bwd) { return bp.K == 1 && !(bwd && bp.eps_stop > 1.0f); }

// The actor tiles' part of a compositing pass (dv_composite_act.cu): the n_tiles tiles of A.tile_order,
// the pass being the forward, the backward (bwd) or the weights export (wex).  `large`: tiles that 5 or
// more actor boxes cover.
void launch_composite_act(CompositeArgs A, int n_tiles, bool bwd, bool wex, bool normals, bool large, cudaStream_t s);

}  // namespace dv
