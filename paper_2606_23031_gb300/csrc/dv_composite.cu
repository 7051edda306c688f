// Front-to-back compositing over each ray's voxel segments (forward) and its
// replay with gradients (backward), plus the SH-colour backward (Sec. 3.4, Alg. 1).
//
//  * The tile's pair list is grouped by octree and, inside an octree, sorted
//    front to back for every ray of the camera (depth-order key, see
//    dv_project.cu).
//  * Tiles that no actor clip box covers are composited here: each CTA renders
//    half of a 16x16 tile (16x8 pixels, 4 warps of 8x4 pixels), one thread per
//    pixel, tiles taken heaviest first; the list streams through a two-slot
//    shared-memory ring (cp.async, one batch ahead).
//  * In the other tiles each pixel splits its ray into background and actor
//    intervals with the actor clip boxes (slab test in each actor's frame,
//    reached through the inverse pose; the box entered first owns any
//    overlap).  dv_composite_act.cu has them, in three phases:
//     1. every interval's segments into a partial (C_A, D_A, T_A) starting from
//        T = 1, nearest first, unless the partials of the ray's earlier intervals
//        already hide it.
//     2. the background sub-list.  A background hit that reaches past the next
//        actor's entry composites its part in front of the box, then applies
//        that actor's partial with the running transmittance (C += T C_A,
//        D += T D_A, T *= T_A), then continues behind the box.  If T T_A < eps_stop
//        the ray stops inside the actor: at the partial's last segment (the whole
//        partial applies) if T times the transmittance before it is not below
//        eps_stop; else the state is recorded for a replay.
//     3. replays walk that actor's sub-list from the recorded state with the
//        exact stop rule.
//    Since T only decreases along the ray, applying a whole partial is exact
//    unless the stop falls inside it, which is exactly when T T_A < eps_stop.
//    (With negative densities, which the identity activation admits, T rises: a
//    ray that enters an interval with T above 1 may walk it instead.)
//  * Per segment: trilinear interpolation of the raw corner densities at K
//    midpoints, exponential-linear activation, tau = l/K sum sigma,
//    alpha = 1 - exp(-tau), C += T alpha c, D += T alpha (t0+t1)/2,
//    T *= 1 - alpha, stop once T < eps_stop.
//  * The backward runs the same phases (identical arithmetic, so the same
//    stops).  With w_k = T_k alpha_k it uses
//    dC/dtau_k = T_{k+1} c_k - sum_{j>k} w_j c_j, the suffix sum being
//    C_final - (prefix through k), so it needs no division by (1 - alpha) and
//    no reverse traversal.  Phase 2 records, for every actor interval reached,
//    the prefix state at its entry; phase 3 then replays every reached actor
//    interval with gradients from that state.
#include "dv_composite.cuh"

namespace dv {

namespace {

// The backward takes a chunk lane by lane where its records cover at most this many of the block's 32 pixels on
// average (8M-leaf six-camera frame / 1080p frame: 0: 2,830 / 209 us, 8: 2,728 / 210, 12: 2,522 / 214, 16: 2,512 /
// 215, any: 2,540 / 253).
constexpr int LANE_PIX = 14;
// Resident CTAs per SM: the forward without normals fits 56 registers (9 CTAs: 1,481 -> 1,455 us on the 8M-leaf
// frame); the others need 64, the backward with normals and several samples 72 (two 1883x1229 views of 168k leaves,
// K = 2: step 1,433 -> 1,393 us).
constexpr int plain_ctas(bool bwd, int ks, bool nrm, bool wex) {
    return !bwd && ks == 1 && !nrm && !wex ? 9 : bwd && ks == 0 && nrm ? 7 : 8;
}

// Tiles that no actor box covers (most of a frame): every ray is background only, so the tile's list
// is the background's.
// BWD: replay with gradients.  WEX: replay that writes every composited segment's (voxel, weight) into
// the pixel's slots of the weights export (no outputs, no gradients).
template <bool BWD, int KS, bool NRM, bool WEX>
__global__ void __launch_bounds__(CT_THREADS, plain_ctas(BWD, KS, NRM, WEX))
    k_composite(const __grid_constant__ CompositeArgs A) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ float4 s_rec[2][CT_THREADS][5];  // rows of 80 bytes: lanes can read different records at once
    __shared__ float4 s_nv[NRM ? 2 : 1][NRM ? CT_THREADS : 1];  // voxel normals of the staged records
    __shared__ uint32_t s_r[2][CT_THREADS];
    __shared__ uint16_t s_m[2][CT_THREADS];  // pixel rectangles of the staged pairs within the tile
    const BatchParams& bp = A.bp;
    const uint32_t* __restrict__ pval = A.pval;
    const uint16_t* __restrict__ prect = A.prect;
    const VoxRec* __restrict__ rec = A.rec;

    const int tid = threadIdx.x;
    const int gtile = (int)__ldg(A.tile_order + (blockIdx.x >> 1));
    const int half = blockIdx.x & 1;
    const int view = view_of(bp, gtile);
    const ViewParams& fp = bp.views[view];
    const OctParams* __restrict__ vo = bp.octs + view * bp.n_oct;
    const int tiles_x = fp.tiles_x;
    const float t_near = fp.near_, t_far = fp.far_;
    const int tile = gtile - bp.tile_base[view];
    const int tx = tile % tiles_x, ty = tile / tiles_x;
    const uint2 rg = tile_slice(A, gtile);
    const int lane = tid & 31, warp = tid >> 5;
    const int bx = warp & 1, by = half * 2 + (warp >> 1);  // this warp's 8x4 block of the tile
    const int u = tx * DV_TILE + bx * 8 + (lane & 7);
    const int v = ty * DV_TILE + by * 4 + (lane >> 3);
    const bool valid = u < fp.W && v < fp.H;
    const int64_t lpix = (int64_t)v * fp.W + u;    // pixel within the view's own images
    const int64_t pix = fp.pix_base + lpix;        // pixel within the call's per-pixel arrays
    float db_[3];
    {
        float dc[3];
        pixel_ray(fp, u, v, dc);
        rotate(vo[0].A, dc, db_);
    }
    const InvDir ib = inv_dir(db_);
    Pix<NRM> ps;
    init_pix<NRM>(ps, valid ? t_far : -1.0f);
    ExportSink ex;
    if constexpr (WEX) init_sink(ex, A, view, pix, valid);
    Bwd<NRM> bw;
    load_bwd<BWD, NRM>(bw, A, fp, lpix, pix, valid);
    // The list is grouped by octree in record order.  Actor voxels can lie outside their box and reach
    // a tile that it does not; such records are at the list's end, at or behind the second octree's
    // first record, and are left out.
    uint32_t q_end = rg.y;
    if (bp.n_oct > 1 && rg.y > rg.x) {
        const uint32_t second = __ldg(A.vis_start + view * bp.n_oct + 1);
        if (rec_index(bp, pval, rg.y - 1) >= second) {
            uint32_t lo = rg.x;
            while (lo < q_end) {
                const uint32_t mid = lo + ((q_end - lo) >> 1);
                if (rec_index(bp, pval, mid) < second)
                    lo = mid + 1;
                else
                    q_end = mid;
            }
        }
    }
    constexpr int NV = GradLayout<NRM>::NV;
    constexpr int GS = GradLayout<NRM>::STRIDE;

    // voxel normal of staged record j (zero without normals)
    auto staged_nv = [&](int slot, uint32_t j) {
        return NRM ? s_nv[NRM ? slot : 0][NRM ? j : 0] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    };
    // the lane's segment of a record: entry and exit, true if it has any length
    auto clip = [&](float4 g, float& t_in, float& t_out) {
        slab_cube(ib, g, t_in, t_out);
        t_in = fmaxf(t_in, t_near);
        t_out = fminf(t_out, ps.end);
        return t_out > t_in;
    };
    // composites the lane's segment of staged record j (backward and export), with its gradient values in acc.
    // A lane meets a record at most once, so with one sample a warp that visits a record together runs the same
    // arithmetic without branches, a lane that misses (hit false) on the empty segment [0, 0], whose optical
    // depth, weight and gradient are exactly zero.
    auto segment = [&](int slot, uint32_t j, float4 g, float t_in, float t_out, bool hit, float* acc) {
        if constexpr (BWD && KS == 1) {
            bwd_single_step<NRM>(ps, bw, bp, g, s_rec[slot][j][1], s_rec[slot][j][2], s_rec[slot][j][3],
                                 staged_nv(slot, j), db_, hit ? t_in : 0.0f, hit ? t_out : 0.0f, hit, acc);
        } else {
            if constexpr (BWD) {
#pragma unroll
                for (int i = 0; i < NV; ++i) acc[i] = 0.0f;
            }
            const float rel[3] = {g.x, g.y, g.z};
            if (hit)
                add_segment<BWD, true, KS, NRM, WEX, BWD>(ps, bw, bp, s_rec[slot][j][1], s_rec[slot][j][2],
                                                          s_rec[slot][j][3], staged_nv(slot, j), rel, db_, t_in, t_out,
                                                          acc, s_r[slot][j], &ex);
        }
    };
    // 32 records of the batch, from c0; pm: the pixels of this warp's 8x4 block that the lane's record may touch.
    // True once the warp is done.  The pixel masks, transposed, are a list of records per lane, and every lane
    // steps through its own, so a record costs only the pixels it covers a step, not the whole warp (8M-leaf
    // six-camera frame: 33 records visited per pixel for 10 met; plain forward 1,717 ->
    // 1,480 us).  The backward does so where the records cover few pixels (at most LANE_PIX on average, the
    // longest lane list at most 1 / LANE_GAIN of the records), each lane adding its own gradient values with
    // vector atomics; elsewhere the warp visits the records together and sums their values first.
    auto chunk = [&](int slot, uint32_t c0, uint32_t pm) -> bool {
        unsigned m = __ballot_sync(0xffffffffu, pm != 0u);
        if (!m) return false;
        if (__all_sync(0xffffffffu, ps.done())) return true;
        const int n = __popc(m);
        bool lanes = true;
        if constexpr (BWD) lanes = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(pm)) <= n * LANE_PIX;
        uint32_t mine = 0;
        if (lanes) {
            mine = warp_transpose(pm);
            if (ps.done()) mine = 0u;
            if constexpr (BWD) lanes = (int)__reduce_max_sync(0xffffffffu, (unsigned)__popc(mine)) * LANE_GAIN <= n;
        }
        if (lanes) {
            if constexpr (!BWD && !WEX) ps.tests += (uint32_t)__popc(mine);
            while (mine) {
                const uint32_t j0 = c0 + (uint32_t)(__ffs(mine) - 1);
                mine &= mine - 1;
                if constexpr (!BWD && !WEX) {
                    // forward, two records at once: both slab tests, both optical depths, then compositing in
                    // list order with the stop rule
                    const bool two = mine != 0u;
                    const uint32_t j1 = two ? c0 + (uint32_t)(__ffs(mine) - 1) : j0;
                    mine &= mine - 1;
                    const float4 g0 = s_rec[slot][j0][0], g1 = s_rec[slot][j1][0];
                    float a0, b0, a1, b1;
                    const bool h0 = clip(g0, a0, b0), h1 = clip(g1, a1, b1) && two;
                    const float4 da0 = s_rec[slot][j0][1], dd0 = s_rec[slot][j0][2], col0 = s_rec[slot][j0][3];
                    const float4 da1 = s_rec[slot][j1][1], dd1 = s_rec[slot][j1][2], col1 = s_rec[slot][j1][3];
                    const float r0[3] = {g0.x, g0.y, g0.z}, r1[3] = {g1.x, g1.y, g1.z};
                    const float tau0 = seg_tau<false, KS>(da0, dd0, col0.w, r0, db_, a0, b0, bp.K, bp.inv_k, bp.act_thr,
                                                          nullptr, nullptr);
                    const float tau1 = seg_tau<false, KS>(da1, dd1, col1.w, r1, db_, a1, b1, bp.K, bp.inv_k, bp.act_thr,
                                                          nullptr, nullptr);
                    if (h0) composite_tau<NRM>(ps, tau0, col0, staged_nv(slot, j0), a0, b0, bp.eps_stop);
                    if (h1 && !ps.done()) composite_tau<NRM>(ps, tau1, col1, staged_nv(slot, j1), a1, b1, bp.eps_stop);
                    if (ps.done()) {
                        ps.tests -= (uint32_t)__popc(mine);
                        mine = 0u;
                    }
                } else {
                    const float4 g = s_rec[slot][j0][0];
                    float t_in, t_out;
                    if (clip(g, t_in, t_out)) {
                        float acc[NV];
                        segment(slot, j0, g, t_in, t_out, true, acc);
                        if constexpr (BWD) lane_add<NRM>(A.grad_rec, s_r[slot][j0], acc);
                    }
                    if (ps.done()) mine = 0u;
                }
            }
            __syncwarp();
        } else if constexpr (BWD) {
            while (m) {
                if (__all_sync(0xffffffffu, ps.done())) return true;
                const uint32_t j = c0 + (uint32_t)(__ffs(m) - 1);
                m &= m - 1;
                const float4 g = s_rec[slot][j][0];
                float t_in, t_out;
                const bool hit = clip(g, t_in, t_out);
                if (!__any_sync(0xffffffffu, hit)) continue;
                float acc[NV];
                segment(slot, j, g, t_in, t_out, hit, acc);
                warp_reduce_add<NV>(acc, A.grad_rec + (size_t)s_r[slot][j] * GS);
            }
        }
        return __all_sync(0xffffffffu, ps.done());
    };

    // The list streams through a two-slot shared-memory ring, CT_THREADS records per batch (cp.async, one
    // batch ahead).  The batch loop, its barriers and its early exit are CTA-uniform.
    const uint32_t n_batch = (q_end - rg.x + CT_THREADS - 1) / CT_THREADS;
    uint32_t r_ahead = 0, m_ahead = 0;
    auto fetch = [&](uint32_t bi) {
        const uint32_t q = rg.x + bi * CT_THREADS + tid;
        if (q < q_end) {
            r_ahead = rec_index(bp, pval, q);
            m_ahead = __ldg(prect + q);
        }
    };
    auto stage = [&](int slot, uint32_t bi) {
        if (rg.x + bi * CT_THREADS + tid < q_end) {
            const float4* R = rec[r_ahead].v;
#pragma unroll
            for (int k = 0; k < 4; ++k) cp_async16(&s_rec[slot][tid][k], R + k);
            if (NRM) cp_async16(&s_nv[NRM ? slot : 0][NRM ? tid : 0], bp.nrm + r_ahead);
            s_r[slot][tid] = r_ahead;
            s_m[slot][tid] = (uint16_t)m_ahead;
        }
        cp_async_commit();
    };
    if (n_batch > 0) {
        fetch(0);
        stage(0, 0);
        fetch(1);
    }
    bool fin = false;
    for (uint32_t bi = 0; bi < n_batch; ++bi) {
        const int slot = bi & 1;
        stage(slot ^ 1, bi + 1);
        fetch(bi + 2);
        cp_async_wait_one();  // batch bi has landed (only batch bi+1 may still be in flight)
        __syncthreads();
        const uint32_t cnt = min((uint32_t)CT_THREADS, q_end - rg.x - bi * CT_THREADS);
        for (uint32_t c0 = 0; c0 < cnt && !fin; c0 += 32) {
            const uint32_t jl = c0 + lane;
            fin = chunk(slot, c0, jl < cnt ? block_pixels(s_m[slot][jl], bx, by) : 0u);
        }
        // every warp is done with this slot before batch bi+2 is copied into it
        if (__syncthreads_or(!fin) == 0) break;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");  // no copy outlives the list (early exit)

    if constexpr (!BWD && !WEX) {
        if (A.work) add_work(A.work, ps.tests, ps.boxes, ps.n);
        if (valid) store_pix<NRM>(ps, A, fp, lpix, pix);
    }
}

// ---------------------------------------------------------------------------
// SH colour backward + scatter of the per-record gradients to the caller's arrays
// ---------------------------------------------------------------------------

__device__ __forceinline__ void sh_basis_f(int deg, float x, float y, float z, float* b) {
    // same basis as the records kernel (real SH, degree <= 3)
    b[0] = 0.28209479177387814f;
    if (deg < 1) return;
    b[1] = -0.48860251190291992f * y;
    b[2] = 0.48860251190291992f * z;
    b[3] = -0.48860251190291992f * x;
    if (deg < 2) return;
    const float xx = x * x, yy = y * y, zz = z * z;
    b[4] = 1.0925484305920792f * x * y;
    b[5] = -1.0925484305920792f * y * z;
    b[6] = 0.31539156525252005f * (2.0f * zz - xx - yy);
    b[7] = -1.0925484305920792f * x * z;
    b[8] = 0.54627421529603959f * (xx - yy);
    if (deg < 3) return;
    b[9] = -0.59004358992664352f * y * (3.0f * xx - yy);
    b[10] = 2.8906114426405538f * x * y * z;
    b[11] = -0.45704579946446572f * y * (4.0f * zz - xx - yy);
    b[12] = 0.3731763325901154f * z * (2.0f * zz - 3.0f * xx - 3.0f * yy);
    b[13] = -0.45704579946446572f * x * (4.0f * zz - xx - yy);
    b[14] = 1.4453057213202769f * z * (xx - yy);
    b[15] = -0.59004358992664352f * x * (xx - 3.0f * yy);
}

struct ShBwdParams {
    BatchParams bp;
    float* d_dens[DV_MAX_OCTREES];
    float* d_sh[DV_MAX_OCTREES];
};

template <bool NRM>
__global__ void __launch_bounds__(256) k_sh_bwd(const __grid_constant__ ShBwdParams sp,
                                                const uint32_t* __restrict__ sorted_g, int64_t n_vis,
                                                const VoxRec* __restrict__ rec, const float* __restrict__ grad_rec) {
    pdl_wait();
    pdl_launch_dependents();
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_vis) return;
    const BatchParams& bp = sp.bp;
    const uint32_t gidx = sorted_g[r];
    const int view = (int)(gidx / (uint64_t)bp.n_vox);
    const int64_t gv = (int64_t)gidx - (int64_t)view * bp.n_vox;
    int lo = 0, hi = bp.n_oct - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (bp.vox_offset[mid] <= gv)
            lo = mid;
        else
            hi = mid - 1;
    }
    const OctParams& P = bp.octs[view * bp.n_oct + lo];
    const int64_t v = gv - bp.vox_offset[lo];
    const float* gr = grad_rec + (size_t)r * GradLayout<NRM>::STRIDE;
    float* d_dens = sp.d_dens[lo];
    float* d_sh = sp.d_sh[lo];
    // several views may touch the same voxel: accumulate with atomics (16-byte vector
    // atomics where the caller's rows are 16-byte aligned)
    float4 g03 = *reinterpret_cast<const float4*>(gr), g47 = *reinterpret_cast<const float4*>(gr + 4);
    if (NRM) {
        // through the voxel normal n_w = R n_l, n_l = -g / |g| with g the corner-difference
        // gradient (as in the records kernel): dL/dg = -(dL/dn_l - n_l (n_l . dL/dn_l)) / |g|,
        // and each corner enters g_a with sign + on the high side of axis a, - on the low side
        const float dw0 = gr[11], dw1 = gr[12], dw2 = gr[13];
        if (d_dens && (dw0 != 0.0f || dw1 != 0.0f || dw2 != 0.0f)) {
            // the raw corner densities, as the records kernel used them for the voxel normal
            const float4* d4 = reinterpret_cast<const float4*>(P.dens + v * 8);
            const float4 da = __ldg(d4), db = __ldg(d4 + 1);
            const float gx = (da.y + da.w + db.y + db.w) - (da.x + da.z + db.x + db.z);
            const float gy = (da.z + da.w + db.z + db.w) - (da.x + da.y + db.x + db.y);
            const float gz = (db.x + db.y + db.z + db.w) - (da.x + da.y + da.z + da.w);
            const float g2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
            if (g2 > 0.0f) {
                const float ig = rsqrtf(g2);
                const float nl[3] = {-gx * ig, -gy * ig, -gz * ig};
                float dn[3];
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    dn[k] = fmaf(P.Rw[0 * 3 + k], dw0, fmaf(P.Rw[1 * 3 + k], dw1, P.Rw[2 * 3 + k] * dw2));
                const float nd = fmaf(nl[0], dn[0], fmaf(nl[1], dn[1], nl[2] * dn[2]));
                const float dgx = -(dn[0] - nl[0] * nd) * ig, dgy = -(dn[1] - nl[1] * nd) * ig,
                            dgz = -(dn[2] - nl[2] * nd) * ig;
                // corner c = (x, y, z) bits: + dg_a where bit a is set, - where clear
                g03.x += -dgx - dgy - dgz;
                g03.y += dgx - dgy - dgz;
                g03.z += -dgx + dgy - dgz;
                g03.w += dgx + dgy - dgz;
                g47.x += -dgx - dgy + dgz;
                g47.y += dgx - dgy + dgz;
                g47.z += -dgx + dgy + dgz;
                g47.w += dgx + dgy + dgz;
            }
        }
    }
    if (d_dens) {
        float* dd = d_dens + v * 8;
        if ((reinterpret_cast<uintptr_t>(dd) & 15) == 0) {
            if (g03.x != 0.0f || g03.y != 0.0f || g03.z != 0.0f || g03.w != 0.0f)
                atomicAdd(reinterpret_cast<float4*>(dd), g03);
            if (g47.x != 0.0f || g47.y != 0.0f || g47.z != 0.0f || g47.w != 0.0f)
                atomicAdd(reinterpret_cast<float4*>(dd) + 1, g47);
        } else {
            const float gd[8] = {g03.x, g03.y, g03.z, g03.w, g47.x, g47.y, g47.z, g47.w};
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (gd[c] != 0.0f) atomicAdd(dd + c, gd[c]);
        }
    }
    // colour channels clamped at zero in the forward (stored clamped in the record) pass no
    // gradient to the SH coefficients
    const float4 col = rec[r].v[3];
    const float m0 = col.x > 0.0f ? gr[8] : 0.0f, m1 = col.y > 0.0f ? gr[9] : 0.0f, m2 = col.z > 0.0f ? gr[10] : 0.0f;
    if (!d_sh || (m0 == 0.0f && m1 == 0.0f && m2 == 0.0f)) return;
    const float4 g = rec[r].v[0];  // (min - camera centre, size): same direction as the records kernel
    float gx = fmaf(0.5f, g.w, g.x);
    float gy = fmaf(0.5f, g.w, g.y);
    float gz = fmaf(0.5f, g.w, g.z);
    const float gl = sqrtf(gx * gx + gy * gy + gz * gz);
    const float ig = gl > 0.0f ? 1.0f / gl : 0.0f;
    gx *= ig;
    gy *= ig;
    gz *= ig;
    float b[16];
    sh_basis_f(P.sh_degree, gx, gy, gz, b);
    const int nsh = (P.sh_degree + 1) * (P.sh_degree + 1);
    float* ds = d_sh + v * nsh * 3;
    if ((nsh * 3) % 4 == 0 && (reinterpret_cast<uintptr_t>(ds) & 15) == 0) {
        // coefficient rows (q, channel) flattened: element e = 3 q + channel
        const float m[3] = {m0, m1, m2};
#pragma unroll
        for (int e0 = 0; e0 < 48; e0 += 4) {
            if (e0 >= nsh * 3) break;
            float x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int e = e0 + i;
                x[i] = b[e / 3] * m[e % 3];
            }
            atomicAdd(reinterpret_cast<float4*>(ds + e0), make_float4(x[0], x[1], x[2], x[3]));
        }
    } else {
        for (int q = 0; q < nsh; ++q) {
            if (m0 != 0.0f) atomicAdd(ds + q * 3 + 0, b[q] * m0);
            if (m1 != 0.0f) atomicAdd(ds + q * 3 + 1, b[q] * m1);
            if (m2 != 0.0f) atomicAdd(ds + q * 3 + 2, b[q] * m2);
        }
    }
}

// Three launches per compositing pass over the three groups of the tile order: the tiles that 5 or more
// actor boxes cover (8 interval slots per ray), those that 1 to 4 cover (4 slots), and the others (this
// file's kernel, no actor machinery, two CTAs per tile).  They run side by side: the two actor launches on
// the context's two extra streams (the device's highest priority, so their CTAs -- the heaviest tiles of
// a frame -- are dispatched first), forked from and joined back into the call's stream by events, the
// plain launch on the call's stream.  Without the extra streams they run one after the other.
template <bool BWD, int KS, bool NRM, bool WEX>
void composite_launch(CompositeArgs A, const Fork* fk, cudaStream_t s) {
    const int n_large = A.bp.n_tiles_large, n_small = A.bp.n_tiles_small;
    const int n_plain = A.bp.n_tiles - n_large - n_small;
    const uint32_t* order = A.tile_order;
    const int groups = (n_large > 0) + (n_small > 0) + (n_plain > 0);
    const bool fork = fk && fk->side && fk->side2 && groups > 1;
    cudaStream_t s_large = s, s_small = s;
    if (fork && cudaEventRecord(fk->ev_fork, s) == cudaSuccess) {
        if (n_large > 0 && cudaStreamWaitEvent(fk->side, fk->ev_fork, 0) == cudaSuccess) s_large = fk->side;
        if (n_small > 0 && cudaStreamWaitEvent(fk->side2, fk->ev_fork, 0) == cudaSuccess) s_small = fk->side2;
    }
    if (n_large > 0) launch_composite_act(A, n_large, BWD, WEX, NRM, true, s_large);
    if (n_small > 0) {
        A.tile_order = order + n_large;
        launch_composite_act(A, n_small, BWD, WEX, NRM, false, s_small);
    }
    if (n_plain > 0) {
        A.tile_order = order + n_large + n_small;
        launch_pdl(k_composite<BWD, KS, NRM, WEX>, dim3(2 * n_plain), dim3(CT_THREADS), s, A);
        count_launches(1);
    }
    if (s_large != s) {
        cudaEventRecord(fk->ev_join, s_large);
        cudaStreamWaitEvent(s, fk->ev_join, 0);
    }
    if (s_small != s) {
        cudaEventRecord(fk->ev_join2, s_small);
        cudaStreamWaitEvent(s, fk->ev_join2, 0);
    }
}

template <bool BWD, bool NRM, bool WEX>
void composite_k(const CompositeArgs& A, const Fork* fk, cudaStream_t s) {
    if (one_sample(A.bp, BWD))
        composite_launch<BWD, 1, NRM, WEX>(A, fk, s);
    else
        composite_launch<BWD, 0, NRM, WEX>(A, fk, s);
}

CompositeArgs make_args(const BatchParams& bp, const VoxRec* rec, const uint32_t* pair_val, const uint16_t* pair_rect,
                        const uint2* tile_range, const uint32_t* vis_start, const uint32_t* tile_order) {
    CompositeArgs A = {};
    A.bp = bp;
    A.rec = rec;
    A.pval = pair_val;
    A.prect = pair_rect;
    A.tile_range = tile_range;
    A.vis_start = vis_start;
    A.tile_order = tile_order;
    return A;
}

}  // namespace

cudaError_t launch_composite_fwd(const BatchParams& bp, const VoxRec* rec, const uint32_t* pair_val,
                                 const uint16_t* pair_rect, const uint2* tile_range, const uint32_t* vis_start,
                                 const uint32_t* tile_order, uint32_t* n_seg, float* t_final,
                                 unsigned long long* work, const Fork* fk, cudaStream_t s) {
    if (bp.n_tiles <= 0) return cudaSuccess;
    CompositeArgs A = make_args(bp, rec, pair_val, pair_rect, tile_range, vis_start, tile_order);
    A.n_seg = n_seg;
    A.t_final = t_final;
    A.work = work;
    if (bp.normals)
        composite_k<false, true, false>(A, fk, s);
    else
        composite_k<false, false, false>(A, fk, s);
    return cudaGetLastError();
}

cudaError_t launch_composite_bwd(const BatchParams& bp, const VoxRec* rec, const uint32_t* pair_val,
                                 const uint16_t* pair_rect, const uint2* tile_range, const uint32_t* vis_start,
                                 const uint32_t* tile_order, const float* t_final, const float* g_rgb,
                                 const float* g_depth, const float* g_alpha, const float* g_normal, float* grad_rec,
                                 const Fork* fk, cudaStream_t s) {
    if (bp.n_tiles <= 0) return cudaSuccess;
    CompositeArgs A = make_args(bp, rec, pair_val, pair_rect, tile_range, vis_start, tile_order);
    // the per-pixel forward results (final T here, C, D, N through the view parameters) are only read
    A.t_final = const_cast<float*>(t_final);
    A.g_rgb = g_rgb;
    A.g_depth = g_depth;
    A.g_alpha = g_alpha;
    A.g_normal = g_normal;
    A.grad_rec = grad_rec;
    if (g_normal)
        composite_k<true, true, false>(A, fk, s);
    else
        composite_k<true, false, false>(A, fk, s);
    return cudaGetLastError();
}

cudaError_t launch_composite_export(const BatchParams& bp, const VoxRec* rec, const uint32_t* pair_val,
                                    const uint16_t* pair_rect, const uint2* tile_range, const uint32_t* vis_start,
                                    const uint32_t* tile_order, const int64_t* offsets, uint32_t* voxel, float* weight,
                                    const Fork* fk, cudaStream_t s) {
    if (bp.n_tiles <= 0) return cudaSuccess;
    CompositeArgs A = make_args(bp, rec, pair_val, pair_rect, tile_range, vis_start, tile_order);
    A.ex_off = offsets;
    A.ex_vid = voxel;
    A.ex_w = weight;
    composite_k<false, false, true>(A, fk, s);
    return cudaGetLastError();
}

cudaError_t launch_sh_bwd(const BatchParams& bp, const uint32_t* sorted_g, int64_t n_vis, const VoxRec* rec,
                          const float* grad_rec, bool with_normals, float* const* d_dens, float* const* d_sh,
                          cudaStream_t s) {
    if (n_vis <= 0) return cudaSuccess;
    ShBwdParams sp;
    sp.bp = bp;
    for (int o = 0; o < DV_MAX_OCTREES; ++o) {
        sp.d_dens[o] = (d_dens && o < bp.n_oct) ? d_dens[o] : nullptr;
        sp.d_sh[o] = (d_sh && o < bp.n_oct) ? d_sh[o] : nullptr;
    }
    if (with_normals)
        launch_pdl(k_sh_bwd<true>, dim3((unsigned)((n_vis + 255) / 256)), dim3(256), s, sp, sorted_g, n_vis, rec, grad_rec);
    else
        launch_pdl(k_sh_bwd<false>, dim3((unsigned)((n_vis + 255) / 256)), dim3(256), s, sp, sorted_g, n_vis, rec, grad_rec);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace dv
