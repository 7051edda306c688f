// Compositing of the tiles that actor clip boxes cover (dv_composite.cu has the others and the
// description of the three phases).
//
// What bounds it.  An actor's voxels are a few pixels on screen or less, so a tile far down the road holds
// tens of thousands of them over a dozen actors while one pixel meets a few hundred, and such a tile is
// one long chain of records: latency, not arithmetic or memory, decides.  Hence:
//  * A warp renders one 8x4 block and streams a sub-list on its own, without CTA barriers: it reads the
//    pairs' pixel rectangles 128 at a time (the next 128 in flight), queues the pairs that touch its
//    block, and stages their records 32 at a time in its own shared-memory buffers (cp.async, one group
//    ahead).  (One ring for four warps, with a barrier per 128 records, left them waiting for each
//    other half of the time.)
//  * The 32 records of a group become one list per lane (a bit transpose of their pixel masks) and every
//    lane steps through its own records, instead of the warp visiting each record for the one or two
//    lanes that meet it.
//  * A tile with SPREAD_MIN or more pairs gets a CTA for each 8x4 block, whose four warps take different
//    actors (a partial and a replay need nothing but the interval and its entry state); other tiles get a
//    CTA per half, a warp per block.
//  * Warps that run apart fetch their instructions apart, and a kernel of this size does not fit the caches near
//    the schedulers: with the walk and the visit inlined wherever they are used, waits for instructions were
//    5.3 cycles an issue on tiles whose voxels cover many pixels (57k leaves, 8 actors, 2442x1704, K = 2: 595 us
//    against 437 for lockstep visits from a CTA-wide ring).  So the forward has one copy of the visit, and with
//    several samples one of the walk for phases 1 and 3 (that render 1,210 -> 1,084 us; 1,120 with two walks, which
//    are the faster with one sample: 480x270 view 0.52 -> 0.48 ms).  The backward is slower with its copies folded
//    (collectives inside the lanes' own loops: 957x541 with normals and K = 4 0.62 -> 0.82 ms) and keeps them.
//  * Measured (GB300, whole renders), lockstep visits from a CTA-wide ring -> this: the 480x270 street
//    view with 20 actors 4.1 -> 0.65 ms, the 32M-leaf render of two 4K cameras 15.4 -> 9.0 ms, a 957x541
//    training step with normals and K = 4 2.2 -> 0.65 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include "dv_composite.cuh"

namespace dv {

namespace {

// Interval slots per ray of the two variants: tiles that 1 to 4 actor boxes cover, and tiles that 5 or
// more cover (a ray with more than 8 intervals takes the per-lane walk for those beyond)
constexpr int NTA_SMALL = 4;
constexpr int NTA_LARGE = 8;
// Tile lists above this length find their sub-lists by binary search (a dozen dependent loads) instead
// of looking at every entry (two dependent loads per 128 entries)
constexpr uint32_t SEARCH_MIN = 512;
// Tiles with this many pairs or more are spread over a CTA per 8x4 block.  2^k - 1, a boundary of the
// tile order's buckets, so that these tiles are the first of their launch.
constexpr uint32_t SPREAD_MIN = 1023;
constexpr int WARPS = CT_THREADS / 32;
constexpr int SCAN = 128;          // pairs a warp looks at per step
constexpr int QCAP = SCAN + 32;    // its queue: what a step adds to a remainder below 32

struct ActInt {
    int o;  // octree index (-1: none)
    int q;  // slot in the lane's interval list (NTA: beyond it)
    float a, b;
};

__device__ __forceinline__ bool slab_box(const float* o, const float* inv, const float* h, float& t0, float& t1) {
    float a = -INFINITY, b = INFINITY;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float ta = (-h[k] - o[k]) * inv[k];
        const float tb = (h[k] - o[k]) * inv[k];
        a = fmaxf(a, fminf(ta, tb));
        b = fminf(b, fmaxf(ta, tb));
    }
    t0 = a;
    t1 = b;
    return a < b;
}

// next actor interval ahead of tau_cur (first-entered box owns overlaps)
__device__ __forceinline__ ActInt next_interval(const OctParams* __restrict__ vo, float t_near, float t_far,
                                                const int16_t* tact, int n_ta, const float* dc, float tau_cur) {
    ActInt r;
    r.o = -1;
    r.q = 1 << 16;  // not in the lane's list
    r.a = INFINITY;
    r.b = 0.0f;
    for (int q = 0; q < n_ta; ++q) {
        const OctParams& P = vo[tact[q]];
        float d[3], inv[3], a, b;
        rotate(P.A, dc, d);
        inv[0] = 1.0f / d[0];
        inv[1] = 1.0f / d[1];
        inv[2] = 1.0f / d[2];
        if (!slab_box(P.o_loc, inv, P.clip_half, a, b)) continue;
        a = fmaxf(a, t_near);
        b = fminf(b, t_far);
        if (!(b > a) || !(b > tau_cur)) continue;
        if (a < r.a) {
            r.o = tact[q];
            r.a = a;
            r.b = b;
        }
    }
    if (r.o >= 0) r.a = fmaxf(r.a, tau_cur);
    return r;
}

template <bool NRM>
__device__ __forceinline__ void atomic_grad(float* grad_rec, uint32_t r, const float* acc) {
    float* gp = grad_rec + (size_t)r * GradLayout<NRM>::STRIDE;
#pragma unroll
    for (int c = 0; c < GradLayout<NRM>::NV; ++c)
        if (acc[c] != 0.0f) atomicAdd(gp + c, acc[c]);
}

// Per-lane walk of one actor's sub-list (divergent; only for a ray's intervals beyond
// the NTA slots).
template <bool GRAD, int KS, bool NRM, bool WEX>
__device__ __noinline__ void walk_actor_lane(Pix<NRM>& ps, const Bwd<NRM>& bw, const BatchParams& bp,
                                             const OctParams* __restrict__ vo, const ActInt& it,
                                             const uint32_t* __restrict__ pval, const uint16_t* __restrict__ prect,
                                             int bx, int by, const VoxRec* __restrict__ rec, uint32_t q0, uint32_t q1,
                                             const float* dc, float* grad_rec, ExportSink* ex) {
    const OctParams& P = vo[it.o];
    float d[3];
    rotate(P.A, dc, d);
    const InvDir inv = inv_dir(d);
    for (uint32_t q = q0; q < q1 && !ps.done(); ++q) {
        if (!((block_pixels(__ldg(prect + q), bx, by) >> (threadIdx.x & 31)) & 1u)) continue;
        ps.tests += 1;
        const uint32_t r = rec_index(bp, pval, q);
        const float4* R = rec[r].v;
        const float4 g = __ldg(R);
        float t0, t1;
        const float rel[3] = {g.x, g.y, g.z};
        slab_cube(inv, g, t0, t1);
        t0 = fmaxf(t0, it.a);
        t1 = fminf(t1, it.b);
        if (!(t1 > t0)) continue;
        float acc[GradLayout<NRM>::NV];
#pragma unroll
        for (int c = 0; c < GradLayout<NRM>::NV; ++c) acc[c] = 0.0f;
        const float4 nv = NRM ? __ldg(bp.nrm + r) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        add_segment<GRAD, true, KS, NRM, WEX, GRAD>(ps, bw, bp, __ldg(R + 1), __ldg(R + 2), __ldg(R + 3), nv, rel, d, t0,
                                              t1, acc, r, ex);
        if (GRAD) atomic_grad<NRM>(grad_rec, r, acc);
    }
}


// Resident CTAs per SM a variant is compiled for: 4, at 128 registers, so that CTAs of the two variants, which run side
// by side, still fit an SM together (the forward's shared memory: 45 KB with 4 slots, 64 KB with 8, with normals 55
// and 80 KB of 227 KB; 5 at 96 registers spill up to 172 bytes: 480x270 view 0.50 -> 0.48 ms, two 4K cameras
// 6.40 -> 6.20 ms; 3 for 8 slots, at 168 registers, 0.52 ms for the view); 3 for the backward with several
// samples, which spills at 128 (957x541 with normals and K = 4 0.62 -> 0.58 ms; with one sample 3 are slower).
template <bool BWD, int KS>
constexpr int act_ctas() {
    return BWD && KS == 0 ? 3 : 4;
}

// A warp's staging buffers
template <bool NRM>
struct WarpRing {
    float4 rec[2][32][5];  // lanes read different records at once: rows of 80 bytes spread them over the banks
    float4 nv[NRM ? 2 : 1][NRM ? 32 : 1];
    uint32_t r[2][32];
    uint32_t q[QCAP];  // queued pairs
};

// Per-lane actor bookkeeping in shared memory: slot k < NTA holds the lane's k-th actor interval along
// its ray (a ray meets few of the boxes that cover its tile, so the slots bound the intervals of one ray,
// not the boxes of the tile)
//   s_iv[k][0/1][px] = the interval [a, b), s_id[k][px] its actor (position in the tile's list)
//   s_st[k][..][px]  = phase 1: the actor's partial; phase 2 overwrites it with the state at the
//                      interval's entry when it is replayed.  Rows:
//     ST_T, ST_N = transmittance and segment count (NO_PARTIAL: left out; phase 2: 0 not reached, 1 partial
//     applied, 2 replay);
//     ST_R = residual sum (backward); ST_B, ST_E = first slot and end of the interval's segments (export);
//     else ST_C.. = C0, C1, C2, D, ST_P = transmittance before the partial's last segment, with normals
//     N0, N1, N2 from ST_V
// A CTA of a spread tile has 32 pixels in its 128 columns, so there slot k sits in row k % NTA, columns
// 32 (k / NTA) and on: four times the slots (rays along the road cross many boxes).
constexpr int ST_T = 0, ST_N = 1, ST_R = 2, ST_B = 2, ST_E = 3, ST_C = 2, ST_P = 6, ST_V = 7;
constexpr float NO_PARTIAL = -1.0f;

// BWD: replay with gradients.  WEX: replay that writes every composited segment's (voxel,
// weight) into the pixel's slots of the weights export (no outputs, no gradients).
template <bool BWD, int KS, bool NRM, bool WEX, int NTA>
__global__ void __launch_bounds__(CT_THREADS, act_ctas<BWD, KS>())
    k_composite_act(const __grid_constant__ CompositeArgs A) {
    pdl_wait();
    pdl_launch_dependents();
    constexpr bool REPLAY = BWD || WEX;  // phase 3 replays every actor interval the ray reached
    // the backward carries the residual form: the actor partials, the states recorded at actor
    // entries and the replays hold (R, T) instead of the prefix colour, depth (and normal)
    constexpr bool RFORM = BWD;
    constexpr int ST_ROWS = RFORM ? 3 : WEX ? 4 : NRM ? 10 : 7;
    constexpr int NV = GradLayout<NRM>::NV;
    constexpr int GS = GradLayout<NRM>::STRIDE;
    __shared__ WarpRing<NRM> s_ring[WARPS];
    __shared__ uint32_t s_sub[DV_MAX_OCTREES + 1];  // sub-list of octree o: [s_sub[o], s_sub[o+1])
    __shared__ uint32_t s_vs[DV_MAX_OCTREES + 1];   // first record of octree o in this view
    __shared__ bool s_flag[DV_MAX_OCTREES];         // actor o's box covers this tile
    __shared__ int16_t s_act[DV_MAX_OCTREES];       // the tile's actors in octree order
    __shared__ int16_t s_near[DV_MAX_OCTREES];      // positions in s_act, nearest box centre first
    __shared__ float s_iv[NTA][2][CT_THREADS];
    __shared__ uint8_t s_id[NTA][CT_THREADS];
    __shared__ uint8_t s_niv[CT_THREADS];           // intervals in the slots
    __shared__ float s_st[NTA][ST_ROWS][CT_THREADS];
    __shared__ int s_nact;
    const BatchParams& bp = A.bp;
    const uint32_t* __restrict__ pval = A.pval;
    const uint16_t* __restrict__ prect = A.prect;
    const VoxRec* __restrict__ rec = A.rec;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the first n_spread tiles have eight CTAs each (those of them below SPREAD_MIN use two), the others two
    const int cta = blockIdx.x, wide = 8 * A.n_spread;
    const int ti = cta < wide ? cta >> 3 : A.n_spread + ((cta - wide) >> 1);
    const int sub = cta < wide ? cta & 7 : (cta - wide) & 1;
    const int gtile = (int)__ldg(A.tile_order + ti);
    const uint2 rg = tile_slice(A, gtile);
    const bool spread = cta < wide && rg.y - rg.x >= SPREAD_MIN;
    if (!spread && sub >= 2) return;
    const int view = view_of(bp, gtile);
    const ViewParams& fp = bp.views[view];
    const OctParams* __restrict__ vo = bp.octs + view * bp.n_oct;
    const int n_oct = bp.n_oct;
    const int tiles_x = fp.tiles_x;
    const float t_near = fp.near_, t_far = fp.far_;
    const int tile = gtile - bp.tile_base[view];
    const int tx = tile % tiles_x, ty = tile / tiles_x;
    // this warp's 8x4 block of the tile, the actors it takes (every nw-th from wi) and the lane's column of
    // the shared per-pixel arrays
    const int block = spread ? sub : sub * 4 + warp;
    const int bx = block & 1, by = block >> 1;
    const int wi = spread ? warp : 0, nw = spread ? WARPS : 1;
    const int px = spread ? lane : tid;
    const bool owner = !spread || warp == 0;  // composites the block's pixels (the other warps only their actors)
    const int u = tx * DV_TILE + bx * 8 + (lane & 7);
    const int v = ty * DV_TILE + by * 4 + (lane >> 3);
    const bool valid = u < fp.W && v < fp.H;
    const int64_t lpix = (int64_t)v * fp.W + u;    // pixel within the view's own images
    const int64_t pix = fp.pix_base + lpix;        // pixel within the call's per-pixel arrays
    WarpRing<NRM>& ring = s_ring[warp];
    const int cap = spread ? NTA * WARPS : NTA;  // slots per ray
    auto iv = [&](int k, int i) -> float& { return s_iv[k % NTA][i][px + k / NTA * 32]; };
    auto id_of = [&](int k) -> uint8_t& { return s_id[k % NTA][px + k / NTA * 32]; };
    auto st = [&](int k, int row) -> float& { return s_st[k % NTA][row][px + k / NTA * 32]; };

    float dc[3], db_[3];
    pixel_ray(fp, u, v, dc);
    rotate(vo[0].A, dc, db_);
    const InvDir ib = inv_dir(db_);
    Pix<NRM> ps;
    init_pix<NRM>(ps, valid ? t_far : -1.0f);
    ExportSink ex;
    if constexpr (WEX)
        init_sink(ex, A, view, pix, valid);
    else
        ex.n = ex.lim = 0;
    Bwd<NRM> bw;
    load_bwd<BWD, NRM>(bw, A, fp, lpix, pix, valid);
    // tile set-up, all loads independent of one another: the view's octree boundaries in
    // the record order, and which actor boxes cover this tile
    for (int i = tid; i <= n_oct; i += CT_THREADS) {
        s_vs[i] = __ldg(A.vis_start + view * n_oct + i);
        s_sub[i] = rg.x;  // every sub-list start stays inside the tile's slice
    }
    for (int o = tid; o < n_oct; o += CT_THREADS) {
        const OctParams& P = vo[o];
        s_flag[o] = o > 0 && P.role == DV_ROLE_ACTOR && P.rect[0] <= tx && tx <= P.rect[2] && P.rect[1] <= ty &&
                    ty <= P.rect[3];
    }
    __syncthreads();
    // the tile's list is grouped by octree (records are in depth-key order, octree above
    // the BSP path), so octree o's sub-list starts at the first entry whose record is at
    // or after s_vs[o].  In a short list every entry finds its octree by a search of s_vs and
    // marks the starts of the octrees between its predecessor's and its own; in a long one
    // every start is a binary search of the list.
    if (rg.y - rg.x > SEARCH_MIN) {
        for (int o = tid; o <= n_oct; o += CT_THREADS) {
            const uint32_t first = s_vs[o];
            uint32_t lo = o < n_oct ? rg.x : rg.y, hi = rg.y;
            while (lo < hi) {
                const uint32_t mid = lo + ((hi - lo) >> 1);
                if (rec_index(bp, pval, mid) < first)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            s_sub[o] = lo;
        }
    } else {
        auto oct_of = [&](uint32_t r) {
            int lo = 0, hi = n_oct - 1;  // largest o with s_vs[o] <= r
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_vs[mid] <= r)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            return lo;
        };
        for (uint32_t base = rg.x; base < rg.y; base += CT_THREADS) {
            const uint32_t q = base + tid;
            if (q < rg.y) {
                const int o = oct_of(rec_index(bp, pval, q));
                const int op = q > rg.x ? oct_of(rec_index(bp, pval, q - 1)) : -1;
                for (int x = op + 1; x <= o; ++x) s_sub[x] = q;
                if (q + 1 == rg.y)
                    for (int x = o + 1; x <= n_oct; ++x) s_sub[x] = rg.y;
            }
        }
    }
    if (tid < 32) {
        // actor list of the tile in octree order (warp 0, ballot compaction)
        int n = 0;
        for (int o0 = 0; o0 < n_oct; o0 += 32) {
            const int o = o0 + tid;
            const bool f = o < n_oct && s_flag[o];
            const unsigned b = __ballot_sync(0xffffffffu, f);
            if (f) s_act[n + __popc(b & ((1u << tid) - 1u))] = (int16_t)o;
            n += __popc(b);
        }
        if (tid == 0) s_nact = n;
    }
    __syncthreads();
    const int n_ta = s_nact;

    // ---- owned actor intervals of this ray, in order along it, and the actors by distance ----
    bool more = false;  // there may be others behind the last slot
    if (owner) {
        int n_iv = 0;
        if (valid) {
            // the boxes the ray meets, inserted by entry (equal entries keep octree order)
            for (int q = 0; q < n_ta; ++q) {
                const OctParams& P = vo[s_act[q]];
                float d[3], inv[3], a, b;
                rotate(P.A, dc, d);
                inv[0] = 1.0f / d[0];
                inv[1] = 1.0f / d[1];
                inv[2] = 1.0f / d[2];
                if (!slab_box(P.o_loc, inv, P.clip_half, a, b)) continue;
                a = fmaxf(a, t_near);
                b = fminf(b, t_far);
                if (!(b > a) || !(b > t_near)) continue;
                if (n_iv == cap) {
                    more = true;
                    break;
                }
                int k = n_iv++;
                for (; k > 0 && iv(k - 1, 0) > a; --k) {
                    iv(k, 0) = iv(k - 1, 0);
                    iv(k, 1) = iv(k - 1, 1);
                    id_of(k) = id_of(k - 1);
                }
                iv(k, 0) = a;
                iv(k, 1) = b;
                id_of(k) = (uint8_t)q;
            }
            ps.boxes += n_ta;
            float tau = t_near;
            if (!more) {
                // the box entered first owns any overlap; a box keeps what lies behind the last one
                const int n = n_iv;
                n_iv = 0;
                for (int k = 0; k < n; ++k) {
                    const float a = iv(k, 0), b = iv(k, 1);
                    const uint8_t id = id_of(k);
                    if (!(b > tau)) continue;
                    iv(n_iv, 0) = fmaxf(a, tau);
                    iv(n_iv, 1) = b;
                    id_of(n_iv) = id;
                    ++n_iv;
                    tau = b;
                }
            } else {
                // more boxes than slots: the first intervals one by one
                for (n_iv = 0; n_iv < cap;) {
                    const ActInt it = next_interval(vo, t_near, t_far, s_act, n_ta, dc, tau);
                    ps.boxes += n_ta;
                    if (it.o < 0) break;
                    int q = 0;
                    while (s_act[q] != it.o) ++q;
                    iv(n_iv, 0) = it.a;
                    iv(n_iv, 1) = it.b;
                    id_of(n_iv) = (uint8_t)q;
                    ++n_iv;
                    tau = it.b;
                }
                more = n_iv == cap;
            }
        }
        for (int k = 0; k < n_iv; ++k) {
            st(k, ST_T) = 1.0f;
            st(k, ST_N) = 0.0f;
        }
        s_niv[px] = (uint8_t)n_iv;
    }
    // phase 1 takes the actors nearest box centre first, so that what hides an actor from a ray is
    // mostly known before the actor's turn
    for (int q = tid; q < n_ta; q += CT_THREADS) {
        const float* m = vo[s_act[q]].m;
        const float dq = fmaf(m[0], m[0], fmaf(m[1], m[1], m[2] * m[2]));
        int rank = 0;
        for (int x = 0; x < n_ta; ++x) {
            const float* mx = vo[s_act[x]].m;
            const float dx = fmaf(mx[0], mx[0], fmaf(mx[1], mx[1], mx[2] * mx[2]));
            rank += (dx < dq || (dx == dq && x < q)) ? 1 : 0;
        }
        s_near[rank] = (int16_t)q;
    }
    __syncthreads();
    const int n_iv = s_niv[px];
    // the lane's slot of the tile's actor q (-1: the ray does not meet it, or beyond the slots)
    auto slot_of = [&](int q) {
        int r = -1;
        for (int k = 0; k < n_iv; ++k)
            if (id_of(k) == q) r = k;
        return r;
    };

    // The records of [q0, q1) that touch the warp's block, 32 at a time: group(b, n, pm) gets the buffer,
    // the number of records and, in lane i, the pixels record i may touch, and returns true once the
    // warp has nothing left to do in this list.
    auto stream = [&](uint32_t q0, uint32_t q1, auto&& group) {
        constexpr int S = SCAN / 32;
        uint32_t rc[S], rc2[S];
        auto fetch = [&](uint32_t base, uint32_t* x) {
#pragma unroll
            for (int i = 0; i < S; ++i) {
                const uint32_t q = base + i * 32 + lane;
                x[i] = q < q1 ? (uint32_t)__ldg(prect + q) : 0x0fu;  // x1 < x0: touches nothing
            }
        };
        fetch(q0, rc);
        int qn = 0, buf = 0, staged = 0;  // queued pairs; records staged in buf ^ 1 and not yet visited
        uint32_t pm_staged = 0;
        bool fin = false;
        for (uint32_t base = q0; base < q1 && !fin; base += SCAN) {
            const bool last = q1 - base <= SCAN;
            if (!last) fetch(base + SCAN, rc2);
#pragma unroll
            for (int i = 0; i < S; ++i) {
                const uint32_t pm = block_pixels(rc[i], bx, by);
                const unsigned b = __ballot_sync(0xffffffffu, pm != 0u);
                if (pm) {
                    const int at = qn + __popc(b & ((1u << lane) - 1u));
                    ring.q[at] = base + i * 32 + lane;
                }
                qn += __popc(b);
                rc[i] = rc2[i];
            }
            __syncwarp();
            int head = 0;
            while (qn - head >= 32 || (last && (qn > head || staged))) {
                const int n = min(qn - head, 32);
                uint32_t pm = 0;
                if (lane < n) {
                    const uint32_t q = ring.q[head + lane];
                    const uint32_t r = rec_index(bp, pval, q);
                    pm = block_pixels(__ldg(prect + q), bx, by);
                    const float4* R = rec[r].v;
#pragma unroll
                    for (int k = 0; k < 4; ++k) cp_async16(&ring.rec[buf][lane][k], R + k);
                    if (NRM) cp_async16(&ring.nv[NRM ? buf : 0][NRM ? lane : 0], bp.nrm + r);
                    ring.r[buf][lane] = r;
                }
                cp_async_commit();
                head += n;
                if (staged) {
                    cp_async_wait_one();  // the group before this one has landed
                    __syncwarp();
                    fin = group(buf ^ 1, staged, pm_staged);
                    __syncwarp();  // every lane is done with it before its buffer is filled again
                    if (fin) break;
                }
                staged = n;
                pm_staged = pm;
                buf ^= 1;
            }
            // the remainder (below 32) to the front of the queue
            const int rest = qn - head;
            const uint32_t q_rest = lane < rest ? ring.q[head + lane] : 0u;
            __syncwarp();
            if (lane < rest) ring.q[lane] = q_rest;
            qn = rest;
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");  // no copy outlives the list (early exit)
        __syncwarp();
    };

    // voxel normal of staged record j (zero without normals)
    auto staged_nv = [&](int b, uint32_t j) {
        return NRM ? ring.nv[NRM ? b : 0][NRM ? j : 0] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    };
    // whether a group with gradients is walked lane by lane
    auto by_lanes = [&](uint32_t mine, int n) {
        return (int)__reduce_max_sync(0xffffffffu, (unsigned)__popc(mine)) * LANE_GAIN <= n;
    };

    // Walk of actor o's sub-list: lanes not yet done composite the segments inside their interval
    // [a, pt.end] of that actor into pt, with the stop rule (and, with G, the per-record gradients), two
    // records at a time without gradients.
    auto walk_actor = [&](Pix<NRM>& pt, int o, float a, auto grad, auto wex) {
        constexpr bool G = decltype(grad)::value;
        constexpr bool X = decltype(wex)::value;
        const OctParams& P = vo[o];
        float d[3];
        rotate(P.A, dc, d);
        const InvDir inv = inv_dir(d);
        auto clip = [&](float4 g, float& t0, float& t1) {
            slab_cube(inv, g, t0, t1);
            t0 = fmaxf(t0, a);
            t1 = fminf(t1, pt.end);
            return t1 > t0;
        };
        stream(s_sub[o], s_sub[o + 1], [&](int bf, int n, uint32_t pm) -> bool {
            if (__all_sync(0xffffffffu, pt.done())) return true;
            uint32_t mine = warp_transpose(pm);
            if (pt.done()) mine = 0u;
            bool lanes = true;
            if constexpr (G) lanes = by_lanes(mine, n);
            if (lanes) {
                while (mine) {
                    const uint32_t j = (uint32_t)(__ffs(mine) - 1);
                    mine &= mine - 1;
                    const float4 g0 = ring.rec[bf][j][0];
                    if constexpr (!G && !X && KS == 1) {
                        // both slab tests and optical depths, then the two compositing steps in list order
                        // with the stop rule -- the arithmetic of two single steps
                        const bool two = mine != 0u;
                        const uint32_t j1 = two ? (uint32_t)(__ffs(mine) - 1) : j;
                        mine &= mine - 1;
                        const float4 g1 = ring.rec[bf][j1][0];
                        float u0, v0, u1, v1;
                        const bool h0 = clip(g0, u0, v0), h1 = clip(g1, u1, v1) && two;
                        const float4 col0 = ring.rec[bf][j][3], col1 = ring.rec[bf][j1][3];
                        const float r0[3] = {g0.x, g0.y, g0.z}, r1[3] = {g1.x, g1.y, g1.z};
                        const float tau0 = seg_tau<false, 1>(ring.rec[bf][j][1], ring.rec[bf][j][2], col0.w, r0, d, u0,
                                                             v0, bp.K, bp.inv_k, bp.act_thr, nullptr, nullptr);
                        const float tau1 = seg_tau<false, 1>(ring.rec[bf][j1][1], ring.rec[bf][j1][2], col1.w, r1, d, u1,
                                                             v1, bp.K, bp.inv_k, bp.act_thr, nullptr, nullptr);
                        auto apply = [&](float tau, float4 col, float4 nv, float t0, float t1) {
                            if constexpr (RFORM) {
                                const float ee = exp_neg(tau);
                                const float w = pt.T * (1.0f - ee);
                                const float mid = 0.5f * (t0 + t1);
                                float sg = fmaf(bw.g0, col.x, fmaf(bw.g1, col.y, fmaf(bw.g2, col.z, bw.gD * mid)));
                                if constexpr (NRM) sg = fmaf(bw.gN0, nv.x, fmaf(bw.gN1, nv.y, fmaf(bw.gN2, nv.z, sg)));
                                pt.R = fmaf(w, sg, pt.R);
                                pt.T = pt.T * ee;
                                pt.n += 1;
                                if (pt.T < bp.eps_stop) pt.stop();
                            } else {
                                composite_tau<NRM>(pt, tau, col, nv, t0, t1, bp.eps_stop);
                            }
                        };
                        pt.tests += 1;
                        if (h0) apply(tau0, col0, staged_nv(bf, j), u0, v0);
                        pt.tests += (two && !pt.done()) ? 1u : 0u;
                        if (h1 && !pt.done()) apply(tau1, col1, staged_nv(bf, j1), u1, v1);
                    } else {
                        pt.tests += 1;
                        float t0, t1;
                        if (clip(g0, t0, t1)) {
                            float acc[NV];
                            if constexpr (G && KS == 1) {
                                bwd_single_step<NRM>(pt, bw, bp, g0, ring.rec[bf][j][1], ring.rec[bf][j][2],
                                                     ring.rec[bf][j][3], staged_nv(bf, j), d, t0, t1, true, acc);
                            } else {
#pragma unroll
                                for (int i = 0; i < NV; ++i) acc[i] = 0.0f;
                                const float rel[3] = {g0.x, g0.y, g0.z};
                                add_segment<G, true, KS, NRM, X, RFORM>(pt, bw, bp, ring.rec[bf][j][1],
                                                                        ring.rec[bf][j][2], ring.rec[bf][j][3],
                                                                        staged_nv(bf, j), rel, d, t0, t1, acc,
                                                                        ring.r[bf][j], &ex);
                            }
                            if constexpr (G) lane_add<NRM>(A.grad_rec, ring.r[bf][j], acc);
                        }
                    }
                    if (pt.done()) mine = 0u;
                }
                __syncwarp();
            } else if constexpr (G) {
                for (uint32_t j = 0; j < (uint32_t)n; ++j) {
                    if (__all_sync(0xffffffffu, pt.done())) return true;
                    const float4 g = ring.rec[bf][j][0];
                    float t0, t1;
                    const bool hit = clip(g, t0, t1);
                    if (!__any_sync(0xffffffffu, hit)) continue;
                    float acc[NV];
                    if constexpr (KS == 1) {
                        // inside one actor interval a lane meets a record at most once
                        bwd_single_step<NRM>(pt, bw, bp, g, ring.rec[bf][j][1], ring.rec[bf][j][2], ring.rec[bf][j][3],
                                             staged_nv(bf, j), d, hit ? t0 : 0.0f, hit ? t1 : 0.0f, hit, acc);
                    } else {
#pragma unroll
                        for (int i = 0; i < NV; ++i) acc[i] = 0.0f;
                        const float rel[3] = {g.x, g.y, g.z};
                        if (hit)
                            add_segment<G, true, KS, NRM, X, RFORM>(pt, bw, bp, ring.rec[bf][j][1], ring.rec[bf][j][2],
                                                                    ring.rec[bf][j][3], staged_nv(bf, j), rel, d, t0,
                                                                    t1, acc, ring.r[bf][j], &ex);
                    }
                    warp_reduce_add<NV>(acc, A.grad_rec + (size_t)ring.r[bf][j] * GS);
                }
            }
            return __all_sync(0xffffffffu, pt.done());
        });
    };

    // ---- phase 2: background walk, applying actor partials in order ----
    auto background = [&]() {
        float tau_cur = t_near;
        ActInt nxt;
        nxt.o = -1;
        nxt.q = -1;
        nxt.a = nxt.b = 0.0f;
        // the interval behind the current one: the lane's next slot, then (beyond the slots) a search
        auto advance = [&]() {
            const int k = nxt.q + 1;
            if (k < n_iv) {
                nxt.o = s_act[id_of(k)];
                nxt.q = k;
                nxt.a = iv(k, 0);
                nxt.b = iv(k, 1);
            } else if (more) {
                nxt = next_interval(vo, t_near, t_far, s_act, n_ta, dc, tau_cur);
                ps.boxes += n_ta;
            } else {
                nxt.o = -1;
            }
        };
        if (valid) advance();
        // enters actor interval `it`: apply its partial, or stop inside it, or walk it per lane
        auto enter_actor = [&](const ActInt& it) {
            // The partial holds for a ray that enters with T <= 1: it may have been left out, or have stopped,
            // because the ray would have stopped by then.  A ray that gets here all the same (T above 1 behind
            // negative densities under the identity activation, or eps_stop above 1 and no segment yet) walks
            // the interval with the exact stop rule.
            bool walk = it.q >= cap;
            if (!walk) {
                const float t = st(it.q, ST_T);
                walk = st(it.q, ST_N) == NO_PARTIAL || (t < bp.eps_stop && !(ps.T * t < bp.eps_stop));
            }
            if (walk) {
                // the out-of-line walk takes copies: an object whose address reaches a call stays in
                // local memory everywhere, so the hot-path state (ps, bw, dc, nxt, ex) never does
                Pix<NRM> pl = ps;
                const Bwd<NRM> bl = bw;
                const ActInt il = it;
                const float dl[3] = {dc[0], dc[1], dc[2]};
                ExportSink xl = ex;
                walk_actor_lane<BWD, KS, NRM, WEX>(pl, bl, bp, vo, il, pval, prect, bx, by, rec, s_sub[il.o],
                                                   s_sub[il.o + 1], dl, A.grad_rec, &xl);
                ps = pl;
                ex = xl;
                return;
            }
            const int k = it.q;
            const float pT = st(k, ST_T);
            const uint32_t pn = (uint32_t)__float_as_int(st(k, ST_N));
            const bool stop_inside = ps.T * pT < bp.eps_stop;
            if constexpr (REPLAY) {
                // record the entry state for the replay, then apply the partial
                if constexpr (RFORM) {
                    const float pR = st(k, ST_R);
                    st(k, ST_R) = ps.R;
                    if (!stop_inside) ps.R = fmaf(ps.T, pR, ps.R);
                } else {
                    // the interval's segments take their place in the pixel's slots, front to back
                    st(k, ST_B) = __int_as_float((int)ex.n);
                    ex.n = stop_inside ? ex.lim : ex.n + pn;
                    st(k, ST_E) = __int_as_float((int)min(ex.n, ex.lim));
                }
                st(k, ST_T) = ps.T;
                st(k, ST_N) = 1.0f;
                if (!stop_inside) {
                    ps.T = ps.T * pT;
                    ps.n += pn;
                }
            } else {
                const float pC0 = st(k, ST_C), pC1 = st(k, ST_C + 1), pC2 = st(k, ST_C + 2);
                const float pD = st(k, ST_C + 3), pP = st(k, ST_P);
                // The ray stops inside when T T_A falls below eps_stop.  If it had not before the
                // partial's last segment (by more than rounding), that segment is where it stops and the
                // whole partial applies; else the interval is replayed from the entry state.
                const bool at_end = ps.T * pP >= bp.eps_stop * 1.00001f && ps.T * pT < bp.eps_stop * 0.99999f;
                const bool replay = stop_inside && !at_end;
                float pN[3] = {0.0f, 0.0f, 0.0f};
                if constexpr (NRM) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) pN[c] = st(k, ST_V + c);
                }
                st(k, ST_N) = replay ? 2.0f : 1.0f;
                if (replay) {
                    st(k, ST_C) = ps.C0;
                    st(k, ST_C + 1) = ps.C1;
                    st(k, ST_C + 2) = ps.C2;
                    st(k, ST_C + 3) = ps.D;
                    st(k, ST_T) = ps.T;
                    if constexpr (NRM) {
                        st(k, ST_V) = ps.N0;
                        st(k, ST_V + 1) = ps.N1;
                        st(k, ST_V + 2) = ps.N2;
                    }
                } else {
                    ps.C0 = fmaf(ps.T, pC0, ps.C0);
                    ps.C1 = fmaf(ps.T, pC1, ps.C1);
                    ps.C2 = fmaf(ps.T, pC2, ps.C2);
                    ps.D = fmaf(ps.T, pD, ps.D);
                    if constexpr (NRM) {
                        ps.N0 = fmaf(ps.T, pN[0], ps.N0);
                        ps.N1 = fmaf(ps.T, pN[1], ps.N1);
                        ps.N2 = fmaf(ps.T, pN[2], ps.N2);
                    }
                    ps.T = ps.T * pT;
                    ps.n += pn;
                }
            }
            if (stop_inside) ps.stop();
        };
        auto clip = [&](float4 g, float& t_in, float& t_out) {
            slab_cube(ib, g, t_in, t_out);
            t_in = fmaxf(t_in, t_near);
            t_out = fminf(t_out, ps.end);
            return t_out > t_in;
        };
        // one lane's segments of staged record j, entering the actor intervals inside them; with
        // gradients the values are added to acc; true if it composited any
        auto visit = [&](int bf, uint32_t j, float* acc) -> bool {
            bool some = false;
            const float4 g = ring.rec[bf][j][0];
            float t_in, t_out;
            ps.tests += 1;
            if (!clip(g, t_in, t_out)) return false;
            const float rel[3] = {g.x, g.y, g.z};
            const float4 da = ring.rec[bf][j][1], dd = ring.rec[bf][j][2], col = ring.rec[bf][j][3];
            const float4 nv = staged_nv(bf, j);
            float cur = fmaxf(t_in, tau_cur);
            while (nxt.o >= 0 && nxt.a < t_out && !ps.done()) {
                if (nxt.a > cur) {
                    add_segment<BWD, true, KS, NRM, WEX, RFORM>(ps, bw, bp, da, dd, col, nv, rel, db_, cur, nxt.a, acc,
                                                                ring.r[bf][j], &ex);
                    some = true;
                    if (ps.done()) break;
                }
                enter_actor(nxt);
                tau_cur = nxt.b;
                cur = fmaxf(cur, nxt.b);
                advance();
            }
            if (!ps.done() && t_out > cur) {
                add_segment<BWD, true, KS, NRM, WEX, RFORM>(ps, bw, bp, da, dd, col, nv, rel, db_, cur, t_out, acc,
                                                            ring.r[bf][j], &ex);
                some = true;
            }
            return some;
        };
        stream(s_sub[0], s_sub[1], [&](int bf, int n, uint32_t pm) -> bool {
            if (__all_sync(0xffffffffu, ps.done())) return true;
            uint32_t mine = warp_transpose(pm);
            if (ps.done()) mine = 0u;
            bool lanes = true;
            if constexpr (BWD) lanes = by_lanes(mine, n);
            if (lanes) {
                while (mine) {
                    const uint32_t j0 = (uint32_t)(__ffs(mine) - 1);
                    mine &= mine - 1;
                    if constexpr (REPLAY) {
                        float acc[NV];
                        if constexpr (BWD) {
#pragma unroll
                            for (int i = 0; i < NV; ++i) acc[i] = 0.0f;
                        }
                        const bool some = visit(bf, j0, acc);
                        if constexpr (BWD) {
                            if (some) lane_add<NRM>(A.grad_rec, ring.r[bf][j0], acc);
                        }
                    } else {
                        // two records at once: both slab tests, then (unless the lane enters an actor
                        // interval inside either segment) both optical depths, then compositing in list
                        // order with the stop rule -- the same arithmetic as two visits
                        const bool two = mine != 0u;
                        const uint32_t j1 = two ? (uint32_t)(__ffs(mine) - 1) : j0;
                        mine &= mine - 1;
                        const float4 g0 = ring.rec[bf][j0][0], g1 = ring.rec[bf][j1][0];
                        float a0, b0, a1, b1;
                        const bool in0 = clip(g0, a0, b0), in1 = clip(g1, a1, b1) && two;
                        if (nxt.o >= 0 && ((in0 && nxt.a < b0) || (in1 && nxt.a < b1))) {
                            // (a loop: one copy of the visit)
#pragma unroll 1
                            for (uint32_t x = 0; x < (two ? 2u : 1u) && !ps.done(); ++x)
                                visit(bf, x ? j1 : j0, nullptr);
                        } else {
                            a0 = fmaxf(a0, tau_cur);
                            a1 = fmaxf(a1, tau_cur);
                            const bool h0 = in0 && b0 > a0, h1 = in1 && b1 > a1;
                            const float4 da0 = ring.rec[bf][j0][1], dd0 = ring.rec[bf][j0][2], col0 = ring.rec[bf][j0][3];
                            const float4 da1 = ring.rec[bf][j1][1], dd1 = ring.rec[bf][j1][2], col1 = ring.rec[bf][j1][3];
                            const float r0[3] = {g0.x, g0.y, g0.z}, r1[3] = {g1.x, g1.y, g1.z};
                            const float tau0 = seg_tau<false, KS>(da0, dd0, col0.w, r0, db_, a0, b0, bp.K, bp.inv_k,
                                                                  bp.act_thr, nullptr, nullptr);
                            const float tau1 = seg_tau<false, KS>(da1, dd1, col1.w, r1, db_, a1, b1, bp.K, bp.inv_k,
                                                                  bp.act_thr, nullptr, nullptr);
                            ps.tests += 1;
                            if (h0) composite_tau<NRM>(ps, tau0, col0, staged_nv(bf, j0), a0, b0, bp.eps_stop);
                            ps.tests += (two && !ps.done()) ? 1u : 0u;
                            if (h1 && !ps.done()) composite_tau<NRM>(ps, tau1, col1, staged_nv(bf, j1), a1, b1, bp.eps_stop);
                        }
                    }
                    if (ps.done()) mine = 0u;
                }
                __syncwarp();
            } else if constexpr (BWD) {
                for (uint32_t j = 0; j < (uint32_t)n; ++j) {
                    if (__all_sync(0xffffffffu, ps.done())) return true;
                    float acc[NV];
                    bool some = false;
                    if constexpr (KS == 1) {
                        // a record that no lane's segment carries into the next actor interval is met at most
                        // once by every lane, so it takes the branch-free step; a record some lane crosses an
                        // actor entry in goes through the general path below
                        const float4 g = ring.rec[bf][j][0];
                        float t_in, t_out;
                        const bool in = clip(g, t_in, t_out);
                        if (!__any_sync(0xffffffffu, in && nxt.o >= 0 && nxt.a < t_out)) {
                            const float cur = fmaxf(t_in, tau_cur);
                            const bool hit = in && t_out > cur;
                            if (!__any_sync(0xffffffffu, hit)) continue;
                            bwd_single_step<NRM>(ps, bw, bp, g, ring.rec[bf][j][1], ring.rec[bf][j][2],
                                                 ring.rec[bf][j][3], staged_nv(bf, j), db_, hit ? cur : 0.0f,
                                                 hit ? t_out : 0.0f, hit, acc);
                            warp_reduce_add<NV>(acc, A.grad_rec + (size_t)ring.r[bf][j] * GS);
                            continue;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < NV; ++i) acc[i] = 0.0f;
                    if (!ps.done()) some = visit(bf, j, acc);
                    // every lane visits record j together: reduce across the warp
                    if (__any_sync(0xffffffffu, some)) warp_reduce_add<NV>(acc, A.grad_rec + (size_t)ring.r[bf][j] * GS);
                }
            }
            return __all_sync(0xffffffffu, ps.done());
        });
        // actor intervals behind the last background hit
        while (nxt.o >= 0 && !ps.done()) {
            enter_actor(nxt);
            tau_cur = nxt.b;
            advance();
        }
        __syncwarp();
    };

    // ---- phase 1: partial composite of the actor intervals ----
    // Transmittance never rises along a ray, so if the partials of the lane's earlier intervals
    // already multiply to less than eps_stop the ray stops before this one, and its partial is
    // not needed (phase 2 multiplies the same factors in the same order, and the background's on
    // top, so with T <= 1 it cannot get past them; enter_actor has the other rays).  Another warp's
    // partial counts once it is written; before that its factor is 1.
    // ---- phase 3: actor intervals replayed from their entry state ----
    //   forward: only those where the ray stops before the partial's end (by the pixels' own warp);
    //   backward and export: every one reached, shared by the CTA's warps
    // (one loop for both, and so one copy of the walk, in the forward with several samples: see the top of the file)
#pragma unroll (REPLAY || KS == 1 ? 2 : 1)
    for (int phase = 1; phase <= 3; phase += 2) {
        const bool partial = phase == 1;
        if (!partial) {
            if (spread) __syncthreads();
            if (owner) background();
            if (REPLAY && spread) __syncthreads();
            if (!REPLAY && !owner) break;
        }
        const bool shared = partial || REPLAY;
        for (int i = shared ? wi : 0; i < n_ta; i += shared ? nw : 1) {
            const int q = s_near[i];
            const int k = valid ? slot_of(q) : -1;
            bool act = k >= 0;
            if (act && partial) {
                float T = 1.0f;
                for (int x = 0; x < k; ++x) T *= *(volatile float*)&st(x, ST_T);
                act = !(T < bp.eps_stop);
                if (!act) st(k, ST_N) = NO_PARTIAL;
            } else if (act) {
                const int status = (int)st(k, ST_N);
                act = REPLAY ? status >= 1 : status == 2;
            }
            if (!__any_sync(0xffffffffu, act)) continue;
            Pix<NRM> pt;
            init_pix<NRM>(pt, act ? iv(k, 1) : -1.0f);
            if (act && !partial) {
                pt.T = st(k, ST_T);
                if constexpr (RFORM) {
                    pt.R = st(k, ST_R);
                } else if constexpr (WEX) {
                    ex.n = (uint32_t)__float_as_int(st(k, ST_B));
                    ex.lim = (uint32_t)__float_as_int(st(k, ST_E));
                } else {
                    pt.C0 = st(k, ST_C);
                    pt.C1 = st(k, ST_C + 1);
                    pt.C2 = st(k, ST_C + 2);
                    pt.D = st(k, ST_C + 3);
                    if constexpr (NRM) {
                        pt.N0 = st(k, ST_V);
                        pt.N1 = st(k, ST_V + 1);
                        pt.N2 = st(k, ST_V + 2);
                    }
                }
            }
            // a lane whose own transmittance already falls below eps_stop will stop inside this actor whatever T
            // it enters with (T <= 1), so its partial may stop there too
            const float a = act ? iv(k, 0) : 0.0f;
            if (!REPLAY || partial)
                walk_actor(pt, s_act[q], a, std::false_type(), std::false_type());
            else
                walk_actor(pt, s_act[q], a, std::integral_constant<bool, BWD>(), std::integral_constant<bool, WEX>());
            ps.tests += pt.tests;
            if (!act) continue;
            if (partial) {
                st(k, ST_N) = __int_as_float((int)pt.n);
                if constexpr (RFORM) {
                    st(k, ST_R) = pt.R;
                } else if constexpr (!WEX) {
                    st(k, ST_C) = pt.C0;
                    st(k, ST_C + 1) = pt.C1;
                    st(k, ST_C + 2) = pt.C2;
                    st(k, ST_C + 3) = pt.D;
                    st(k, ST_P) = pt.Tp;
                    if constexpr (NRM) {
                        st(k, ST_V) = pt.N0;
                        st(k, ST_V + 1) = pt.N1;
                        st(k, ST_V + 2) = pt.N2;
                    }
                }
                *(volatile float*)&st(k, ST_T) = pt.T;
            } else if constexpr (WEX) {
                // the replay's T can differ in the last bits from the entry's T times the partial's, on which the
                // forward counted the segments; slots of segments that it does not get to have weight 0
                for (; ex.n < ex.lim; ++ex.n) {
                    ex.vid[ex.base + ex.n] = 0u;
                    ex.w[ex.base + ex.n] = 0.0f;
                }
            } else if constexpr (!REPLAY) {
                ps.C0 = pt.C0;
                ps.C1 = pt.C1;
                ps.C2 = pt.C2;
                ps.D = pt.D;
                if constexpr (NRM) {
                    ps.N0 = pt.N0;
                    ps.N1 = pt.N1;
                    ps.N2 = pt.N2;
                }
                ps.T = pt.T;
                ps.n += pt.n;
            }
        }
    }

    if constexpr (!REPLAY) {
        if (A.work) add_work(A.work, ps.tests, ps.boxes, ps.n);
        if (owner && valid) store_pix<NRM>(ps, A, fp, lpix, pix);
    }
}

template <bool BWD, bool NRM, bool WEX>
void launch_variant(const CompositeArgs& A, unsigned grid, bool large, cudaStream_t s) {
    const dim3 g(grid), b(CT_THREADS);
    if (one_sample(A.bp, BWD)) {
        if (large)
            launch_pdl(k_composite_act<BWD, 1, NRM, WEX, NTA_LARGE>, g, b, s, A);
        else
            launch_pdl(k_composite_act<BWD, 1, NRM, WEX, NTA_SMALL>, g, b, s, A);
    } else {
        if (large)
            launch_pdl(k_composite_act<BWD, 0, NRM, WEX, NTA_LARGE>, g, b, s, A);
        else
            launch_pdl(k_composite_act<BWD, 0, NRM, WEX, NTA_SMALL>, g, b, s, A);
    }
    count_launches(1);
}

}  // namespace

void launch_composite_act(CompositeArgs A, int n_tiles, bool bwd, bool wex, bool normals, bool large, cudaStream_t s) {
    // The tiles with SPREAD_MIN pairs or more come first in the order, and the call's pairs allow for at most
    // n_pairs / SPREAD_MIN of them: that many tiles get eight CTAs (a lighter one among them leaves six at once).
    A.n_spread = (int)(A.bp.n_pairs / SPREAD_MIN < n_tiles ? A.bp.n_pairs / SPREAD_MIN : n_tiles);
    const unsigned grid = 8u * (unsigned)A.n_spread + 2u * (unsigned)(n_tiles - A.n_spread);
    if (bwd) {
        if (normals)
            launch_variant<true, true, false>(A, grid, large, s);
        else
            launch_variant<true, false, false>(A, grid, large, s);
    } else if (wex) {
        launch_variant<false, false, true>(A, grid, large, s);
    } else if (normals) {
        launch_variant<false, true, false>(A, grid, large, s);
    } else {
        launch_variant<false, false, false>(A, grid, large, s);
    }
}

}  // namespace dv
