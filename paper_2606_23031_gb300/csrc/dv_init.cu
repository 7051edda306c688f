// LiDAR-guided initialisation of the background octree (Sec. 3.3): shared grid corners, the
// soft density prior of Eq. 1 and one round of proximity subdivision.
//
//  * Shared corners: every leaf emits its 8 corner grid points (finest-level integer
//    coordinates) tagged with (leaf, corner); one radix sort groups equal points, a scan
//    numbers the distinct ones, and every (leaf, corner) gets its index.
//  * Eq. 1: the LiDAR points are bucketed in a uniform grid of cell h = 3 s (a hash table of the
//    cells that hold points); each corner scans the 27 cells around it for its nearest point.  A point
//    farther than 3 s changes the prior by at most 8 exp(-18) ~ 1e-7, below float32 resolution at
//    v_far, so beyond that radius the corner takes v_far.
//  * Subdivision: every LiDAR point visits, for each level, the leaf cells whose box lies within
//    the threshold of it (exact point-box distance) and looks each up in a hash table of the leaf keys;
//    found leaves are flagged.  At levels where the cells in reach of a point are many (a threshold of several
//    leaves), every leaf looks for a point in reach of it instead, in a grid of the points.  The output keeps the unflagged leaves in input order, then the
//    children of the flagged ones, child 0 of every flagged leaf first, then child 1, ...
//
// What bounds these kernels.  Their results are defined in FP64, and this GPU issues FP64 at 1/64 of the
// FP32 rate (2 per SM and cycle), so a kernel that computes everything in FP64 waits for that pipe
// alone.  They decide in FP32 with an error bound and go to FP64 only where the FP32 value is too
// close to the threshold (or, for a nearest point, could be the nearest), so every result is that of
// the FP64 arithmetic.  Their searches are hash probes, one or two independent loads each, instead of
// binary searches of sorted keys, twenty dependent ones, and need no sort.  On the 500k-leaf background with
// 1.35M points (GB300): prior 3,250 -> 550 us, flags 3,260 -> 420 us,
// visibility over six cameras 843 -> 95 us, beside the sorts of 1.35M points and 500k keys that are gone.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "dv_internal.cuh"

namespace dv {

namespace {

constexpr uint64_t kIMask = (1ull << 19) - 1;
constexpr int kCellBits = 21;
constexpr int64_t kCellOff = 1ll << (kCellBits - 1);

__device__ __forceinline__ uint64_t pack_grid(uint64_t x, uint64_t y, uint64_t z) {
    return (z << 42) | (y << 21) | x;
}

// corner points as sort keys of 3 b bits, b = max_level + 1 (a coordinate of a leaf inside the root is at most
// 2^max_level): the same order as the packed points, in fewer radix passes (5 instead of 8 at level 12).  b = 21, the
// packed point itself, where some leaf lies outside the root.
__global__ void k_corner_emit(const uint64_t* __restrict__ keys, int64_t n, int max_level, int b,
                              uint64_t* __restrict__ ck, uint32_t* __restrict__ cv) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * 8) return;
    const int64_t v = t >> 3;
    const int c = (int)(t & 7);
    const uint64_t k = keys[v];
    const int lev = (int)((k >> 57) & 31);
    const int sh = max_level > lev ? max_level - lev : 0;  // a level above max_level is rejected by the caller
    const uint64_t i = ((k & kIMask) + (c & 1)) << sh;
    const uint64_t j = (((k >> 19) & kIMask) + ((c >> 1) & 1)) << sh;
    const uint64_t kk = (((k >> 38) & kIMask) + ((c >> 2) & 1)) << sh;
    ck[t] = (kk << (2 * b)) | (j << b) | i;
    cv[t] = (uint32_t)t;
}

__global__ void k_corner_flag(const uint64_t* __restrict__ sk, int64_t m, uint32_t* __restrict__ first) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    first[t] = (t == 0 || sk[t] != sk[t - 1]) ? 1u : 0u;
}

// pos = exclusive scan of first: sorted entry t belongs to distinct point pos[t] + first[t] - 1
__global__ void k_corner_assign(const uint64_t* __restrict__ sk, const uint32_t* __restrict__ sv,
                                const uint32_t* __restrict__ first, const uint32_t* __restrict__ pos, int64_t m,
                                int b, uint64_t* __restrict__ grid_out, uint32_t* __restrict__ index_out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    const uint32_t id = pos[t] + first[t] - 1u;
    index_out[sv[t]] = id;
    if (first[t]) {
        const uint64_t k = sk[t], m1 = (1ull << b) - 1;
        grid_out[id] = pack_grid(k & m1, (k >> b) & m1, k >> (2 * b));
    }
}

__device__ __forceinline__ uint64_t cell_key(int64_t cx, int64_t cy, int64_t cz) {
    auto cl = [](int64_t a) {
        a += kCellOff;
        return (uint64_t)(a < 0 ? 0 : (a >= (1ll << kCellBits) ? (1ll << kCellBits) - 1 : a));
    };
    return (cl(cz) << (2 * kCellBits)) | (cl(cy) << kCellBits) | cl(cx);
}

struct Frame {
    double root_min[3];
    double unit;  // finest grid step (root / 2^max_level)
};

// floor(x / unit), the quotient rounded as an FP64 division rounds it.  x times the reciprocal differs
// from it by a few parts in 2^53, so only a product next to an integer needs the division.
__device__ __forceinline__ double floor_div(double x, double unit, double inv) {
    const double t = x * inv;
    const double f = floor(t), r = t - f;
    return (r < 1e-6 || r > 1.0 - 1e-6) ? floor(x / unit) : f;
}

// ---- open-addressing tables of 64-bit keys (power-of-two capacity, at most half full) ----
// A key is entered within HT_PROBES slots of its home, or the call's flag is set and the host takes a
// larger table and, with another salt, other homes, so every probe loop has a fixed bound.  Searches are made by whole warps in step (a lane's
// own loop would run its lanes one after another).
constexpr uint64_t HT_EMPTY = ~0ull;  // never a cell key (63 bits) nor a key looked up (62 bits)
constexpr int HT_PROBES = 64;
constexpr int HT_TRIES = 4;  // tables of 1, 2, 4, 8 times the capacity
// of a try; 0 for the first.  (Any odd multiplier: the keys differ from the salted ones by bits all over the word.)
constexpr uint64_t ht_salt(int more) { return (uint64_t)more * 0xd6e8feb86659fd93ull; }

__device__ __forceinline__ uint32_t ht_first(uint64_t key, int bits, uint64_t salt) {
    key ^= salt;
    key ^= key >> 32;
    key *= 0x9e3779b97f4a7c15ull;  // 2^64 / golden ratio, odd
    key ^= key >> 29;
    key *= 0x9e3779b97f4a7c15ull;
    return (uint32_t)(key >> (64 - bits));
}

// the key's slot, entering it where it is new
__device__ __forceinline__ uint32_t ht_enter(uint64_t* table, int bits, uint64_t salt, uint64_t key, uint32_t* fail) {
    const uint32_t mask = (uint32_t)((1ull << bits) - 1);
    uint32_t h = ht_first(key, bits, salt);
    for (int i = 0; i < HT_PROBES; ++i) {
        const unsigned long long old = atomicCAS(reinterpret_cast<unsigned long long*>(table + h), HT_EMPTY, key);
        if (old == HT_EMPTY || old == key) return h;
        h = (h + 1) & mask;
    }
    *fail = 1u;
    return h;
}

// the slots of the warp's keys, ~0u where a key is absent or its lane not active (all 32 lanes call)
__device__ __forceinline__ uint32_t ht_find(const uint64_t* __restrict__ table, int bits, uint64_t salt, uint64_t key,
                                            bool active) {
    const uint32_t mask = (uint32_t)((1ull << bits) - 1);
    uint32_t h = ht_first(key, bits, salt), found = ~0u;
    for (int i = 0; i < HT_PROBES; ++i) {
        if (!__any_sync(0xffffffffu, active)) break;
        if (active) {
            const uint64_t k = __ldg(table + h);
            if (k == key) found = h;
            active = k != key && k != HT_EMPTY;
            h = (h + 1) & mask;
        }
        __syncwarp();
    }
    return found;
}

int ht_bits(int64_t n) {
    int b = 10;
    while (((int64_t)1 << b) < 2 * n) ++b;
    return b;
}

// ---- point grid of the soft prior: cell -> [start, start + cnt) of the points ordered by cell ----

// some cell near the coordinate's FP64 quotient, a monotone function of it: kept in range as a number before it is
// converted (a point may be anything)
__device__ __forceinline__ int near_cell(float x, double root_min, double inv_h) {
    return (int)fminf(fmaxf((x - (float)root_min) * (float)inv_h, -1e6f), 1e6f);
}

// EXACT: the cell of the FP64 quotient (the prior's cells); else near_cell
template <bool EXACT>
__global__ void __launch_bounds__(256) k_cell_count(const float* __restrict__ cloud, int64_t m, Frame f, double h,
                                                    double inv_h, uint64_t* __restrict__ table, int bits, uint64_t salt,
                                                    uint32_t* __restrict__ cnt, uint32_t* __restrict__ slot,
                                                    uint32_t* __restrict__ rank, uint32_t* __restrict__ fail) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    int64_t c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if constexpr (EXACT)
            c[a] = (int64_t)floor_div((double)cloud[t * 3 + a] - f.root_min[a], h, inv_h);
        else
            c[a] = near_cell(cloud[t * 3 + a], f.root_min[a], inv_h);
    }
    const uint32_t s = ht_enter(table, bits, salt, cell_key(c[0], c[1], c[2]), fail);
    slot[t] = s;
    rank[t] = atomicAdd(cnt + s, 1u);
}

// the cells' ranges, in any order: one reservation per block
__global__ void __launch_bounds__(256) k_cell_alloc(const uint32_t* __restrict__ cnt, int64_t n_slot,
                                                    uint32_t* __restrict__ start, uint32_t* __restrict__ total) {
    __shared__ uint32_t ws[8], base;
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t c = i < n_slot ? cnt[i] : 0u;
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int w = 0; w < 8; ++w) {
            const uint32_t y = ws[w];
            ws[w] = run;
            run += y;
        }
        base = run ? atomicAdd(total, run) : 0u;
    }
    __syncthreads();
    if (c) start[i] = base + ws[warp] + x - c;
}

__global__ void __launch_bounds__(256) k_cell_scatter(const float* __restrict__ cloud, int64_t m,
                                                      const uint32_t* __restrict__ slot,
                                                      const uint32_t* __restrict__ rank,
                                                      const uint32_t* __restrict__ start, float4* __restrict__ pts) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    pts[start[slot[t]] + rank[t]] = make_float4(cloud[t * 3], cloud[t * 3 + 1], cloud[t * 3 + 2], 0.0f);
}

// One thread per corner.  The 27 cells around it, its own first; a cell is skipped when its box is no
// nearer than the best point so far.  Distances are FP32, from the corner split into two floats (relative
// error below 1e-6 of the square beyond `tiny`); the nearest point's is then taken in FP64, and where a
// second point comes within 2e-5 of it, all such points' are.
__global__ void __launch_bounds__(256) k_soft_prior(const uint64_t* __restrict__ grid, int64_t n_corners, Frame f,
                                                    double h, double inv_h, const uint64_t* __restrict__ table,
                                                    int bits, uint64_t salt, const uint32_t* __restrict__ cnt,
                                                    const uint32_t* __restrict__ start, int64_t m,
                                                    const float4* __restrict__ pts, float s, float v_close,
                                                    float v_far, float* __restrict__ dens) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = t < n_corners;
    const uint64_t g = live ? grid[t] : 0ull;
    double q[3];
    q[0] = f.root_min[0] + (double)(g & ((1ull << 21) - 1)) * f.unit;
    q[1] = f.root_min[1] + (double)((g >> 21) & ((1ull << 21) - 1)) * f.unit;
    q[2] = f.root_min[2] + (double)((g >> 42) & ((1ull << 21) - 1)) * f.unit;
    double best = INFINITY;
    if (m > 0) {
        int64_t c[3];
        float qh[3], ql[3], into[3];
        float big = 0.0f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            c[a] = (int64_t)floor_div(q[a] - f.root_min[a], h, inv_h);
            qh[a] = (float)q[a];
            ql[a] = (float)(q[a] - (double)qh[a]);
            big = fmaxf(big, fabsf(qh[a]));
            into[a] = (float)(q[a] - (f.root_min[a] + (double)c[a] * h));
        }
        const float tiny = 1e-22f * big * big, hf = (float)h;
        // lower bound of the distance along an axis to the cells at -1, 0, +1: a point's cell comes from a quotient
        // below 2^21 in FP64, so it can sit at most ~5e-10 h across a cell boundary; 1e-6 h covers the FP32 too
        auto gap = [&](int a, int d) {
            return d == 0 ? 0.0f : fmaxf((d < 0 ? into[a] : hf - into[a]) - 1e-6f * hf, 0.0f);
        };
        float b1 = INFINITY, b2 = INFINITY;  // the two smallest FP32 squares
        uint32_t at = 0;
        // squares above it cannot be the smallest in FP64
        auto bound = [&]() { return fmaf(b1, 1.00002f, tiny); };
        auto cells = [&](auto&& visit) {
            for (int it = 0; it < 27; ++it) {
                const int r = (it + 13) % 27;  // it = 0: the corner's own cell
                const int dx = r % 3 - 1, dy = (r / 3) % 3 - 1, dz = r / 9 - 1;
                const float gx = gap(0, dx), gy = gap(1, dy), gz = gap(2, dz);
                const bool look = live && !(fmaf(gx, gx, fmaf(gy, gy, gz * gz)) * 0.99999f > bound());
                const uint32_t slot = ht_find(table, bits, salt, cell_key(c[0] + dx, c[1] + dy, c[2] + dz), look);
                if (slot != ~0u) {
                    const uint32_t e0 = start[slot], n = min(cnt[slot], (uint32_t)m - e0);
                    for (uint32_t i = 0; i < n; ++i) {
                        const float4 p = __ldg(pts + e0 + i);
                        const float fx = (p.x - qh[0]) - ql[0], fy = (p.y - qh[1]) - ql[1], fz = (p.z - qh[2]) - ql[2];
                        visit(e0 + i, fmaf(fx, fx, fmaf(fy, fy, fz * fz)));
                    }
                }
                __syncwarp();
            }
        };
        cells([&](uint32_t e, float d2) {
            b2 = fminf(b2, fmaxf(d2, b1));
            if (d2 < b1) {
                b1 = d2;
                at = e;
            }
        });
        auto exact = [&](uint32_t e) {
            const float4 p = __ldg(pts + e);
            const double ex = (double)p.x - q[0], ey = (double)p.y - q[1], ez = (double)p.z - q[2];
            best = fmin(best, ex * ex + ey * ey + ez * ez);
        };
        const bool any = b1 < INFINITY, close = any && b2 <= bound();
        if (any) exact(at);
        if (__any_sync(0xffffffffu, close)) {
            const float lim = close ? bound() : -1.0f;
            cells([&](uint32_t e, float d2) {
                if (d2 <= lim) exact(e);
            });
        }
    }
    if (!live) return;
    // Eq. 1 (beyond the 27-cell radius the exponential is below float resolution at v_far)
    const double ss = (double)s * (double)s;
    const double e = best < INFINITY ? exp(-2.0 * best / ss) : 0.0;
    dens[t] = (float)((double)v_far + ((double)v_close - (double)v_far) * e);
}

// ---- subdivision ----

constexpr int SD_FINE = 18;   // finest level: cell indices are taken there once and shifted
constexpr int SD_COARSE = 6;  // leaves of this level or finer note their level in the coarse cell they lie in
constexpr int SD_SIDE = 1 << SD_COARSE;

// enters every leaf key (the lowest index of equal keys counts) and the levels below each coarse cell
__global__ void __launch_bounds__(256) k_leaf_enter(const uint64_t* __restrict__ keys, int64_t n,
                                                    uint64_t* __restrict__ table, uint32_t* __restrict__ idx, int bits,
                                                    uint64_t salt, uint32_t* __restrict__ coarse,
                                                    uint32_t* __restrict__ fail) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) {
        const uint64_t k = keys[t];
        const int l = (int)((k >> 57) & 31);
        const uint32_t lev = 1u << l;
        if (k != HT_EMPTY) atomicMin(idx + ht_enter(table, bits, salt, k, fail), (uint32_t)t);
        if (l >= SD_COARSE) {
            const int sh = l - SD_COARSE;
            const uint32_t x = (uint32_t)((k & kIMask) >> sh), y = (uint32_t)(((k >> 19) & kIMask) >> sh),
                           z = (uint32_t)(((k >> 38) & kIMask) >> sh);
            if (x < SD_SIDE && y < SD_SIDE && z < SD_SIDE) {
                uint32_t* w = coarse + (z * SD_SIDE + y) * SD_SIDE + x;
                if (!(*(volatile uint32_t*)w & lev)) atomicOr(w, lev);
            }
        }
    }
}

// Whether a point (from the root's corner) lies within thr of the box of cell (x, y, z) of level l.  Out of
// line: few points need it.
__device__ __noinline__ bool box_within(double root_size, int l, int x, int y, int z, double p0, double p1, double p2,
                                        double thr) {
    const double s = ldexp(root_size, -l);
    const double p[3] = {p0, p1, p2};
    const int ij[3] = {x, y, z};
    double d2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double b0 = (double)ij[a] * s, b1 = b0 + s;
        const double g = fmax(fmax(b0 - p[a], 0.0), p[a] - b1);
        d2 += g * g;
    }
    return !(d2 > thr * thr);
}

// One thread per LiDAR point, the points ordered by cell so that a warp's lanes look at much the same leaves:
// flags the leaves whose box lies within thr of it.  Cell indices: floors at the finest level, shifted (the
// levels' cell sizes are the root's times powers of two, so the quotients are too).  They and the distances come
// from the point's integer and fractional parts in finest-level units (the fractions in FP32); an index whose
// fraction is within 1e-5 of a step, and a distance within 2e-5 of the threshold (or any, for thresholds below
// 0.05 units or from 1e9 units), is taken from FP64.
__global__ void __launch_bounds__(256) k_subdiv_flags(const float4* __restrict__ pts, int64_t m, Frame f,
                                                      double root_size, double fine, double inv_fine,
                                                      uint32_t look_at, double thr,
                                                      const uint64_t* __restrict__ table,
                                                      const uint32_t* __restrict__ idx, int bits, uint64_t salt,
                                                      const uint32_t* __restrict__ coarse, uint8_t* __restrict__ split) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = t < m;
    const float4 pt = live ? pts[t] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float pc[3] = {pt.x, pt.y, pt.z};
    const double thr_d = fmin(thr * inv_fine, 1e9), thr_i = floor(thr_d);
    const float thr_u = (float)thr_d, thr_f = (float)(thr_d - thr_i);
    const bool huge = thr_d == 1e9;  // not the threshold any more: every index and distance from FP64
    double p[3];
    int flo[3], fhi[3], pi[3];
    float pf[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        p[a] = (double)pc[a] - f.root_min[a];
        const double u = fmin(fmax(p[a] * inv_fine, -1e9), 1e9);  // -1e9 for a point that is not a number
        const double ui = floor(u);
        pi[a] = (int)ui;
        pf[a] = (float)(u - ui);
        // floor((p -+ thr) / fine), kept just outside the grid where it leaves it
        auto index = [&](float fr, int64_t base, double x) {
            const float fl = floorf(fr), r = fr - fl;
            int64_t i = base + (int)fl;
            if (huge || r < 1e-5f || r > 1.0f - 1e-5f) {
                const double e = floor(x / fine);
                i = (int64_t)fmin(fmax(e, -1.0), (double)(1 << SD_FINE));
            }
            return (int)min(max(i, (int64_t)-1), (int64_t)1 << SD_FINE);
        };
        flo[a] = index(pf[a] - thr_f, (int64_t)pi[a] - (int64_t)thr_i, p[a] - thr);
        fhi[a] = index(pf[a] + thr_f, (int64_t)pi[a] + (int64_t)thr_i, p[a] + thr);
    }
    uint32_t levels = live ? look_at : 0u;  // the levels looked at from the points
    {
        // only levels that some coarse cell around the point holds
        int c0[3], c1[3], n = 1;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            c0[a] = max(flo[a] >> (SD_FINE - SD_COARSE), 0);
            c1[a] = min(fhi[a] >> (SD_FINE - SD_COARSE), SD_SIDE - 1);
            n *= max(c1[a] - c0[a] + 1, 0);
        }
        if (n == 0) levels = 0u;
        if (n <= 8) {
            uint32_t have = (1u << SD_COARSE) - 1u;
            for (int z = c0[2]; z <= c1[2]; ++z)
                for (int y = c0[1]; y <= c1[1]; ++y)
                    for (int x = c0[0]; x <= c1[0]; ++x) have |= __ldg(coarse + (z * SD_SIDE + y) * SD_SIDE + x);
            levels &= have;
        }
    }
    __syncwarp();
    const bool fp32 = thr_u >= 0.05f && thr_u < 1e9f;
    const float t2_lo = thr_u * thr_u * (1.0f - 2e-5f), t2_hi = thr_u * thr_u * (1.0f + 2e-5f);
    // The warp takes the levels and cells in step, so that lanes in the same cell ask for the same keys.
    for (uint32_t todo = __reduce_or_sync(0xffffffffu, levels); todo; todo &= todo - 1) {
        const int l = __ffs((int)todo) - 1, sh = SD_FINE - l;
        const int lim = (1 << l) - 1;
        int lo[3], n[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = max(flo[a] >> sh, 0);
            n[a] = max(min(fhi[a] >> sh, lim) - lo[a] + 1, 0);
        }
        const int64_t mine = (levels >> l) & 1u ? (int64_t)n[0] * n[1] * n[2] : 0;
        // distance along one axis to cell i, in finest units
        auto gap = [&](int a, int i) {
            const float below = (float)((i << sh) - pi[a]) - pf[a];
            const float above = (float)(pi[a] - ((i + 1) << sh)) + pf[a];
            return fmaxf(fmaxf(below, above), 0.0f);
        };
        int x = lo[0], y = lo[1], z = lo[2];
        for (int64_t i = 0; __any_sync(0xffffffffu, i < mine); ++i) {
            bool look = i < mine;
            if (look) {
                const float gx = gap(0, x), gy = gap(1, y), gz = gap(2, z);
                const float d2f = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
                if (fp32 && d2f > t2_hi)
                    look = false;
                else if (!fp32 || d2f >= t2_lo)
                    look = box_within(root_size, l, x, y, z, p[0], p[1], p[2], thr);
            }
            __syncwarp();
            const uint64_t key = ((uint64_t)l << 57) | ((uint64_t)z << 38) | ((uint64_t)y << 19) | (uint64_t)x;
            const uint32_t e = ht_find(table, bits, salt, key, look);
            if (e != ~0u) split[idx[e]] = 1;
            // the next cell, x fastest
            if (++x == lo[0] + n[0]) {
                x = lo[0];
                if (++y == lo[1] + n[1]) {
                    y = lo[1];
                    ++z;
                }
            }
        }
    }
}

constexpr int64_t FAR_CELLS = 4096;  // cells of the point grid a leaf looks into at most, else at all points

// One warp per leaf of the levels in `far`: flags the leaf if a point is within thr of its box.  The points lie in a
// grid of cells of half the threshold, so those in reach of a leaf (a third of the threshold or smaller, see
// subdivide_round) are in at most 7^3 cells: every lane probes one, the leaf's own first, and the warp tests the
// points of the cells found until one is in reach.  (k_subdiv_flags looks at (2 thr / leaf + 2)^3 cells for a point.)
// A point's cell is a monotone function of its coordinates, so the cells of the reach's two ends bound those of the
// points in it; where they are too many (coordinates that FP32 hardly resolves at the threshold, thresholds beyond
// the root), all points are tested.  Decided in FP32 from the leaf's centre split into two floats, within 2e-5
// of the threshold in FP64 by k_subdiv_flags' rule.
__global__ void __launch_bounds__(256) k_subdiv_far(const uint64_t* __restrict__ keys, int64_t n, uint32_t far, Frame f,
                                                    double root_size, double thr, const uint64_t* __restrict__ table,
                                                    const uint32_t* __restrict__ idx, int bits,
                                                    const uint64_t* __restrict__ cells, int cell_bits, uint64_t salt,
                                                    const uint32_t* __restrict__ cnt, const uint32_t* __restrict__ start,
                                                    const float4* __restrict__ pts, int64_t m, double inv_h,
                                                    uint8_t* __restrict__ split) {
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (t >= n) return;
    const uint64_t k = keys[t];
    const int l = (int)((k >> 57) & 31);
    if (!((far >> l) & 1u)) return;
    const int x = (int)(k & kIMask), y = (int)((k >> 19) & kIMask), z = (int)((k >> 38) & kIMask);
    // a key that is no cell of the grid is in no point's reach; of equal keys the lowest index counts
    if (k >> 62 || (x | y | z) >> l) return;
    const uint32_t e = ht_find(table, bits, salt, k, true);
    if (e == ~0u || (int64_t)idx[e] != t) return;
    const double s = ldexp(root_size, -l);
    const int at[3] = {x, y, z};
    float qh[3], ql[3];
    int c0[3], w[3];
    int64_t n_cell = 1;
    float big = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double b0 = f.root_min[a] + (double)at[a] * s, q = b0 + 0.5 * s;
        qh[a] = (float)q;
        ql[a] = (float)(q - (double)qh[a]);
        big = fmaxf(big, fabsf(qh[a]));
        // the cells k_cell_count gives to the ends of the reach
        const float lo = __double2float_rd(b0 - thr * (1.0 + 1e-9)), hi = __double2float_ru(b0 + s + thr * (1.0 + 1e-9));
        c0[a] = near_cell(lo, f.root_min[a], inv_h);
        w[a] = near_cell(hi, f.root_min[a], inv_h) - c0[a] + 1;
        n_cell *= min(max(w[a], 1), 1 << 20);
    }
    const float thr_u = (float)thr, half = (float)(0.5 * s);
    const bool fp32 = thr_u > 1e-15f && thr_u < 1e15f && thr_u > 1e-8f * big;
    const float t2_lo = thr_u * thr_u * (1.0f - 2e-5f), t2_hi = thr_u * thr_u * (1.0f + 2e-5f);
    auto reached = [&](float4 pt) {
        if (fp32) {
            auto gap = [&](float p, int a) {
                const float g = fabsf((p - qh[a]) - ql[a]) - half;
                return g <= 0.0f ? 0.0f : g;  // (not a number stays that)
            };
            const float gx = gap(pt.x, 0), gy = gap(pt.y, 1), gz = gap(pt.z, 2);
            const float d2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
            if (!(d2 <= t2_hi)) return false;
            if (d2 < t2_lo) return true;
        }
        const float pc[3] = {pt.x, pt.y, pt.z};
        double p[3];
        bool in = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            p[a] = (double)pc[a] - f.root_min[a];
            const double i0 = floor((p[a] - thr) / s), i1 = floor((p[a] + thr) / s);
            in = in && fmax(i0, -1.0) <= (double)at[a] && fmax(i1, -1.0) >= (double)at[a];
        }
        return in && box_within(root_size, l, x, y, z, p[0], p[1], p[2], thr);
    };
    // the points [e0, e0 + m0), the lanes in turn; true if one is in reach
    auto any_reached = [&](int64_t e0, int64_t m0) {
        for (int64_t j = 0; j < m0; j += 32)
            if (__any_sync(0xffffffffu, j + lane < m0 && reached(__ldg(pts + e0 + j + lane)))) return true;
        return false;
    };
    bool hit = false;
    if (n_cell > FAR_CELLS) {
        hit = any_reached(0, m);
    } else {
        const int nc = (int)n_cell;
        for (int b = 0; b < nc && !hit; b += 32) {
            const int c = (b + lane + nc / 2) % nc;
            const uint64_t key = cell_key(c0[0] + c % w[0], c0[1] + c / w[0] % w[1], c0[2] + c / (w[0] * w[1]));
            const uint32_t slot = ht_find(cells, cell_bits, salt, key, b + lane < nc);
            const uint32_t e0 = slot != ~0u ? start[slot] : 0u, m0 = slot != ~0u ? cnt[slot] : 0u;
            for (unsigned found = __ballot_sync(0xffffffffu, m0 != 0u); found && !hit; found &= found - 1) {
                const int src = __ffs((int)found) - 1;
                const int64_t from = __shfl_sync(0xffffffffu, e0, src), many = __shfl_sync(0xffffffffu, m0, src);
                hit = any_reached(from, min(many, m - from));
            }
        }
    }
    if (hit && lane == 0) split[t] = 1;
}

__global__ void k_subdiv_write(const uint64_t* __restrict__ keys, int64_t n, const uint8_t* __restrict__ split,
                               const uint32_t* __restrict__ pos_keep, const uint32_t* __restrict__ pos_split,
                               int64_t n_keep, int64_t n_split, uint64_t* __restrict__ out) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const uint64_t k = keys[v];
    if (!split[v]) {
        out[pos_keep[v]] = k;
        return;
    }
    const uint64_t lev = (k >> 57) & 31, i = k & kIMask, j = (k >> 19) & kIMask, kk = (k >> 38) & kIMask;
    for (int c = 0; c < 8; ++c)
        out[n_keep + (int64_t)c * n_split + pos_split[v]] =
            ((lev + 1) << 57) | ((2 * kk + ((c >> 2) & 1)) << 38) | ((2 * j + ((c >> 1) & 1)) << 19) |
            (2 * i + (c & 1));
}

__global__ void k_not(const uint8_t* __restrict__ a, int64_t n, uint32_t* __restrict__ yes, uint32_t* __restrict__ no) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    yes[t] = a[t] ? 1u : 0u;
    no[t] = a[t] ? 0u : 1u;
}

unsigned nb(int64_t n) { return (unsigned)((n + 255) / 256); }

// per-leaf densities [n][8] from shared corner values, and the transpose for gradients
__global__ void k_corner_gather(const uint32_t* __restrict__ index, int64_t n8, const float* __restrict__ corner,
                                float* __restrict__ dens) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n8) return;
    dens[t] = corner[index[t]];
}

__global__ void k_corner_scatter(const uint32_t* __restrict__ index, int64_t n8, const float* __restrict__ d_dens,
                                 float* __restrict__ d_corner) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n8) return;
    const float g = d_dens[t];
    if (g != 0.0f) atomicAdd(d_corner + index[t], g);
}

// levels of the keys (bit mask), to validate against max_level, and whether some key's index is outside its level's grid
__global__ void __launch_bounds__(256) k_levels(const uint64_t* __restrict__ keys, int64_t n, uint32_t* __restrict__ levels) {
    uint32_t lev = 0, outside = 0;
    for (int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x; t < n; t += (int64_t)gridDim.x * 256) {
        const uint64_t k = keys[t];
        const int l = (int)((k >> 57) & 31);
        lev |= 1u << l;
        outside |= (((k & kIMask) | ((k >> 19) & kIMask) | ((k >> 38) & kIMask)) >> l) != 0 ? 1u : 0u;
    }
    lev = __reduce_or_sync(0xffffffffu, lev);
    outside = __reduce_or_sync(0xffffffffu, outside);
    if ((threadIdx.x & 31) == 0 && (lev & ~*(volatile uint32_t*)levels)) atomicOr(levels, lev);
    if ((threadIdx.x & 31) == 0 && outside) levels[1] = 1u;
}

// A leaf is kept if its box top reaches z_min and some camera sees it (see the header).  A camera's verdict comes
// from the leaf's bounding sphere in FP32 where it is certain (the radius covers the rounding: 8e-6 of the
// coordinates' size), from the 8 corners in FP64 where the sphere meets a plane.  The block gathers the (leaf,
// camera) pairs left to FP64 and takes them densely: left in their own lanes, one of them holds the whole warp
// for two hundred FP64 instructions (500k leaves, six cameras: 217 -> 92 us).
__global__ void __launch_bounds__(256) k_visible(const uint64_t* __restrict__ keys, int64_t n, Frame f, double root_size,
                                                 const InitCam* __restrict__ cams, int n_cam, double z_min,
                                                 uint32_t* __restrict__ keep) {
    __shared__ uint32_t s_vis[256];
    __shared__ uint16_t s_leaf[256];
    __shared__ uint8_t s_cam[256];
    __shared__ int s_n;
    const int tid = threadIdx.x;
    const int64_t v = (int64_t)blockIdx.x * 256 + tid;
    s_vis[tid] = 0u;
    uint64_t open = 0;  // cameras left to FP64 (at most 64)
    const uint64_t k = v < n ? keys[v] : 0ull;
    if (v < n) {
        const double s = ldexp(root_size, -(int)((k >> 57) & 31));
        const double lo2 = f.root_min[2] + (double)((k >> 38) & kIMask) * s;
        if (lo2 + s >= z_min) {
            const float sf = (float)s;
            float ctr[3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                ctr[a] = fmaf((float)((k >> (19 * a)) & kIMask) + 0.5f, sf, (float)f.root_min[a]);
            const float size = fabsf(ctr[0]) + fabsf(ctr[1]) + fabsf(ctr[2]) + (float)root_size;
            for (int c = 0; c < n_cam; ++c) {
                const InitCam& C = cams[c];
                const float p0 = ctr[0] - C.tf[0], p1 = ctr[1] - C.tf[1], p2 = ctr[2] - C.tf[2];
                const float x = fmaf(C.Rf[0], p0, fmaf(C.Rf[3], p1, C.Rf[6] * p2));
                const float y = fmaf(C.Rf[1], p0, fmaf(C.Rf[4], p1, C.Rf[7] * p2));
                const float z = fmaf(C.Rf[2], p0, fmaf(C.Rf[5], p1, C.Rf[8] * p2));
                const float err = C.scale * 8e-6f * (size + fabsf(C.tf[0]) + fabsf(C.tf[1]) + fabsf(C.tf[2]));
                const float rad = fmaf(0.8661f * C.scale, sf, err);
                if (z + rad < C.nearf[0] || z - rad > C.farf[1]) continue;  // before near, or beyond far, with all corners
                if (z - rad > C.nearf[1]) {
                    // all corners behind near: the image's left and right sides, its top and bottom
                    const float l = fmaf(C.fxf, x, C.side[0] * z), r = fmaf(C.fxf, x, C.side[1] * z);
                    const float u = fmaf(C.fyf, y, C.side[2] * z), d = fmaf(C.fyf, y, C.side[3] * z);
                    if (l < -C.len[0] * rad || r > C.len[1] * rad || u < -C.len[2] * rad || d > C.len[3] * rad) continue;
                    if (z + rad < C.farf[0] && l > C.len[0] * err && r < -C.len[1] * err && u > C.len[2] * err &&
                        d < -C.len[3] * err) {
                        // the centre projects into the image, and the corners' rectangle holds it
                        s_vis[tid] = 1u;
                        open = 0;
                        break;
                    }
                }
                open |= 1ull << c;
            }
        }
    }
    // one open camera of every leaf that is not yet seen, in turn
    for (int turn = 0; turn < 64; ++turn) {
        if (tid == 0) s_n = 0;
        __syncthreads();
        const bool ask = open != 0 && s_vis[tid] == 0u;
        const unsigned b = __ballot_sync(0xffffffffu, ask);
        int base = 0;
        if ((tid & 31) == 0 && b) base = atomicAdd(&s_n, __popc(b));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (ask) {
            const int at = base + __popc(b & ((1u << (tid & 31)) - 1u));
            s_leaf[at] = (uint16_t)tid;
            s_cam[at] = (uint8_t)(__ffsll((long long)open) - 1);
            open &= open - 1;
        }
        __syncthreads();
        const int n_ask = s_n;
        if (n_ask == 0) break;
        if (tid < n_ask) {
            const uint64_t kk = keys[(int64_t)blockIdx.x * 256 + s_leaf[tid]];
            const double s = ldexp(root_size, -(int)((kk >> 57) & 31));
            const double lo[3] = {f.root_min[0] + (double)(kk & kIMask) * s,
                                  f.root_min[1] + (double)((kk >> 19) & kIMask) * s,
                                  f.root_min[2] + (double)((kk >> 38) & kIMask) * s};
            const InitCam& C = cams[s_cam[tid]];
            int behind = 0, beyond = 0;
            double u0 = INFINITY, u1 = -INFINITY, w0 = INFINITY, w1 = -INFINITY;
            for (int q = 0; q < 8; ++q) {
                const double p[3] = {lo[0] + ((q & 1) ? s : 0.0) - C.t[0], lo[1] + ((q & 2) ? s : 0.0) - C.t[1],
                                     lo[2] + ((q & 4) ? s : 0.0) - C.t[2]};
                // camera frame: R^T (p - t), R row-major camera -> world
                const double x = C.R[0] * p[0] + C.R[3] * p[1] + C.R[6] * p[2];
                const double y = C.R[1] * p[0] + C.R[4] * p[1] + C.R[7] * p[2];
                const double z = C.R[2] * p[0] + C.R[5] * p[1] + C.R[8] * p[2];
                behind += z < C.near_;
                beyond += z > C.far_;
                if (z >= C.near_) {
                    const double u = C.fx * x / z + C.cx, w = C.fy * y / z + C.cy;
                    u0 = fmin(u0, u);
                    u1 = fmax(u1, u);
                    w0 = fmin(w0, w);
                    w1 = fmax(w1, w);
                }
            }
            if (behind != 8 && beyond != 8 &&
                (behind > 0 || (u1 >= 0.0 && u0 <= (double)C.W && w1 >= 0.0 && w0 <= (double)C.H)))
                s_vis[s_leaf[tid]] = 1u;
        }
        __syncthreads();
    }
    if (v < n) keep[v] = s_vis[tid];
}

__global__ void k_compact_keys(const uint64_t* __restrict__ keys, int64_t n, const uint32_t* __restrict__ keep,
                               const uint32_t* __restrict__ pos, uint64_t* __restrict__ out) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n || !keep[v]) return;
    out[pos[v]] = keys[v];
}

}  // namespace

static Frame make_frame(const double* center, double root_size, int max_level);

cudaError_t visibility_prune(const uint64_t* keys, int64_t n, const double* center, double root_size,
                             const InitCam* cams_host, int n_cam, double z_min, uint64_t* out, int64_t* n_out,
                             Arena& ar, cudaStream_t s) {
    *n_out = 0;
    if (n <= 0) return cudaSuccess;
    const Frame f = make_frame(center, root_size, 0);
    InitCam* cams = ar.alloc<InitCam>((size_t)(n_cam > 0 ? n_cam : 1));
    uint32_t* keep = ar.alloc<uint32_t>(n);
    uint32_t* pos = ar.alloc<uint32_t>(n);
    uint32_t* tot = ar.alloc<uint32_t>(1);
    if (ar.err != cudaSuccess) return ar.err;
    cudaError_t e = cudaSuccess;
    if (n_cam > 0) e = cudaMemcpyAsync(cams, cams_host, sizeof(InitCam) * n_cam, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    k_visible<<<nb(n), 256, 0, s>>>(keys, n, f, root_size, cams, n_cam, z_min, keep);
    count_launches(1);
    e = scan_u32_to_u32(keep, pos, n, tot, ar, s);
    if (e != cudaSuccess) return e;
    k_compact_keys<<<nb(n), 256, 0, s>>>(keys, n, keep, pos, out);
    count_launches(1);
    uint32_t h = 0;
    e = cudaMemcpyAsync(&h, tot, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    *n_out = h;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t corner_gather(const uint32_t* index, int64_t n, const float* corner, float* dens, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_corner_gather<<<nb(n * 8), 256, 0, s>>>(index, n * 8, corner, dens);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t corner_scatter(const uint32_t* index, int64_t n, const float* d_dens, float* d_corner, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_corner_scatter<<<nb(n * 8), 256, 0, s>>>(index, n * 8, d_dens, d_corner);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t key_levels(const uint64_t* keys, int64_t n, uint32_t levels_host[2], Arena& ar, cudaStream_t s) {
    levels_host[0] = levels_host[1] = 0;
    if (n <= 0) return cudaSuccess;
    uint32_t* d = ar.alloc<uint32_t>(2);
    if (!d) return ar.err;
    cudaError_t e = cudaMemsetAsync(d, 0, 2 * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    k_levels<<<std::min<unsigned>(nb(n), 2u * (unsigned)sm_count()), 256, 0, s>>>(keys, n, d);
    count_launches(1);
    e = cudaMemcpyAsync(levels_host, d, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e;
}

cudaError_t shared_corners(const uint64_t* keys, int64_t n, int max_level, bool outside, uint64_t* grid_out,
                           uint32_t* index_out, int64_t* n_corners, Arena& ar, cudaStream_t s, bool* sort_timeout) {
    *n_corners = 0;
    *sort_timeout = false;
    if (n <= 0) return cudaSuccess;
    const int64_t m = n * 8;
    const int b = outside ? 21 : max_level + 1;  // bits of a coordinate
    uint64_t* k0 = ar.alloc<uint64_t>(m);
    uint64_t* k1 = ar.alloc<uint64_t>(m);
    uint32_t* v0 = ar.alloc<uint32_t>(m);
    uint32_t* v1 = ar.alloc<uint32_t>(m);
    uint32_t* first = ar.alloc<uint32_t>(m);
    uint32_t* pos = ar.alloc<uint32_t>(m);
    uint32_t* total = ar.alloc<uint32_t>(2);  // [0] distinct corners, [1] the sort's wait flag
    if (ar.err != cudaSuccess) return ar.err;
    cudaError_t e = cudaMemsetAsync(total + 1, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    k_corner_emit<<<nb(m), 256, 0, s>>>(keys, n, max_level, b, k0, v0);
    count_launches(1);
    uint64_t* kk = k0;
    uint32_t* vv = v0;
    e = radix_sort_u64(kk, vv, k1, v1, m, 3 * b, ar, s, total + 1);
    if (e != cudaSuccess) return e;
    k_corner_flag<<<nb(m), 256, 0, s>>>(kk, m, first);
    count_launches(1);
    e = scan_u32_to_u32(first, pos, m, total, ar, s);
    if (e != cudaSuccess) return e;
    k_corner_assign<<<nb(m), 256, 0, s>>>(kk, vv, first, pos, m, b, grid_out, index_out);
    count_launches(1);
    uint32_t h[2] = {0, 0};
    e = cudaMemcpyAsync(h, total, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    *n_corners = h[0];
    *sort_timeout = h[1] != 0;
    return e == cudaSuccess ? cudaGetLastError() : e;
}

static Frame make_frame(const double* center, double root_size, int max_level) {
    Frame f;
    for (int a = 0; a < 3; ++a) f.root_min[a] = center[a] - 0.5 * root_size;
    f.unit = ldexp(root_size, -max_level);
    return f;
}

cudaError_t soft_prior(const uint64_t* grid, int64_t n_corners, const double* center, double root_size, int max_level,
                       const float* cloud, int64_t m, float s_min, float v_close, float v_far, float* dens, Arena& ar,
                       cudaStream_t s, bool* no_room) {
    *no_room = false;
    if (n_corners <= 0) return cudaSuccess;
    const Frame f = make_frame(center, root_size, max_level);
    const double h = 3.0 * (double)s_min, inv_h = 1.0 / h;
    if (m <= 0) {
        k_soft_prior<<<nb(n_corners), 256, 0, s>>>(grid, n_corners, f, h, inv_h, nullptr, 0, 0, nullptr, nullptr, 0, nullptr,
                                                   s_min, v_close, v_far, dens);
        count_launches(1);
        return cudaGetLastError();
    }
    uint32_t* slot = ar.alloc<uint32_t>(m);
    uint32_t* rank = ar.alloc<uint32_t>(m);
    float4* pts = ar.alloc<float4>(m);
    const int held = ar.n;
    for (int more = 0; more < HT_TRIES; ++more) {
        ar.release(held);  // a table that was too small
        const int bits = std::min(ht_bits(m) + more, 32);
        const uint64_t salt = ht_salt(more);
        const size_t cap = (size_t)1 << bits;
        uint64_t* table = ar.alloc<uint64_t>(cap);
        uint32_t* cnt = ar.alloc<uint32_t>(cap + 2);  // then: points placed so far, a key without a slot
        uint32_t* start = ar.alloc<uint32_t>(cap);
        if (ar.err != cudaSuccess) return ar.err;
        cudaError_t e = cudaMemsetAsync(table, 0xff, cap * sizeof(uint64_t), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (cap + 2) * sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
        k_cell_count<true><<<nb(m), 256, 0, s>>>(cloud, m, f, h, inv_h, table, bits, salt, cnt, slot, rank, cnt + cap + 1);
        k_cell_alloc<<<(unsigned)(cap / 256), 256, 0, s>>>(cnt, (int64_t)cap, start, cnt + cap);
        k_cell_scatter<<<nb(m), 256, 0, s>>>(cloud, m, slot, rank, start, pts);
        k_soft_prior<<<nb(n_corners), 256, 0, s>>>(grid, n_corners, f, h, inv_h, table, bits, salt, cnt, start, m, pts, s_min,
                                                   v_close, v_far, dens);
        count_launches(4);
        uint32_t failed = 0;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&failed, cnt + cap + 1, sizeof(failed), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess || !failed) return e;
    }
    *no_room = true;  // no table up to eight times the capacity has room within HT_PROBES of every key's home
    return cudaSuccess;
}

// Levels at which a leaf looks for points: those where the cells in reach of a point may be more than FAR_FROM, and more
// than this share of the leaves.  Without them a threshold of some leaves' size runs for minutes ((2 thr / leaf + 2)^3
// cells a point and level, all in lockstep).  Both sides, all levels one way, in ms at thresholds of 3, 6, 12 and
// 16 of the finest leaves (512 to 39,304 cells): 30k leaves and 81k points 1.0, 4.7, 38, 87 from the points and 0.6, 0.3,
// 0.4, 0.3 from the leaves; 500k and 1.35M 4.4, 23, 163, 373 and 29, 17, 1.9, 1.8; 1M and 2.7M 8.1, 44, 321, 728
// and 314, 194, 4.6, 3.9 (points in many cells around a leaf and none in its reach cost the most).
constexpr double FAR_FROM = 512.0, FAR_SHARE = 1.0 / 100.0;

cudaError_t subdivide_round(const uint64_t* keys, int64_t n, uint32_t levels, const double* center, double root_size,
                            int max_level, const float* cloud, int64_t m, float thr, uint64_t* out, int64_t* n_out,
                            Arena& ar, cudaStream_t s, bool* no_room) {
    *n_out = n;
    *no_room = false;
    if (n <= 0) return cudaSuccess;
    const Frame f = make_frame(center, root_size, max_level);
    constexpr int COARSE = SD_SIDE * SD_SIDE * SD_SIDE;
    uint32_t* coarse = ar.alloc<uint32_t>(COARSE);
    uint8_t* split = ar.alloc<uint8_t>(n);
    uint32_t* yes = ar.alloc<uint32_t>(n);
    uint32_t* no = ar.alloc<uint32_t>(n);
    uint32_t* pos_s = ar.alloc<uint32_t>(n);
    uint32_t* pos_k = ar.alloc<uint32_t>(n);
    uint32_t* tot = ar.alloc<uint32_t>(3);  // split, kept, a key without a slot
    if (ar.err != cudaSuccess) return ar.err;
    uint32_t far = 0;
    for (int l = 0; l <= max_level; ++l) {
        const double side = std::min(2.0 * (double)thr / ldexp(root_size, -l) + 2.0, ldexp(1.0, l));
        if (side * side * side > std::max(FAR_FROM, FAR_SHARE * (double)n)) far |= levels & (1u << l);
    }
    uint32_t hd[3] = {0, 0, 0};
    const int held = ar.n;
    for (int more = 0; more < HT_TRIES; ++more) {
        ar.release(held);  // a table that was too small
        const uint64_t salt = ht_salt(more);
        cudaError_t e = cudaMemsetAsync(split, 0, n, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(tot, 0, 3 * sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
        if (m > 0) {
            // The points ordered by cells of 16 thresholds (flags kernel with the points as they come 1,300 us, cells of
            // 1, 4, 16, 64 thresholds 1,284, 924, 730, 714 us, and 75 to 110 us for the order; since the levels come
            // as an argument 420 us with 16): a point that finds no
            // slot counts in its last slot, the order is all that matters.  Where leaves look for points, cells of half
            // a threshold, in which every point has its slot.
            const int pbits = std::min(ht_bits(m) + (far ? more : 0), 32), bits = ht_bits(n) + more;
            const size_t pcap = (size_t)1 << pbits, cap = (size_t)1 << bits;
            uint64_t* cells = ar.alloc<uint64_t>(pcap);
            uint32_t* cnt = ar.alloc<uint32_t>(pcap + 2);
            uint32_t* start = ar.alloc<uint32_t>(pcap);
            uint32_t* slot = ar.alloc<uint32_t>(m);
            uint32_t* rank = ar.alloc<uint32_t>(m);
            float4* pts = ar.alloc<float4>(m);
            uint64_t* table = ar.alloc<uint64_t>(cap);
            uint32_t* idx = ar.alloc<uint32_t>(cap);
            if (ar.err != cudaSuccess) return ar.err;
            e = cudaMemsetAsync(cells, 0xff, pcap * sizeof(uint64_t), s);
            if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (pcap + 2) * sizeof(uint32_t), s);
            if (e == cudaSuccess) e = cudaMemsetAsync(table, 0xff, cap * sizeof(uint64_t), s);
            if (e == cudaSuccess) e = cudaMemsetAsync(idx, 0xff, cap * sizeof(uint32_t), s);
            if (e == cudaSuccess) e = cudaMemsetAsync(coarse, 0, COARSE * sizeof(uint32_t), s);
            if (e != cudaSuccess) return e;
            const double h = far ? 0.5 * std::min((double)thr, 4.0 * root_size)
                                 : std::max(16.0 * (double)thr, ldexp(root_size, -SD_FINE));
            k_cell_count<false><<<nb(m), 256, 0, s>>>(cloud, m, f, h, 1.0 / h, cells, pbits, salt, cnt, slot, rank,
                                                      far ? tot + 2 : cnt + pcap + 1);
            k_cell_alloc<<<(unsigned)(pcap / 256), 256, 0, s>>>(cnt, (int64_t)pcap, start, cnt + pcap);
            k_cell_scatter<<<nb(m), 256, 0, s>>>(cloud, m, slot, rank, start, pts);
            k_leaf_enter<<<nb(n), 256, 0, s>>>(keys, n, table, idx, bits, salt, coarse, tot + 2);
            count_launches(4);
            if (levels & ~far) {
                k_subdiv_flags<<<nb(m), 256, 0, s>>>(pts, m, f, root_size, ldexp(root_size, -SD_FINE),
                                                     (double)(1 << SD_FINE) / root_size, levels & ~far, thr, table, idx,
                                                     bits, salt, coarse, split);
                count_launches(1);
            }
            if (far) {
                k_subdiv_far<<<(unsigned)((n + 7) / 8), 256, 0, s>>>(keys, n, far, f, root_size, thr, table, idx, bits, cells,
                                                                     pbits, salt, cnt, start, pts, m, 1.0 / h, split);
                count_launches(1);
            }
        }
        k_not<<<nb(n), 256, 0, s>>>(split, n, yes, no);
        count_launches(1);
        e = scan_u32_to_u32(yes, pos_s, n, tot, ar, s);
        if (e == cudaSuccess) e = scan_u32_to_u32(no, pos_k, n, tot + 1, ar, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hd, tot, sizeof(hd), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
        if (!hd[2]) break;
    }
    if (hd[2]) {  // see soft_prior
        *no_room = true;
        *n_out = 0;
        return cudaSuccess;
    }
    const int64_t n_split = hd[0], n_keep = hd[1];
    k_subdiv_write<<<nb(n), 256, 0, s>>>(keys, n, split, pos_k, pos_s, n_keep, n_split, out);
    count_launches(1);
    *n_out = n_keep + 8 * n_split;
    return cudaGetLastError();
}

}  // namespace dv

namespace dv {

namespace {

// leaf t of the uniform grid: (i, j, k) = (t mod n, (t / n) mod n, t / n^2), n = 2^level
__global__ void k_asset_grid(int level, float v_init, int64_t n_leaf, uint64_t* __restrict__ keys,
                             float4* __restrict__ dens) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_leaf) return;
    const uint64_t n = 1ull << level;
    const uint64_t i = (uint64_t)t & (n - 1), j = ((uint64_t)t >> level) & (n - 1), k = (uint64_t)t >> (2 * level);
    keys[t] = ((uint64_t)level << 57) | (k << 38) | (j << 19) | i;
    const float4 v = make_float4(v_init, v_init, v_init, v_init);
    dens[2 * t] = v;
    dens[2 * t + 1] = v;
}

}  // namespace

cudaError_t asset_grid(int level, float v_init, uint64_t* keys, float* dens, cudaStream_t s) {
    const int64_t n = (int64_t)1 << (3 * level);
    k_asset_grid<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(level, v_init, n, keys, reinterpret_cast<float4*>(dens));
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace dv
