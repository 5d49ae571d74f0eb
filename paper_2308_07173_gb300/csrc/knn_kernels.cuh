// The search and covariance kernels, shared by knn_cov.cu (whole-map
// searches) and knn_window.cu (searches restricted to a window, WIN = true):
// each translation unit instantiates one window variant, so the whole-map
// kernels carry no window code and the two compile in parallel.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>
#include <utility>

#include "pc_device.cuh"
#include "pc_internal.h"
#include "pc_search.cuh"

using namespace pcdev;

namespace {

typedef unsigned long long u64;

__device__ __forceinline__ u64 umin64(u64 a, u64 b) { return a < b ? a : b; }
__device__ __forceinline__ u64 umax64(u64 a, u64 b) { return a < b ? b : a; }

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Bitonic sort of one key per lane into DESCENDING lane order.
__device__ __forceinline__ u64 sort32_desc(u64 x, int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            u64 y = __shfl_xor_sync(FULL, x, stride);
            bool desc_block = (lane & size) == 0;  // all lanes at size 32
            bool lower = (lane & stride) == 0;
            x = (lower == desc_block) ? umax64(x, y) : umin64(x, y);
        }
    }
    return x;
}

// Bitonic merge of a bitonic lane sequence into ASCENDING lane order.
__device__ __forceinline__ u64 merge32_asc(u64 x, int lane) {
#pragma unroll
    for (int stride = 16; stride > 0; stride >>= 1) {
        u64 y = __shfl_xor_sync(FULL, x, stride);
        x = ((lane & stride) == 0) ? umin64(x, y) : umax64(x, y);
    }
    return x;
}

template <int SLOTS>
struct SearchState {
    u64 L[SLOTS];  // lane l: rank l (slot 0) and rank 32 + l (slot 1)
    u64 kth;       // warp-uniform: the rank k-1 key, EMPTY_KEY until k exist
    int npend;     // warp-uniform: survivors staged in shared memory
};

template <int SLOTS>
__device__ __forceinline__ void state_reset(SearchState<SLOTS>& S) {
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) S.L[s] = EMPTY_KEY;
    S.kth = EMPTY_KEY;
    S.npend = 0;
}

template <int SLOTS>
__device__ __forceinline__ u64 topk_rank(const SearchState<SLOTS>& S, int r) {
    u64 v = (SLOTS == 2 && r >= 32) ? S.L[SLOTS - 1] : S.L[0];
    return __shfl_sync(FULL, v, r & 31);
}

// Merge 32 staged keys (one per lane, any order) into the sorted top list.
// A ascending + B descending -> min(A, B) is bitonic and holds the smallest
// |A| of A u B; for two slots the 64-list [L0, min(L1, c)] is bitonic.
template <int SLOTS>
__device__ __forceinline__ void topk_merge(SearchState<SLOTS>& S, u64 c, int k, int lane) {
    c = sort32_desc(c, lane);
    if (SLOTS == 1) {
        S.L[0] = merge32_asc(umin64(S.L[0], c), lane);
    } else {
        u64 b = umin64(S.L[SLOTS - 1], c);
        u64 lo = umin64(S.L[0], b), hi = umax64(S.L[0], b);
        S.L[0] = merge32_asc(lo, lane);
        S.L[SLOTS - 1] = merge32_asc(hi, lane);
    }
    S.kth = topk_rank(S, k - 1);
}

template <int SLOTS>
__device__ __forceinline__ void offer(SearchState<SLOTS>& S, bool pass, u64 key, u64* pend, int k,
                                      int lane) {
    unsigned m = __ballot_sync(FULL, pass);
    if (m == 0u) return;
    if (pass) pend[S.npend + __popc(m & lanemask_lt())] = key;
    S.npend += __popc(m);
    __syncwarp();
    if (S.npend >= 32) {
        topk_merge(S, pend[lane], k, lane);
        __syncwarp();
        const int rest = S.npend - 32;
        if (lane < rest) pend[lane] = pend[32 + lane];
        __syncwarp();
        S.npend = rest;
    }
}

template <int SLOTS>
__device__ __forceinline__ void flush(SearchState<SLOTS>& S, u64* pend, int k, int lane) {
    if (S.npend > 0) {
        u64 c = lane < S.npend ? pend[lane] : EMPTY_KEY;
        topk_merge(S, c, k, lane);
        S.npend = 0;
    }
    __syncwarp();
}

// One pass over up to 32 point ranges (one per lane): every point becomes a
// candidate, 32 per step, each lane finding its owning range by a binary
// search over the warp's exclusive prefix of counts.  Keys carry the point's
// index plus ibase (the appended-points grid numbers its points after the
// main grid's).
template <int SLOTS>
__device__ __forceinline__ void scan_ranges(const Grid& g, float qx, float qy, float qz,
                                            uint32_t start, uint32_t cnt, float tau,
                                            SearchState<SLOTS>& S, u64* pend, int k, int lane,
                                            uint32_t ibase) {
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
    }
    const uint32_t total = __shfl_sync(FULL, incl, 31);
    const uint32_t excl = incl - cnt;
    for (uint32_t cb = 0; cb < total; cb += 32) {
        const uint32_t t = cb + lane;
        int j = 0;
#pragma unroll
        for (int s = 16; s >= 1; s >>= 1) {
            uint32_t e = __shfl_sync(FULL, excl, j + s);
            if (e <= t) j += s;
        }
        const uint32_t st = __shfl_sync(FULL, start, j);
        const uint32_t ej = __shfl_sync(FULL, excl, j);
        bool pass = false;
        u64 key = EMPTY_KEY;
        if (t < total) {
            const float4 p = __ldg(&g.pts[st + (t - ej)]);
            const float d2 = sqdist_pinned(qx, qy, qz, p.x, p.y, p.z);
            key = ((u64)__float_as_uint(d2) << 32) | (u64)(__float_as_uint(p.w) + ibase);
            pass = (d2 <= tau) && (key < S.kth) && (!g.windowed || in_window(g, p));
        }
        offer(S, pass, key, pend, k, lane);
    }
}

// Lower bound on the binary32 d2 from q to any point of cell (cx, cy, cz);
// same margin argument as certified_tau.
__device__ __forceinline__ float cell_lower_bound2(const Grid& g, float qx, float qy, float qz,
                                                   int cx, int cy, int cz) {
    float qm = fmaxf(fabsf(qx), fmaxf(fabsf(qy), fabsf(qz)));
    int cm = max(cx, max(cy, cz)) + 1;
    float eta = 0x1p-20f * (g.coord_scale + qm + (float)cm * g.h);
    float s = 0.0f;
    {
        float lo = g.ox + (float)cx * g.h, hi = g.ox + (float)(cx + 1) * g.h;
        float d = fmaxf(fmaxf(lo - qx, qx - hi), 0.0f) - eta;
        if (d > 0.0f) s = s + d * d;
    }
    {
        float lo = g.oy + (float)cy * g.h, hi = g.oy + (float)(cy + 1) * g.h;
        float d = fmaxf(fmaxf(lo - qy, qy - hi), 0.0f) - eta;
        if (d > 0.0f) s = s + d * d;
    }
    {
        float lo = g.oz + (float)cz * g.h, hi = g.oz + (float)(cz + 1) * g.h;
        float d = fmaxf(fmaxf(lo - qz, qz - hi), 0.0f) - eta;
        if (d > 0.0f) s = s + d * d;
    }
    return s * (1.0f - 0x1p-20f);
}

// The rows of the box [lx, lx + ex) x [ly, ly + ey) x [lz, lz + ez) through
// the row index, one row per lane and 32 per step: each is one range of pts,
// cut to the chord of the smaller of tau and the current k-th distance.  A
// box of half-width R cells costs ~(2R + 1) row lookups per level of z where
// the hash costs (2R + 1)^2 cell probes, so the search can widen to any
// distance; the per-row cut drops the rows that the k found so far exclude.
// Measured on a 131k-point scan searched with itself, k = 20, where the 700 to
// 1,000 queries in its sparse rim find their 20th neighbour up to 100 cells away
// and, cell by cell, ended in the scan of every occupied cell: 9.8-36 ms by
// cells, 0.16-0.25 ms by rows from k_knn_rest.
template <int SLOTS>
__device__ void scan_rows(const Grid& g, float qx, float qy, float qz, int lx, int ly, int lz,
                          int ex, int ey, int ez, float eta, float tau, SearchState<SLOTS>& S, u64* pend,
                          int k, int lane, uint32_t ibase) {
    const int64_t nrows = (int64_t)ey * ez;
    for (int64_t base = 0; base < nrows; base += 32) {
        const int64_t r = base + lane;
        uint2 v = make_uint2(0u, 0u);
        if (r < nrows) {
            const int cz = lz + (int)(r / ey), cy = ly + (int)(r % ey);
            const float kd = S.kth == EMPTY_KEY ? INFINITY : __uint_as_float((uint32_t)(S.kth >> 32));
            const float tm = fminf(tau, kd);
            v = row_part(g, qx, qy, qz, cy, cz, lx, lx + ex - 1, eta, tm, tm * (1.0f + 0x1p-18f));
        }
        scan_ranges(g, qx, qy, qz, v.x, v.y, tau, S, pend, k, lane, ibase);
    }
}

template <int SLOTS>
__device__ void scan_box(const Grid& g, float qx, float qy, float qz, int lx, int ly, int lz,
                         int ex, int ey, int ez, float tau, SearchState<SLOTS>& S, u64* pend,
                         int k, int lane, uint32_t ibase) {
    const int ncl = ex * ey * ez;
    for (int base = 0; base < ncl; base += 32) {
        const int c = base + lane;
        uint32_t start = 0u, cnt = 0u;
        if (c < ncl) {
            const int cx = lx + c % ex;
            const int r = c / ex;
            const int cy = ly + r % ey;
            const int cz = lz + r / ey;
            const uint2 v = lookup_cell(g, pack_key(cx, cy, cz, g.bx, g.by));
            start = v.x;
            cnt = v.y;
        }
        scan_ranges(g, qx, qy, qz, start, cnt, tau, S, pend, k, lane, ibase);
    }
}

template <int SLOTS>
__device__ void scan_all_cells(const Grid& g, float qx, float qy, float qz, SearchState<SLOTS>& S,
                               u64* pend, int k, int lane, uint32_t ibase) {
    const u64 mx = (1ull << g.bx) - 1ull, my = (1ull << g.by) - 1ull;
    for (int64_t ub = 0; ub < g.ncells; ub += 32) {
        const int64_t u = ub + lane;
        uint32_t start = 0u, cnt = 0u;
        if (u < g.ncells) {
            const u64 key = g.cell_keys[u];
            const int cx = (int)(key & mx), cy = (int)((key >> g.bx) & my),
                      cz = (int)(key >> (g.bx + g.by));
            const float lb2 = cell_lower_bound2(g, qx, qy, qz, cx, cy, cz);
            const float kd = S.kth == EMPTY_KEY ? INFINITY : __uint_as_float((uint32_t)(S.kth >> 32));
            const bool win = cx >= g.wlx && cx <= g.whx && cy >= g.wly && cy <= g.why &&
                             cz >= g.wlz && cz <= g.whz;
            if (win && lb2 <= kd) {
                start = g.cell_start[u];
                cnt = g.cell_start[u + 1] - start;
            }
        }
        scan_ranges(g, qx, qy, qz, start, cnt, INFINITY, S, pend, k, lane, ibase);
    }
}

// The cell box of radius rho around q on one grid, clamped to its window
// range (the whole grid when no window is set), and the certified tau of
// the unclamped box.
struct WarpBox {
    int lx, ly, lz;
    int ex, ey, ez;
    int64_t ncl;
    float tau, eta;
    bool all;  // the box holds the whole window range: nothing is left outside it
};

__device__ __forceinline__ WarpBox warp_box(const Grid& g, float qx, float qy, float qz, float rho) {
    const int lx = cell_of(__fsub_rn(qx, rho), g.ox, g.inv_h);
    const int hx = cell_of(__fadd_rn(qx, rho), g.ox, g.inv_h);
    const int ly = cell_of(__fsub_rn(qy, rho), g.oy, g.inv_h);
    const int hy = cell_of(__fadd_rn(qy, rho), g.oy, g.inv_h);
    const int lz = cell_of(__fsub_rn(qz, rho), g.oz, g.inv_h);
    const int hz = cell_of(__fadd_rn(qz, rho), g.oz, g.inv_h);
    WarpBox b;
    b.tau = certified_tau(g, qx, qy, qz, lx, hx, ly, hy, lz, hz);
    b.lx = max(lx, g.wlx);
    b.ly = max(ly, g.wly);
    b.lz = max(lz, g.wlz);
    b.ex = max(min(hx, g.whx) - b.lx + 1, 0);
    b.ey = max(min(hy, g.why) - b.ly + 1, 0);
    b.ez = max(min(hz, g.whz) - b.lz + 1, 0);
    b.ncl = (int64_t)b.ex * b.ey * b.ez;
    const int cm = max(max(max(abs(lx), abs(hx + 1)), max(abs(ly), abs(hy + 1))), max(abs(lz), abs(hz + 1)));
    const float qm = fmaxf(fabsf(qx), fmaxf(fabsf(qy), fabsf(qz)));
    b.eta = 0x1p-20f * (g.coord_scale + qm + (float)cm * g.h);
    b.all = lx <= g.wlx && hx >= g.whx && ly <= g.wly && hy >= g.why && lz <= g.wlz && hz >= g.whz;
    return b;
}

// Distance from q to the cells that a search may answer from (the window's, or
// the whole grid): no point lies nearer.
__device__ __forceinline__ float range_gap(const Grid& g, float qx, float qy, float qz) {
    auto gap = [&](float q, float o, int lo, int hi) {
        return fmaxf(fmaxf(o + (float)lo * g.h - q, q - (o + (float)(hi + 1) * g.h)), 0.0f);
    };
    const float x = gap(qx, g.ox, g.wlx, g.whx), y = gap(qy, g.oy, g.wly, g.why), z = gap(qz, g.oz, g.wlz, g.whz);
    return sqrtf(x * x + y * y + z * z);
}

// Whether the widening search may scan this box.  Through the row index (and
// where the exact scan of every occupied cell is allowed to follow) the cost
// is its rows: up to as many as there are occupied cells, beyond which that
// scan is the cheaper one.  Otherwise its cells, up to max_box_cells.
__device__ __forceinline__ bool box_allowed(const Grid& g, const WarpBox& b) {
    if (g.dstart && g.exhaustive)
        return (int64_t)b.ey * b.ez <= max(g.ncells, (int64_t)4096) || b.ncl <= (int64_t)g.max_box_cells;
    return b.ncl <= (int64_t)g.max_box_cells;
}

// Whether a group (k <= 32) searches a box of so many cells in so many rows.
__device__ __forceinline__ bool group_allowed(const Grid& g, int64_t ncl, int64_t nrows) {
    return ncl <= 4096 && nrows <= 256 && (g.dstart || ncl <= 256);
}

// Where the exact scan may not follow (exhaustive = 0), the radii decide which
// queries are answered.  Those of a group search follow the counts it finds, so
// for the queries it leaves k_knn_rest has LIMITED_RADII fixed ones, in boxes as
// large as a group's: LIMITED_START times the calibrated radius, LIMITED_STEP
// times the one before.  Then it widens from LIMITED_START up to max_box_cells.
constexpr int LIMITED_RADII = 3;
constexpr float LIMITED_START = 1.46f, LIMITED_STEP = 1.8f;

template <int SLOTS>
__device__ __forceinline__ void scan_warp_box(const Grid& g, float qx, float qy, float qz, const WarpBox& b, float tau,
                                              SearchState<SLOTS>& S, u64* pend, int k, int lane, uint32_t ibase) {
    if (b.ncl <= 0) return;
    if (g.dstart)
        scan_rows(g, qx, qy, qz, b.lx, b.ly, b.lz, b.ex, b.ey, b.ez, b.eta, tau, S, pend, k, lane, ibase);
    else
        scan_box(g, qx, qy, qz, b.lx, b.ly, b.lz, b.ex, b.ey, b.ez, tau, S, pend, k, lane, ibase);
}

// Exact k nearest neighbours of one query (warp-uniform control flow).
// Returns SEARCH_OK, SEARCH_LIMIT (max_box_cells reached with exhaustive =
// 0) or SEARCH_SHORT (the exhaustive scan found fewer than k points: the
// window holds fewer than k).  With DEL the search runs over the union of
// g and the appended-points grid dg, whose point j is g.m + j: every
// attempt scans both grids' boxes of the same radius, filtered by the
// smaller of their two certified taus (a point of either grid outside its
// box lies beyond both), and the exhaustive scan covers both grids.  FIXED: the
// first attempts have the fixed radii above, from rho, and the widening proper
// starts from rho1.
constexpr int SEARCH_OK = 0, SEARCH_LIMIT = 1, SEARCH_SHORT = 2;
template <int SLOTS, bool DEL, bool FIXED = false>
__device__ int knn_search(const Grid& g, const Grid& dg, float qx, float qy, float qz, int k, float& rho,
                          SearchState<SLOTS>& S, u64* pend, int lane, float rho1 = 0.0f) {
    int fixed = FIXED ? LIMITED_RADII : 0;
    for (int attempt = 0; attempt < 40 + LIMITED_RADII; ++attempt) {
        const WarpBox b = warp_box(g, qx, qy, qz, rho);
        WarpBox d = b;
        float tau = b.tau;
        bool all = b.all;
        const bool group = attempt < fixed;
        auto allowed = [&](const Grid& gr, const WarpBox& x) {
            return group ? group_allowed(gr, x.ncl, (int64_t)x.ey * x.ez) : box_allowed(gr, x);
        };
        bool may = allowed(g, b);
        if (DEL) {
            d = warp_box(dg, qx, qy, qz, rho);
            tau = fminf(tau, d.tau);
            all = all && d.all;
            may = may && allowed(dg, d);
        }
        if (!may) {
            if (!group) break;
            fixed = 0;
            rho = rho1;
            continue;
        }
        if (all && g.exhaustive) tau = INFINITY;  // no point lies outside the box
        state_reset(S);
        scan_warp_box(g, qx, qy, qz, b, tau, S, pend, k, lane, 0u);
        if (DEL) scan_warp_box(dg, qx, qy, qz, d, tau, S, pend, k, lane, (uint32_t)g.m);
        flush(S, pend, k, lane);
        if (S.kth != EMPTY_KEY) return SEARCH_OK;
        if (all && g.exhaustive) return SEARCH_SHORT;  // every point of the window was seen
        if (group) {
            rho = attempt + 1 < fixed ? rho * LIMITED_STEP : rho1;
            continue;
        }
        if (g.exhaustive && b.ncl <= 0 && (!DEL || d.ncl <= 0)) {  // to where the points begin
            rho = fminf(fmaxf(2.0f * rho, rho + fminf(range_gap(g, qx, qy, qz), DEL ? range_gap(dg, qx, qy, qz) : INFINITY)),
                        1e30f);
            continue;
        }
        int found = 0;
#pragma unroll
        for (int s = 0; s < SLOTS; ++s) found += __popc(__ballot_sync(FULL, S.L[s] != EMPTY_KEY));
        float f = 1.3f * sqrtf((float)k / (float)max(found, 1));
        f = fminf(fmaxf(f, 1.5f), 4.0f);
        rho = fminf(fmaxf(rho, 1e-3f * g.h) * f, 1e30f);
    }
    if (!g.exhaustive) return SEARCH_LIMIT;
    if (lane == 0) atomicAdd(&g.stats[2], 1ull);
    state_reset(S);
    scan_all_cells(g, qx, qy, qz, S, pend, k, lane, 0u);
    if (DEL) scan_all_cells(dg, qx, qy, qz, S, pend, k, lane, (uint32_t)g.m);
    flush(S, pend, k, lane);
    return S.kth != EMPTY_KEY ? SEARCH_OK : SEARCH_SHORT;
}

// ---------------------------------------------------------------- covariance

// Unit null vector of the symmetric 3x3 matrix with rows r0, r1, r2 (of
// rank 2 up to rounding): the cross product of two rows is orthogonal to
// both, and of the three pairs the one with the largest cross product is
// the best conditioned.  A zero matrix gives e_z.
__host__ __device__ __forceinline__ float3 cross3(float3 a, float3 b) {
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__host__ __device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

__host__ __device__ __forceinline__ float3 null_vector(float3 r0, float3 r1, float3 r2) {
    const float3 c01 = cross3(r0, r1), c02 = cross3(r0, r2), c12 = cross3(r1, r2);
    const float d01 = dot3(c01, c01), d02 = dot3(c02, c02), d12 = dot3(c12, c12);
    float3 c = c01;
    float d = d01;
    if (d02 > d) { c = c02; d = d02; }
    if (d12 > d) { c = c12; d = d12; }
    if (!(d > 0.0f)) return make_float3(0.0f, 0.0f, 1.0f);
    const float inv = 1.0f / sqrtf(d);
    return make_float3(c.x * inv, c.y * inv, c.z * inv);
}

// Unit eigenvector of the smallest eigenvalue of a symmetric 3x3 matrix A,
// in closed form, binary32.  The matrix is first scaled by an exact power
// of two; a zero matrix gives e_z.
//
// Eigenvalues by the trigonometric form (Smith 1961): with m = tr(A)/3,
// B = A - m I, p = sqrt(tr(B^2)/6) and r = det(B)/(2 p^3) in [-1, 1],
// phi = acos(r)/3, the eigenvalues are m + 2p cos(phi + 2 pi j/3),
// j = 0 (largest), 1 (smallest), 2.  Which one is computed decides the
// accuracy (the hybrid of Kopp 2008, "Efficient numerical diagonalization
// of hermitian 3x3 matrices"):
// * r < 0: the middle eigenvalue is nearer the largest, so the smallest is
//   the isolated one (lambda2 - lambda3 >= (lambda1 - lambda3)/2) and its
//   value has a bounded derivative in r.  The normal is the null vector of
//   A - lambda3 I.
// * r >= 0: the two smallest are the close pair; the largest is isolated
//   and accurate, its eigenvector e1 is the null vector of A - lambda1 I,
//   and the normal is the smaller eigenvector of A restricted to the plane
//   orthogonal to e1 (a 2x2 problem solved by one Jacobi rotation, exact
//   for any separation of the pair, a repeated pair included).
// Either way the normal's error is ~ u ||A|| / (lambda2 - lambda3), the
// perturbation bound itself, as for an iterative solver.
__host__ __device__ float3 min_eigvec(float a00, float a01, float a02, float a11, float a12, float a22) {
    const float amax = fmaxf(fmaxf(fabsf(a00), fabsf(a11)),
                             fmaxf(fabsf(a22), fmaxf(fmaxf(fabsf(a01), fabsf(a02)), fabsf(a12))));
    if (!(amax > 0.0f) || !isfinite(amax)) return make_float3(0.0f, 0.0f, 1.0f);
    int e;
    frexpf(amax, &e);
    const float sc = ldexpf(1.0f, -e);
    a00 *= sc; a01 *= sc; a02 *= sc; a11 *= sc; a12 *= sc; a22 *= sc;
    const float m = (a00 + a11 + a22) / 3.0f;
    const float b00 = a00 - m, b11 = a11 - m, b22 = a22 - m;
    const float p2 = (b00 * b00 + b11 * b11 + b22 * b22 + 2.0f * (a01 * a01 + a02 * a02 + a12 * a12)) / 6.0f;
    if (!(p2 > 0.0f)) return make_float3(0.0f, 0.0f, 1.0f);  // A = m I: every direction
    const float p = sqrtf(p2);
    const float det = b00 * (b11 * b22 - a12 * a12) - a01 * (a01 * b22 - a12 * a02) + a02 * (a01 * a12 - b11 * a02);
    const float r = fminf(fmaxf(det / (2.0f * p2 * p), -1.0f), 1.0f);
    const float phi = acosf(r) / 3.0f;
    if (r < 0.0f) {
        const float l3 = m + 2.0f * p * cosf(phi + 2.09439510f);
        return null_vector(make_float3(a00 - l3, a01, a02), make_float3(a01, a11 - l3, a12),
                           make_float3(a02, a12, a22 - l3));
    }
    const float l1 = m + 2.0f * p * cosf(phi);
    const float3 e1 = null_vector(make_float3(a00 - l1, a01, a02), make_float3(a01, a11 - l1, a12),
                                  make_float3(a02, a12, a22 - l1));
    // orthonormal u, v spanning the plane orthogonal to e1
    const float ax = fabsf(e1.x), ay = fabsf(e1.y), az = fabsf(e1.z);
    const float3 w = (ax <= ay && ax <= az) ? make_float3(1.0f, 0.0f, 0.0f)
                   : (ay <= az ? make_float3(0.0f, 1.0f, 0.0f) : make_float3(0.0f, 0.0f, 1.0f));
    float3 u = cross3(e1, w);
    const float iu = 1.0f / sqrtf(dot3(u, u));
    u = make_float3(u.x * iu, u.y * iu, u.z * iu);
    const float3 v = cross3(e1, u);
    const float3 Au = make_float3(a00 * u.x + a01 * u.y + a02 * u.z, a01 * u.x + a11 * u.y + a12 * u.z,
                                  a02 * u.x + a12 * u.y + a22 * u.z);
    const float3 Av = make_float3(a00 * v.x + a01 * v.y + a02 * v.z, a01 * v.x + a11 * v.y + a12 * v.z,
                                  a02 * v.x + a12 * v.y + a22 * v.z);
    const float suu = dot3(u, Au), suv = dot3(v, Au), svv = dot3(v, Av);
    // the rotation (c, s) that diagonalises [[suu, suv], [suv, svv]] (the
    // smaller root t of t^2 + 2 t theta - 1 = 0, Golub & Van Loan sec. 8.5):
    // eigenvector (c, -s) for suu - t suv, (s, c) for svv + t suv
    float c = 1.0f, sn = 0.0f, lu = suu, lv = svv;
    if (suv != 0.0f) {
        const float theta = (svv - suu) / (2.0f * suv);
        const float at = fabsf(theta);
        const float t = at > 1e18f ? 0.5f / theta : copysignf(1.0f, theta) / (at + sqrtf(theta * theta + 1.0f));
        c = 1.0f / sqrtf(t * t + 1.0f);
        sn = t * c;
        lu = suu - t * suv;
        lv = svv + t * suv;
    }
    const float x = lu <= lv ? c : sn, y = lu <= lv ? -sn : c;
    const float3 nv = make_float3(x * u.x + y * v.x, x * u.y + y * v.y, x * u.z + y * v.z);
    const float in = 1.0f / sqrtf(dot3(nv, nv));
    return make_float3(nv.x * in, nv.y * in, nv.z * in);
}

// Covariance of one neighbourhood (Sec. III-C1, C_i of Eq. 19) from its
// points in rank order, get(j) for j = 0..k-1.  Two passes in binary32,
// both shifted by the first (nearest) neighbour p0 so the sums stay small:
// mean m of (p_j - p0), then the centred moments of (p_j - p0) - m, divided
// by k.  Built with --fmad=false, so every + and * below is rounded once;
// every caller runs this same code on the same values, so the fused kernel
// and pc_cov agree bit for bit.
// The six packed entries of one covariance row: three 8-byte stores when
// the row is 8-byte aligned (every row of an aligned [N,6] array is).
__device__ __forceinline__ void store6(float* out, float a, float b, float c, float d, float e, float f) {
    if ((reinterpret_cast<uintptr_t>(out) & 7) == 0) {
        float2* o2 = reinterpret_cast<float2*>(out);
        o2[0] = make_float2(a, b);
        o2[1] = make_float2(c, d);
        o2[2] = make_float2(e, f);
    } else {
        out[0] = a; out[1] = b; out[2] = c; out[3] = d; out[4] = e; out[5] = f;
    }
}

// The end of every plain covariance: centred sums / k, then, for eps >= 0,
// the plane regularisation C' = I - (1 - eps) n n^T; stored packed.
__device__ __forceinline__ void cov_finish(float cxx, float cxy, float cxz, float cyy, float cyz, float czz,
                                           float fk, float eps, float* out) {
    cxx = cxx / fk; cxy = cxy / fk; cxz = cxz / fk;
    cyy = cyy / fk; cyz = cyz / fk; czz = czz / fk;
    if (eps < 0.0f) {
        store6(out, cxx, cxy, cxz, cyy, cyz, czz);
        return;
    }
    const float3 n = min_eigvec(cxx, cxy, cxz, cyy, cyz, czz);
    const float f = 1.0f - eps;
    store6(out, 1.0f - f * n.x * n.x, -f * n.x * n.y, -f * n.x * n.z, 1.0f - f * n.y * n.y, -f * n.y * n.z,
           1.0f - f * n.z * n.z);
}

// C' = I - (1 - eps) n n^T in place of a packed covariance; eps < 0 keeps the
// covariance.
__device__ __forceinline__ void cov_regularise(float* c, float eps) {
    if (eps < 0.0f) return;
    const float3 n = min_eigvec(c[0], c[1], c[2], c[3], c[4], c[5]);
    const float f = 1.0f - eps;
    c[0] = 1.0f - f * n.x * n.x;
    c[1] = -f * n.x * n.y;
    c[2] = -f * n.x * n.z;
    c[3] = 1.0f - f * n.y * n.y;
    c[4] = -f * n.y * n.z;
    c[5] = 1.0f - f * n.z * n.z;
}

template <typename G>
__device__ __forceinline__ void cov_core(G&& get, int k, float eps, float* out) {
    const float4 p0 = get(0);
    float sx = 0.0f, sy = 0.0f, sz = 0.0f;
    for (int j = 0; j < k; ++j) {
        const float4 p = get(j);
        sx = sx + (p.x - p0.x);
        sy = sy + (p.y - p0.y);
        sz = sz + (p.z - p0.z);
    }
    const float fk = (float)k;
    const float mx = sx / fk, my = sy / fk, mz = sz / fk;
    float cxx = 0.0f, cxy = 0.0f, cxz = 0.0f, cyy = 0.0f, cyz = 0.0f, czz = 0.0f;
    for (int j = 0; j < k; ++j) {
        const float4 p = get(j);
        const float dx = (p.x - p0.x) - mx;
        const float dy = (p.y - p0.y) - my;
        const float dz = (p.z - p0.z) - mz;
        cxx = __fmaf_rn(dx, dx, cxx);
        cxy = __fmaf_rn(dx, dy, cxy);
        cxz = __fmaf_rn(dx, dz, cxz);
        cyy = __fmaf_rn(dy, dy, cyy);
        cyz = __fmaf_rn(dy, dz, cyz);
        czz = __fmaf_rn(dz, dz, czz);
    }
    cov_finish(cxx, cxy, cxz, cyy, cyz, czz, fk, eps, out);
}

__device__ __forceinline__ void nan_row(float* out) {
    const float nan = __int_as_float(0x7fc00000);
    for (int e = 0; e < 6; ++e) out[e] = nan;
}

// Covariance of the neighbourhood row nb[0], nb[st], ..., nb[(k-1) st]
// (caller indices, read from the caller-order copy).  `check`: validate
// every index (pc_cov); otherwise a leading -1 marks an unanswered row.
__device__ void cov_row(const Grid& g, const int32_t* nb, int st, int k, float eps, float* out,
                        bool check) {
    bool bad = nb[0] < 0;
    if (check) {
        bool oob = false;
        for (int j = 0; j < k; ++j) oob |= (nb[j * st] < 0) || ((int64_t)nb[j * st] >= g.m);
        if (oob) atomicOr(g.status, ST_BAD_INDEX);
        bad = oob;
    }
    if (bad) {
        nan_row(out);
        return;
    }
    cov_core([&](int j) { return __ldg(&g.xyz[nb[j * st]]); }, k, eps, out);
}

// Positions in the lane lists: a main-grid position, or an appended-points
// grid position with DTAG set (both grids hold fewer than 2^31 points).
constexpr uint32_t DTAG = 0x80000000u;

template <bool DEL>
__device__ __forceinline__ float4 pt_at(const Grid& g, const Grid& dg, uint32_t tp) {
    if (!DEL) return __ldg(&g.pts[tp]);
    const float4* base = (tp & DTAG) ? dg.pts : g.pts;
    return __ldg(&base[tp & ~DTAG]);
}

// Index of the point at tagged position tp in the union numbering: main
// points keep their index, appended point j is g.m + j.
template <bool DEL>
__device__ __forceinline__ uint32_t union_index(const Grid& g, uint32_t tp, float4 p) {
    const uint32_t i = __float_as_uint(p.w);
    return (DEL && (tp & DTAG)) ? (uint32_t)g.m + i : i;
}

// cov_row over the union numbering (a leading -1 marks an unanswered row).
template <bool DEL>
__device__ void cov_row_union(const Grid& g, const Grid& dg, const int32_t* nb, int k, float eps, float* out) {
    if (!DEL) {
        cov_row(g, nb, 1, k, eps, out, false);
        return;
    }
    if (nb[0] < 0) {
        nan_row(out);
        return;
    }
    cov_core([&](int j) {
        const int64_t i = nb[j];
        return i < g.m ? __ldg(&g.xyz[i]) : __ldg(&dg.xyz[i - g.m]);
    }, k, eps, out);
}

// Kernel-descriptor weighted covariance of one neighbourhood (Sec. III-C1:
// the covariance is computed "using the kernel descriptors" of Table I).
// For query x = q and its k neighbours y_j in rank order:
//   w_j = K(x, y_j),  W = sum w_j,
//   mu = sum w_j y_j / W,  C = sum w_j (y_j - mu)(y_j - mu)^T / W,
// then, for eps >= 0, C' = I - (1 - eps) n n^T with n the smallest-eigenvalue
// eigenvector (the same closed form as the plain covariance).  Binary32,
// two passes shifted by the nearest neighbour y_0 like the plain form.  A row
// whose W is not positive and finite is NaN.  The search kernels call it in
// place of cov_core when a descriptor is set, reading the neighbours from the
// cell-sorted copy they already hold in cache.
__device__ __forceinline__ float kd_weight(const CovKernel& ck, float qx, float qy, float qz, float4 p) {
    const float dx = qx - p.x, dy = qy - p.y, dz = qz - p.z;
    const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, dx * dx));
    switch (ck.type) {
        case 1:  // RBF
        case 2:  // Gaussian (s = 1 / (2 sigma^2))
            return expf(-r2 * ck.s);
        case 3: {  // Polynomial on coordinates relative to the bounding-box minimum
            const float ax = qx - ck.ox, ay = qy - ck.oy, az = qz - ck.oz;
            const float bx = p.x - ck.ox, by = p.y - ck.oy, bz = p.z - ck.oz;
            const float dot = __fmaf_rn(az, bz, __fmaf_rn(ay, by, ax * bx));
            return powf(__fmaf_rn(ck.alpha, dot, ck.c), ck.d);
        }
        case 4: {  // histogram intersection, same relative coordinates
            const float ax = qx - ck.ox, ay = qy - ck.oy, az = qz - ck.oz;
            const float bx = p.x - ck.ox, by = p.y - ck.oy, bz = p.z - ck.oz;
            return (fminf(ax, bx) + fminf(ay, by) + fminf(az, bz)) / (ax + ay + az);
        }
        case 5:  // Laplacian (s = 1 / sigma)
            return expf(-sqrtf(r2) * ck.s);
    }
    return 1.0f;
}

template <typename G>
__device__ void weighted_core(G&& get, const CovKernel& ck, float qx, float qy, float qz, int k, float eps,
                              float* out) {
    if (!isfinite(qx) || !isfinite(qy) || !isfinite(qz)) {
        nan_row(out);
        return;
    }
    const float4 p0 = get(0);
    float W = 0.0f, sx = 0.0f, sy = 0.0f, sz = 0.0f;
    for (int j = 0; j < k; ++j) {
        const float4 p = get(j);
        const float w = kd_weight(ck, qx, qy, qz, p);
        W = W + w;
        sx = __fmaf_rn(w, p.x - p0.x, sx);
        sy = __fmaf_rn(w, p.y - p0.y, sy);
        sz = __fmaf_rn(w, p.z - p0.z, sz);
    }
    if (!(W > 0.0f) || !isfinite(W)) {
        nan_row(out);
        return;
    }
    const float mx = sx / W, my = sy / W, mz = sz / W;
    float cxx = 0.0f, cxy = 0.0f, cxz = 0.0f, cyy = 0.0f, cyz = 0.0f, czz = 0.0f;
    for (int j = 0; j < k; ++j) {
        const float4 p = get(j);
        const float w = kd_weight(ck, qx, qy, qz, p);
        const float dx = (p.x - p0.x) - mx, dy = (p.y - p0.y) - my, dz = (p.z - p0.z) - mz;
        const float wx = w * dx, wy = w * dy;
        cxx = __fmaf_rn(wx, dx, cxx);
        cxy = __fmaf_rn(wx, dy, cxy);
        cxz = __fmaf_rn(wx, dz, cxz);
        cyy = __fmaf_rn(wy, dy, cyy);
        cyz = __fmaf_rn(wy, dz, cyz);
        czz = __fmaf_rn(w * dz, dz, czz);
    }
    cxx = cxx / W; cxy = cxy / W; cxz = cxz / W;
    cyy = cyy / W; cyz = cyz / W; czz = czz / W;
    if (eps < 0.0f) {
        out[0] = cxx; out[1] = cxy; out[2] = cxz; out[3] = cyy; out[4] = cyz; out[5] = czz;
        return;
    }
    const float3 n = min_eigvec(cxx, cxy, cxz, cyy, cyz, czz);
    const float f = 1.0f - eps;
    out[0] = 1.0f - f * n.x * n.x;
    out[1] = -f * n.x * n.y;
    out[2] = -f * n.x * n.z;
    out[3] = 1.0f - f * n.y * n.y;
    out[4] = -f * n.y * n.z;
    out[5] = 1.0f - f * n.z * n.z;
}

// ---------------------------------------------------------------- tiles

// The covariance of a written row (caller or union indices; a leading -1
// marks an unanswered row), plain or weighted by the descriptor in a.
template <bool DEL>
__device__ void cov_row_any(const Grid& g, const Grid& dg, const int32_t* nb, int k, const TileArgs& a, float qx,
                            float qy, float qz, float* out) {
    if (a.ck.type == 0) {
        cov_row_union<DEL>(g, dg, nb, k, a.eps, out);
        return;
    }
    if (nb[0] < 0) {
        nan_row(out);
        return;
    }
    weighted_core([&](int j) {
        const int64_t i = nb[j];
        return (!DEL || i < g.m) ? __ldg(&g.xyz[i]) : __ldg(&dg.xyz[i - g.m]);
    }, a.ck, qx, qy, qz, k, a.eps, out);
}

// ---------------------------------------------------------------- group search
// k <= 32: a group of G lanes (4, or 8 for small calls) answers a query, and a
// block is one warp: a unit of 32 / G queries.
//
// 1. Walk: the rows of the box around the starting radius are resolved one
//    per lane and handed round the group, whose lanes take the points of G
//    rows in turn as one run.  Every point with d2 <= t = min(r^2, tau), tau
//    certified for the box, goes to the lane's list in shared memory (d2 and
//    position).  With at least k points and no list overflowing, the k
//    smallest of them are the k nearest overall: all points with d2 <= t lie
//    in the box.  Otherwise the radius is scaled by what the count says about
//    the density and the query walks again (131k scan: 1.04 walks a warp).
// 2. Selection, when the lists hold more than CAP points: thresholds placed
//    by linear interpolation in d2 (a surface's count grows evenly in d2)
//    are counted over the lists, four at a time, until one holds between k
//    and CAP points.
// 3. Sort: 32-bit keys (d2 bits << 1, low TB bits replaced by the list slot)
//    sorted across the group: Batcher's network on each lane's CAP / G
//    registers, then bitonic merges between lanes.  The keys order d2 to
//    within 2^(TB-1) ulps; a group that finds two neighbours in one such
//    bucket is put in exact (d2, index) order by an insertion sort.
// 4. Rows are written by the warp as one contiguous block; three lanes of
//    the group carry the covariance sums.  (Into host memory off 128-byte
//    lines, by a block of four warps: k_knn_host.)
//
// k_knn_rest follows every launch.  It turns the covariances into normals and
// C' (eps >= 0), one query per lane, and answers the queries that no attempt
// settled (fewer than k points within reach, or more than CAP equal
// distances): their row's first d2 word is UNANSWERED, and the sign bit of
// the unit's first d2 word marks the unit.  Squared distances are never
// negative and never NaN, so neither mark can be mistaken for a result, and
// no workspace or counter is shared between calls in flight.
//
// What bounds it: issue slots (68-72 % of them used) in the row walk, two
// thirds of the time.  One lane per query on blocks of four warps (the layout
// before) kept 32 different point streams in a warp, walked twice, held 95
// registers and ran 1.35 waves of long warps.
constexpr int MAX_ATTEMPTS = 6;
constexpr float START = 1.4f;  // first radius over the calibrated starting radius; 1.26 and 1.54: 8 and 12 % slower
constexpr int64_t SMALL_MAP = 2048;  // points a group may well walk several times
constexpr int BATCH = 2;       // point loads a lane has in flight; 1 and 3: 3 % slower on scans
constexpr uint32_t UNANSWERED = 0xffffffffu, UNIT_FLAG = 0x80000000u;
constexpr uint32_t NAN_ROW = 0x7fc00000u;  // every entry of a covariance row without a value

// Search modes: 0 = group search with room for 32 sorted survivors (k <= 24),
// 1 = with room for 64 (k <= 32), 2 = warp path only (k > 32).
__host__ __device__ __forceinline__ int search_mode(int k) { return k <= 24 ? 0 : (k <= 32 ? 1 : 2); }
// List slots of a lane: 64 (k <= 24) or 96 points per query over G lanes.
__host__ __device__ constexpr int lane_slots(int cap, int g) { return (cap == 32 ? 64 : 96) / g; }
// Shared memory of one warp: the lists (d2, position), then CAP sort keys per
// query.
__host__ __device__ constexpr size_t group_warp_smem(int cap, int g) {
    return (size_t)lane_slots(cap, g) * 32 * 8 + (size_t)(32 / g) * cap * sizeof(uint32_t);
}

__device__ __forceinline__ void cas32(uint32_t& a, uint32_t& b) {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}

// Batcher's odd-even merge sort over NN registers, ascending: merges sorted
// runs of length p into runs of 2p; within a merge, elements k apart are
// compared, k halving from p, and only pairs inside the same run of 2p.  The
// comparator list is computed at compile time and expanded as a parameter
// pack, so every register index is a constant.
template <int NN>
struct OemNet {
    struct Table {
        int a[NN * NN], b[NN * NN];
        int n;
    };
    __host__ __device__ static constexpr Table make() {
        Table t{};
        t.n = 0;
        for (int p = 1; p < NN; p <<= 1)
            for (int k = p; k >= 1; k >>= 1)
                for (int j = k % p; j + k < NN; j += 2 * k)
                    for (int i = 0; i < k && i + j + k < NN; ++i)
                        if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) {
                            t.a[t.n] = i + j;
                            t.b[t.n] = i + j + k;
                            ++t.n;
                        }
        return t;
    }
};

template <int NN, int... Cs>
__device__ __forceinline__ void oem_apply(uint32_t (&K)[NN], std::integer_sequence<int, Cs...>) {
    (cas32(K[std::integral_constant<int, OemNet<NN>::make().a[Cs]>::value],
           K[std::integral_constant<int, OemNet<NN>::make().b[Cs]>::value]),
     ...);
}

template <int NN>
__device__ __forceinline__ void sort_regs(uint32_t (&K)[NN]) {
    oem_apply<NN>(K, std::make_integer_sequence<int, OemNet<NN>::make().n>{});
}

// Ascending order of a bitonic sequence in NN registers.
template <int NN>
__device__ __forceinline__ void merge_regs(uint32_t (&K)[NN]) {
#pragma unroll
    for (int s = NN / 2; s >= 1; s >>= 1)
#pragma unroll
        for (int i = 0; i < NN; ++i)
            if ((i & s) == 0) cas32(K[i], K[i + s]);
}

// Sorts the group's G * NN keys: lane sub of the group ends with the keys
// of ranks sub * NN .. sub * NN + NN - 1.  Runs of w lanes are merged into
// runs of 2w by comparing each key with its mirror in the other run, which
// leaves two bitonic halves, then by exchanges between lanes w / 2 .. 1 apart
// and a merge inside each lane.
template <int NN, int G>
__device__ __forceinline__ void sort_group(uint32_t (&K)[NN], int sub) {
    sort_regs<NN>(K);
#pragma unroll
    for (int w = 1; w < G; w <<= 1) {
        const bool lower = (sub & w) == 0;
        uint32_t y[NN];
#pragma unroll
        for (int i = 0; i < NN; ++i) y[i] = __shfl_xor_sync(FULL, K[NN - 1 - i], 2 * w - 1);
#pragma unroll
        for (int i = 0; i < NN; ++i) K[i] = lower ? min(K[i], y[i]) : max(K[i], y[i]);
#pragma unroll
        for (int s = w >> 1; s >= 1; s >>= 1) {
            const bool low = (sub & s) == 0;
#pragma unroll
            for (int i = 0; i < NN; ++i) {
                const uint32_t z = __shfl_xor_sync(FULL, K[i], s);
                K[i] = low ? min(K[i], z) : max(K[i], z);
            }
        }
        merge_regs<NN>(K);
    }
}

// Sum of v over the lanes of a group.
template <int G>
__device__ __forceinline__ uint32_t group_sum(uint32_t v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// Visits every point of the box [l, h] (clamped to the grid) whose row -- or,
// without the row index, whose cell -- can hold a point within sqrt(t) of q,
// as f(position, point), the points of a row spread over the group's lanes.
// Control flow is uniform over the warp but for the innermost loops; groups
// with act = false take part with empty boxes.
template <int G, bool WIN, typename F>
__device__ __forceinline__ void group_walk(const Grid& g, bool act, float qx, float qy, float qz, int lx, int hx,
                                           int ly, int hy, int lz, int hz, float eta, float t, int sub,
                                           uint32_t& visits, F&& f) {
    const bool rows = g.dstart != nullptr;
    const int nx = rows ? 1 : hx - lx + 1, ny = hy - ly + 1, nz = hz - lz + 1;
    const int units = act && lx <= hx && ny > 0 && nz > 0 ? nx * ny * nz : 0;
    const int last = __reduce_max_sync(FULL, (unsigned)units);
    const float tx = t * (1.0f + 0x1p-18f);
    const bool wx = WIN && g.windowed && (lx == g.tlx || hx == g.thx);
    int cx = lx, cy = ly, cz = lz;
    auto advance = [&](int n) {
        if (!rows) {
            cx += n;
            n = 0;
            while (cx > hx) {
                cx -= nx;
                ++n;
            }
        }
        cy += n;
        while (cy > hy) {
            cy -= ny;
            ++cz;
        }
    };
    if (sub < units) advance(sub);
    for (int base = 0; base < last; base += G) {
        uint2 r = make_uint2(0u, 0u);
        if (base + sub < units) {
            if (rows) {
                r = row_part(g, qx, qy, qz, cy, cz, lx, hx, eta, t, tx);
            } else {
                const float lb2 = box_gap2(g, qx, qy, qz, cx, cy, cz, eta);
                if (!(lb2 * (1.0f - 0x1p-20f) > t)) r = lookup_cell(g, pack_key(cx, cy, cz, g.bx, g.by));
            }
            visits += r.y;
            // a row (cell) on a boundary cell of the window tests its points
            if (WIN && g.windowed &&
                ((rows ? wx : cx == g.tlx || cx == g.thx) || cy == g.tly || cy == g.thy || cz == g.tlz ||
                 cz == g.thz))
                r.y |= 0x80000000u;
            advance(G);
        }
        // The G rows as one run of c points: point i of it is pts[i + off],
        // off set by the last row that starts at or before i.
        uint32_t start[G], upto[G];  // of row j: start less the points before it; points before row j + 1
        uint32_t c = 0, test = 0;
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const uint32_t cj = __shfl_sync(FULL, r.y, j, G);
            start[j] = __shfl_sync(FULL, r.x, j, G) - c;
            if (WIN) test |= (cj >> 31) << j;
            c += WIN ? cj & 0x7fffffffu : cj;
            upto[j] = c;
        }
        for (uint32_t i0 = sub; i0 < c; i0 += G * BATCH) {
            float4 p[BATCH];
            uint32_t pos[BATCH];
#pragma unroll
            for (int b = 0; b < BATCH; ++b) {
                const uint32_t i = i0 + G * b;
                uint32_t off = start[0];
                bool cut = WIN && (test & 1u);
#pragma unroll
                for (int j = 1; j < G; ++j)
                    if (i >= upto[j - 1]) {
                        off = start[j];
                        if (WIN) cut = test >> j & 1u;
                    }
                pos[b] = i + off;
                if (i < c) p[b] = window_cut<WIN>(g, cut, __ldg(&g.pts[pos[b]]));
            }
#pragma unroll
            for (int b = 0; b < BATCH; ++b)
                if (i0 + G * b < c) f(pos[b], p[b]);
        }
    }
}

// The starting radius of a query where the map's density is uneven: the
// points of the 27 cells around q (counted through the row index, no point
// is read) set a surface density n / (9 h^2), and the radius of a disc
// holding k points at that density is c h sqrt(k / n); at most 3 h (and 3 h
// when the block is empty).  Only the search's speed depends on it.
template <int G, bool WIN>
__device__ __forceinline__ float probe_radius(const Grid& g, bool act, float qx, float qy, float qz, int k, float c,
                                              int sub) {
    uint32_t n = 0;
    if (act && g.dstart) {
        const int cx = cell_of(qx, g.ox, g.inv_h), cy = cell_of(qy, g.oy, g.inv_h), cz = cell_of(qz, g.oz, g.inv_h);
        const int x0 = max(cx - 1, WIN ? g.wlx : 0), x1 = min(cx + 1, WIN ? g.whx : g.dimx - 1);
        const int y0 = max(cy - 1, WIN ? g.wly : 0), y1 = min(cy + 1, WIN ? g.why : g.dimy - 1);
        const int z0 = max(cz - 1, WIN ? g.wlz : 0), z1 = min(cz + 1, WIN ? g.whz : g.dimz - 1);
        const int ny = y1 - y0 + 1, nz = z1 - z0 + 1;
        if (x0 <= x1 && ny > 0 && nz > 0)
            for (int u = sub; u < ny * nz; u += G) n += row_range(g, y0 + u % ny, z0 + u / ny, x0, x1).y;
    }
    n = group_sum<G>(n);
    const float cap = 3.0f * g.h;
    return n > 0 ? fminf(c * g.h * sqrtf((float)k / (float)n), cap) : cap;
}

// The cell box of half-width r around q on one grid, clamped to the grid (or
// its window range), with its certified tau and eta; big: too many rows or
// cells for a group; none: it misses the grid (k_knn_rest takes both).
struct GroupBox {
    int lx, hx, ly, hy, lz, hz;
    float tau, eta;
    bool big, none;
};
template <bool WIN>
__device__ __forceinline__ GroupBox group_box(const Grid& g, float qx, float qy, float qz, float r) {
    const int lx = cell_of(__fsub_rn(qx, r), g.ox, g.inv_h), hx = cell_of(__fadd_rn(qx, r), g.ox, g.inv_h);
    const int ly = cell_of(__fsub_rn(qy, r), g.oy, g.inv_h), hy = cell_of(__fadd_rn(qy, r), g.oy, g.inv_h);
    const int lz = cell_of(__fsub_rn(qz, r), g.oz, g.inv_h), hz = cell_of(__fadd_rn(qz, r), g.oz, g.inv_h);
    GroupBox b;
    b.tau = certified_tau(g, qx, qy, qz, lx, hx, ly, hy, lz, hz);
    const int cm = max(max(max(abs(lx), abs(hx + 1)), max(abs(ly), abs(hy + 1))), max(abs(lz), abs(hz + 1)));
    const float qm = fmaxf(fabsf(qx), fmaxf(fabsf(qy), fabsf(qz)));
    b.eta = 0x1p-20f * (g.coord_scale + qm + (float)cm * g.h);
    b.lx = max(lx, WIN ? g.wlx : 0);
    b.hx = min(hx, WIN ? g.whx : g.dimx - 1);
    b.ly = max(ly, WIN ? g.wly : 0);
    b.hy = min(hy, WIN ? g.why : g.dimy - 1);
    b.lz = max(lz, WIN ? g.wlz : 0);
    b.hz = min(hz, WIN ? g.whz : g.dimz - 1);
    const int64_t nrows = (int64_t)max(b.hy - b.ly + 1, 0) * max(b.hz - b.lz + 1, 0);
    const int64_t ncl = nrows * max(b.hx - b.lx + 1, 0);
    b.big = !group_allowed(g, ncl, nrows);
    b.none = ncl == 0;
    return b;
}

// The covariance of a query from its k neighbours' coordinates in rank order
// (c[r CS], c[(KMAX + r) CS], c[(2 KMAX + r) CS] for x, y, z of rank r; the
// next KMAX CS entries are free for weights).  Lane sub < 3 of the group
// carries one coordinate u: its mean, its square sum and its product sum with
// the next coordinate v, divided into uu and uv.  Every sum runs over the
// ranks in order with the operations of cov_core / weighted_core, so the
// results are theirs bit for bit: the split is over the sums, not over the
// neighbours.  Returns the divisor (k, or the total weight).
template <int CS, int KMAX, int G, bool weighted>
__device__ __forceinline__ float group_moments(float* c, const TileArgs& a, float qx, float qy, float qz, int sub,
                                               float& uu, float& uv) {
    const int k = a.k, cu = sub < 3 ? sub : 0, cv = cu == 2 ? 0 : cu + 1;
    const float* u = c + cu * KMAX * CS;
    const float* v = c + cv * KMAX * CS;
    float* const wt = c + 3 * KMAX * CS;
    const float u0 = u[0], v0 = v[0];
    float total = (float)k, s = 0.0f;
    uu = uv = 0.0f;
    if constexpr (weighted) {
        for (int j = sub; j < k; j += G)
            wt[j * CS] = kd_weight(a.ck, qx, qy, qz,
                                   make_float4(c[j * CS], c[(KMAX + j) * CS], c[(2 * KMAX + j) * CS], 0.0f));
        __syncwarp();
        total = 0.0f;
        for (int j = 0; j < k; ++j) {
            const float w = wt[j * CS];
            total = total + w;
            s = __fmaf_rn(w, u[j * CS] - u0, s);
        }
    } else {
#pragma unroll 4
        for (int j = 0; j < k; ++j) s = s + (u[j * CS] - u0);
    }
    const float mu = s / total, mv = __shfl_sync(FULL, mu, cv, G);
    if constexpr (weighted) {
        for (int j = 0; j < k; ++j) {
            const float w = wt[j * CS];
            const float du = (u[j * CS] - u0) - mu, dv = (v[j * CS] - v0) - mv;
            // products weighted on the earlier coordinate, as in weighted_core
            uu = __fmaf_rn(w * du, du, uu);
            uv = cu == 2 ? __fmaf_rn(w * dv, du, uv) : __fmaf_rn(w * du, dv, uv);
        }
    } else {
#pragma unroll 4
        for (int j = 0; j < k; ++j) {
            const float du = (u[j * CS] - u0) - mu, dv = (v[j * CS] - v0) - mv;
            uu = __fmaf_rn(du, du, uu);
            uv = __fmaf_rn(du, dv, uv);
        }
    }
    uu = uu / total;
    uv = uv / total;
    return total;
}

// One unit of cnt <= 32 / G queries on one warp.  With DEL the search covers
// the union of the main grid g and the grid dg of appended points (point j of
// dg is g.m + j): both grids' boxes are walked, filtered by the smaller of
// their certified taus, and list entries from dg carry DTAG.  idx, d2 and cov
// point at the unit's own rows in device memory (HOST = 0), in mapped host memory
// (1: covariances are finished here) or in shared memory on their way there (2:
// so are they, and the caller sets the mark).  Returns whether the unit has
// queries left for k_knn_rest.
template <int CAP, int G, int COV, bool WIN, bool DEL, int HOST>
__device__ __forceinline__ bool group_unit(const Grid& g, const Grid& dg, const float* __restrict__ q, int cnt,
                                           const TileArgs& a, float rho0, int32_t* __restrict__ idx,
                                           float* __restrict__ d2, float* __restrict__ cov, unsigned char* smem) {
    constexpr int SLOTS = lane_slots(CAP, G), WQ = 32 / G, NN = CAP / G;
    constexpr int TB = SLOTS * G <= 64 ? 6 : 7;
    constexpr uint32_t TAG = (1u << TB) - 1u;
    constexpr int KMAX = CAP == 32 ? 24 : 32, ROUNDS = (WQ * KMAX + 31) / 32, CS = WQ + 1;
    static_assert(4 * KMAX * CS <= SLOTS * 64 && 6 * WQ <= WQ * CAP, "coordinates and weights overlay the lists");
    static_assert(SLOTS * G <= (1 << TB), "list slots must fit the key tag");
    // k_knn_rest may be set up while the last blocks run (it waits for them)
    cudaTriggerProgrammaticLaunchCompletion();
    const int k = a.k;
    const int lane = HOST == 2 ? threadIdx.x & 31 : threadIdx.x, sub = lane & (G - 1);
    float* const ld = reinterpret_cast<float*>(smem);
    uint32_t* const lp = reinterpret_cast<uint32_t*>(smem + SLOTS * 32 * 4);
    uint32_t* const kb = reinterpret_cast<uint32_t*>(smem + SLOTS * 32 * 8);
    const int qi = lane / G;  // query of the unit
    uint32_t* const kq = kb + qi * CAP;
    const bool active = qi < cnt;
    float qx = 0.0f, qy = 0.0f, qz = 0.0f;
    if (active) {
        const float* p = q + 3 * qi;
        qx = __ldg(p);
        qy = __ldg(p + 1);
        qz = __ldg(p + 2);
    }
    const bool finite = active && isfinite(qx) && isfinite(qy) && isfinite(qz);
    uint32_t visits = 0;  // points of the rows this lane resolved

    // ---- walk
    float r2;
    {
        float r = rho0;
        if (a.probe_c > 0.0f) r = probe_radius<G, WIN>(g, finite, qx, qy, qz, k, a.probe_c, sub);
        r *= START;
        r2 = fminf(r * r, 1e30f);
    }
    float lo2 = 0.0f, hi2 = -1.0f;  // squared radii known to hold too few / too many (hi2 > 0)
    bool todo = finite, ok = false;
    int w = 0, m = 0;
    float t = -1.0f;
    for (int attempt = 0; attempt < MAX_ATTEMPTS; ++attempt) {
        if (!__any_sync(FULL, todo)) break;
        GroupBox b, e;
        float tt = -1.0f;
        b.lx = b.ly = b.lz = e.lx = e.ly = e.lz = 0;
        b.hx = b.hy = b.hz = e.hx = e.hy = e.hz = -1;
        b.eta = e.eta = 0.0f;
        if (todo) {
            const float r = sqrtf(r2);
            b = group_box<WIN>(g, qx, qy, qz, r);
            float tau = b.tau;
            bool big = b.big, none = b.none;
            if (DEL) {
                e = group_box<WIN>(dg, qx, qy, qz, r);
                tau = fminf(tau, e.tau);
                big = big || e.big;
                none = none && e.none;
            }
            tt = fminf(r2, tau);
            // A query off the grid or its window by more than its radius: widened by
            // a factor, the ball would hold thousands of points, walked by four
            // lanes several times.  60k queries, three quarters of them outside a
            // window of a quarter of the map, us here / with k_knn_rest: maps of
            // 1k points 133 / 231, 2k 296 / 338, 4k 570 / 501, 8k 762 / 523, 32k
            // 2017 / 476, 200k 13388 / 2241.
            if (big || (none && g.exhaustive && g.m > SMALL_MAP)) todo = false;
            else w = 0;
        }
        const bool act = todo && tt >= 0.0f;
        auto keep = [&](uint32_t pos, const float4 p) {
            const float d = sqdist_pinned(qx, qy, qz, p.x, p.y, p.z);
            if (d <= tt) {
                if (w < SLOTS) {
                    ld[w * 32 + lane] = d;
                    lp[w * 32 + lane] = pos;
                }
                ++w;
            }
        };
        group_walk<G, WIN>(g, act, qx, qy, qz, b.lx, b.hx, b.ly, b.hy, b.lz, b.hz, b.eta, tt, sub, visits, keep);
        if (DEL)
            group_walk<G, WIN>(dg, act, qx, qy, qz, e.lx, e.hx, e.ly, e.hy, e.lz, e.hz, e.eta, tt, sub, visits,
                            [&](uint32_t pos, const float4 p) { keep(pos | DTAG, p); });
        const uint32_t mm = group_sum<G>((uint32_t)w);
        const bool over = (__ballot_sync(FULL, w > SLOTS) >> (lane & ~(G - 1)) & ((1u << G) - 1u)) != 0u;
        if (todo) {
            if (mm < (uint32_t)k) {  // widen; a wider box also certifies further
                lo2 = r2;
                const float f = fminf(fmaxf(1.7f * (float)k / (float)max(mm, 1u), 1.5f), 9.0f);
                r2 = hi2 > 0.0f ? 0.5f * (lo2 + hi2) : fminf(fmaxf(r2, 1e-6f * g.h * g.h) * f, 1e30f);
            } else if (over) {  // narrow
                hi2 = tt;
                r2 = lo2 > 0.0f ? 0.5f * (lo2 + hi2)
                                : tt * fminf(fmaxf(1.6f * (float)k / (float)mm, 0.02f), 0.8f);
            } else {
                ok = true;
                todo = false;
                m = (int)mm;
                t = tt;
            }
        }
    }
    if (!ok) w = 0;

    // ---- selection
    int u = w;  // entries of this lane that are kept
    if (__any_sync(FULL, ok && m > CAP)) {
        bool need = ok && m > CAP;
        float lo = 0.0f, hi = t, sel = t;
        int kept = m;
        for (int round = 0; round < 10; ++round) {
            if (!__any_sync(FULL, need)) break;
            float th[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
                th[j] = round == 0 ? t * (((float)k + (float)(CAP - k) * (0.25f * (float)j + 0.125f)) / (float)m)
                                   : lo + (hi - lo) * (0.2f * (float)(j + 1));
            uint32_t c = 0;
            if (need)
                for (int i = 0; i < w; ++i) {
                    const float d = ld[i * 32 + lane];
                    c += (d <= th[0] ? 1u : 0u) + (d <= th[1] ? 1u << 8 : 0u) + (d <= th[2] ? 1u << 16 : 0u) +
                         (d <= th[3] ? 1u << 24 : 0u);
                }
            c = group_sum<G>(c);  // at most SLOTS * G < 256 each
            if (need) {
                bool found = false;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int cj = (int)(c >> (8 * j) & 255u);
                    if (!found && cj >= k) {
                        found = true;
                        sel = th[j];
                        kept = cj;
                    }
                    if (!found) lo = fmaxf(lo, th[j]);
                }
                if (found) hi = fminf(hi, sel);
                need = !found || kept > CAP;
            }
        }
        if (need) ok = false;  // more than CAP points at one distance
        else if (ok) {
            m = kept;
            u = 0;
            for (int i = 0; i < w; ++i) u += ld[i * 32 + lane] <= sel ? 1 : 0;
            t = sel;
        }
        if (!ok) w = u = m = 0;
    }

    // ---- keys, in a compact row per query
    {
        int at = u;
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const int y = __shfl_up_sync(FULL, at, o, G);
            if (sub >= o) at += y;
        }
        at -= u;
        for (int i = 0; i < w; ++i) {
            const float d = ld[i * 32 + lane];
            if (d <= t) kq[at++] = ((__float_as_uint(d) << 1) & ~TAG) | (uint32_t)(i * G + sub);
        }
        for (int i = m + sub; i < CAP; i += G) kq[i] = 0xffffffffu;
    }
    __syncwarp();
    uint32_t K[NN];
    uint4* const kv = reinterpret_cast<uint4*>(kq + sub * NN);
#pragma unroll
    for (int i = 0; i < NN / 4; ++i) {
        const uint4 v = kv[i];
        K[4 * i] = v.x;
        K[4 * i + 1] = v.y;
        K[4 * i + 2] = v.z;
        K[4 * i + 3] = v.w;
    }
    sort_group<NN, G>(K, sub);
#pragma unroll
    for (int i = 0; i < NN / 4; ++i) kv[i] = make_uint4(K[4 * i], K[4 * i + 1], K[4 * i + 2], K[4 * i + 3]);
    bool amb = false;
#pragma unroll
    for (int i = 0; i + 1 < NN; ++i) amb |= (sub * NN + i + 1 < m) && ((K[i] ^ K[i + 1]) <= TAG);
    {
        const uint32_t nx = __shfl_down_sync(FULL, K[0], 1, G);
        amb |= sub + 1 < G && (sub + 1) * NN < m && ((K[NN - 1] ^ nx) <= TAG);
    }
    __syncwarp();
    const unsigned ambs = __ballot_sync(FULL, amb);
    if (ambs) {
        if (sub == 0 && (ambs >> lane & ((1u << G) - 1u)) != 0u) {
            auto before = [&](uint32_t ka, uint32_t kc) {  // exact (d2, index) order of two entries
                const int ia = (int)(ka & TAG), ic = (int)(kc & TAG);
                const int sa = (ia / G) * 32 + lane + ia % G, sc = (ic / G) * 32 + lane + ic % G;
                const float da = ld[sa], dc = ld[sc];
                if (da != dc) return da < dc;
                const uint32_t pa = lp[sa], pc = lp[sc];
                return union_index<DEL>(g, pa, pt_at<DEL>(g, dg, pa)) < union_index<DEL>(g, pc, pt_at<DEL>(g, dg, pc));
            };
            for (int i = 1; i < m; ++i) {
                const uint32_t x = kq[i];
                int j = i;
                while (j > 0 && ((kq[j - 1] ^ x) <= TAG) && before(x, kq[j - 1])) {
                    kq[j] = kq[j - 1];
                    --j;
                }
                kq[j] = x;
            }
        }
        __syncwarp();
    }

    // ---- rows, one block per unit; the neighbours' coordinates go over the
    // lists (at rank * (WQ + 1) + query: no bank conflicts, whether written
    // rank by rank or read query by query)
    const unsigned okm = __ballot_sync(FULL, ok), finm = __ballot_sync(FULL, finite);
    const unsigned badm = finm & ~okm;
    const bool with_cov = COV && cov != nullptr;
    {
        uint32_t* const d2b = reinterpret_cast<uint32_t*>(d2);
        const uint32_t inv = (65536u + (uint32_t)k - 1u) / (uint32_t)k;  // e / k for e < 8 * 32
        float nx[ROUNDS], ny[ROUNDS], nz[ROUNDS];
        int to[ROUNDS];
#pragma unroll
        for (int it = 0; it < ROUNDS; ++it) {
            const int e = lane + 32 * it;
            to[it] = -1;
            if (e < cnt * k) {
                const int qe = (int)((uint32_t)e * inv >> 16), r = e - qe * k;
                int iv = -1;
                uint32_t dv = 0x7f800000u;  // +inf
                if (okm >> (qe * G) & 1u) {
                    const uint32_t tag = kb[qe * CAP + r] & TAG;
                    const int at = (int)(tag / G) * 32 + qe * G + (int)(tag % G);
                    dv = __float_as_uint(ld[at]);
                    const uint32_t tp = lp[at];
                    const float4 p = pt_at<DEL>(g, dg, tp);
                    iv = (int)union_index<DEL>(g, tp, p);
                    nx[it] = p.x;
                    ny[it] = p.y;
                    nz[it] = p.z;
                    to[it] = r * CS + qe;
                } else if (finm >> (qe * G) & 1u) {
                    dv = UNANSWERED;
                }
                if (HOST < 2 && e == 0 && badm) dv |= UNIT_FLAG;
                idx[e] = iv;
                d2b[e] = dv;
            }
        }
        if (with_cov) {
            __syncwarp();  // the lists are done with
#pragma unroll
            for (int it = 0; it < ROUNDS; ++it)
                if (to[it] >= 0) {
                    ld[to[it]] = nx[it];
                    ld[KMAX * CS + to[it]] = ny[it];
                    ld[2 * KMAX * CS + to[it]] = nz[it];
                }
            __syncwarp();
        }
    }
    visits = __reduce_add_sync(FULL, visits);
    if (lane == 0) {
        atomicAdd(&g.stats[3], (unsigned long long)visits);
        if (badm) atomicAdd(&g.stats[1], (unsigned long long)(__popc(badm) / G));
        if (__popc(finm) < cnt * G) atomicOr(g.status, ST_NONFINITE);
    }
    // ---- covariances
    if (with_cov) {
        float uu, uv;
        const float total = group_moments<CS, KMAX, G, COV == 2>(ld + qi, a, qx, qy, qz, sub, uu, uv);
        float* const sc = HOST == 2 ? cov : reinterpret_cast<float*>(kb);  // the keys are done with
        const bool some = ok && total > 0.0f && isfinite(total);
        const float nan = __uint_as_float(NAN_ROW);
        if (sub < 3) {  // xx, xy; yy, yz; zz, xz
            sc[6 * qi + (sub == 0 ? 0 : sub + 2 + (sub >> 1))] = some ? uu : nan;
            sc[6 * qi + (sub == 0 ? 1 : sub == 1 ? 4 : 2)] = some ? uv : nan;
        }
        __syncwarp();
        if constexpr (HOST > 0) {  // a kernel of its own: as a branch it cost calls into device memory 2 us in spills
            if (sub == 0 && some) cov_regularise(sc + 6 * qi, a.eps);
            __syncwarp();
        }
        if constexpr (HOST < 2)
            for (int i = lane; i < 6 * cnt; i += 32) cov[i] = sc[i];
    }
    return badm != 0u;
}

// k > 32: the warp-cooperative search for each query of the tile in turn.
template <bool COV, bool DEL>
__device__ void warp_tile(const Grid& g, const Grid& dg, const float* __restrict__ q, int64_t n0, int cnt,
                          const TileArgs& a, float rho0, int32_t* __restrict__ idx,
                          float* __restrict__ d2, float* __restrict__ cov, u64* pend,
                          int lane) {
    const int k = a.k;
    float rho = rho0;
    if (lane == 0) {
        atomicAdd(&g.stats[0], (unsigned long long)cnt);
        atomicAdd(&g.stats[1], (unsigned long long)cnt);
    }
    for (int i = 0; i < cnt; ++i) {
        const int64_t n = n0 + i;
        const float qx = __ldg(q + 3 * n), qy = __ldg(q + 3 * n + 1), qz = __ldg(q + 3 * n + 2);
        const bool finite = isfinite(qx) && isfinite(qy) && isfinite(qz);
        SearchState<2> S;
        state_reset(S);
        int sr = SEARCH_LIMIT;
        if (finite) sr = knn_search<2, DEL>(g, dg, qx, qy, qz, k, rho, S, pend, lane);
        const bool ok = finite && sr == SEARCH_OK;
        if (!ok && lane == 0)
            atomicOr(g.status, !finite ? ST_NONFINITE : sr == SEARCH_SHORT ? ST_SHORT : ST_SEARCH_LIMIT);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int r = s * 32 + lane;
            if (r < k) {
                const u64 key = S.L[s];
                const int32_t oi = ok ? (int32_t)(uint32_t)key : -1;
                idx[n * k + r] = oi;
                d2[n * k + r] = ok ? __uint_as_float((uint32_t)(key >> 32)) : INFINITY;
            }
        }
        if (ok) {
            const float dk = __uint_as_float((uint32_t)(S.kth >> 32));
            rho = fminf(fmaxf(sqrtf(dk) * 1.15f, 1e-2f * g.h), 1e30f);
        }
    }
    if (COV && cov != nullptr) {
        __syncwarp();
        if (lane < cnt) {
            const int64_t nl = n0 + lane;
            cov_row_any<DEL>(g, dg, idx + nl * k, k, a, __ldg(q + 3 * nl), __ldg(q + 3 * nl + 1),
                             __ldg(q + 3 * nl + 2), cov + 6 * nl);
        }
        __syncwarp();
    }
}

// Work items are issued last-first.  A spinning LiDAR scan stored ring by ring
// with rising elevation ends with its farthest, sparsest points, whose units
// cost the most; starting them first lets the cheap near-range units fill the
// end of the launch.  (The order never changes a result.)  An item is one
// block of the group search (CAP > 0) and one warp of the warp path (CAP = 0).
template <int CAP>
__device__ __forceinline__ int64_t work_item(int64_t items, int last_first) {
    const int64_t w = CAP ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    return w >= items ? -1 : (last_first ? items - 1 - w : w);
}

// The scan that owns work item `item` of a batch's tile table.
__device__ __forceinline__ int scan_of_item(const ScanDesc* __restrict__ scans, int nscans, int64_t item) {
    int lo = 0, hi = nscans - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (scans[mid].tile0 <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <int CAP, int G, int COV, bool WIN, bool DEL, int HOST = 0>
__device__ __forceinline__ void process_tile(const Grid& g, const Grid& dg, const float* __restrict__ q, int64_t n0,
                                             int cnt, const TileArgs& a, float rho0, int32_t* __restrict__ idx,
                                             float* __restrict__ d2, float* __restrict__ cov) {
    if constexpr (CAP > 0) {
        __shared__ __align__(16) unsigned char smem[group_warp_smem(CAP, G)];
        group_unit<CAP, G, COV, WIN, DEL, HOST>(g, dg, q + 3 * n0, cnt, a, rho0, idx + n0 * a.k, d2 + n0 * a.k,
                                          cov ? cov + 6 * n0 : nullptr, smem);
    } else {
        __shared__ u64 pend[8][64];
        warp_tile<COV != 0, DEL>(g, dg, q, n0, cnt, a, rho0, idx, d2, cov, pend[threadIdx.x >> 5], threadIdx.x & 31);
    }
}

// Threads of a block and, for the group search, blocks an SM should hold: 32
// one-warp blocks (64 registers, 5 KB each), 24 (80 registers) with 64 sorted
// survivors, and with eight lanes a query under a window, with weights or over
// two grids, which spill up to 190 bytes at 64: calls of 300 to 4,000 queries,
// k = 10 to 20, take 20-23 us with 64 and 18-21 with 80 registers (of 20,000, 29
// and 27). The plain form does not spill and gains nothing.
constexpr int block_threads(int cap) { return cap ? 32 : 256; }
constexpr int block_target(int cap, bool heavy) { return cap == 32 ? (heavy ? 24 : 32) : cap == 64 ? 24 : 1; }
constexpr bool heavy_form(int g, int cov, bool win, bool del) { return g == 8 && (cov == 2 || win || del); }

template <int CAP, int G, int COV, bool WIN, int HOST = 0>
__global__ void __launch_bounds__(block_threads(CAP), block_target(CAP, heavy_form(G, COV, WIN, false)))
    k_knn(Grid g, const float* __restrict__ q, int64_t N, int tile, TileArgs a, float rho0, int32_t* __restrict__ idx,
          float* __restrict__ d2, float* __restrict__ cov) {
    const int64_t t = work_item<CAP>((N + tile - 1) / tile, a.last_first);
    if (t < 0) return;
    const int64_t n0 = t * tile;
    process_tile<CAP, G, COV, WIN, false, HOST>(g, g, q, n0, (int)min((int64_t)tile, N - n0), a, rho0, idx, d2, cov);
}

// Batched form: work items are the (scan, tile) pairs of the scans'
// prefix-summed tile table, found by a binary search over the table.
template <int CAP, int G, int COV, bool WIN, int HOST = 0>
__global__ void __launch_bounds__(block_threads(CAP), block_target(CAP, heavy_form(G, COV, WIN, false)))
    k_knn_batch(Grid g, const ScanDesc* __restrict__ scans, int nscans, int64_t total_tiles, int tile, TileArgs a,
                float rho0) {
    const int64_t item = work_item<CAP>(total_tiles, a.last_first);
    if (item < 0) return;
    const ScanDesc sd = scans[scan_of_item(scans, nscans, item)];
    const int64_t n0 = (item - sd.tile0) * tile;
    process_tile<CAP, G, COV, WIN, false, HOST>(g, g, sd.q, n0, (int)min((int64_t)tile, sd.n - n0), a, rho0, sd.idx,
                                                sd.d2, sd.cov);
}

// Search over a map grown by appended points: the main grid g and the
// appended-points grid dg as one map (indices of dg's points follow g's).
template <int CAP, int G, int COV, bool WIN>
__global__ void __launch_bounds__(block_threads(CAP), block_target(CAP, heavy_form(G, COV, WIN, true)))
    k_knn_union(Grid g, Grid dg, const float* __restrict__ q, int64_t N, int tile, TileArgs a, float rho0,
                int32_t* __restrict__ idx, float* __restrict__ d2, float* __restrict__ cov) {
    const int64_t t = work_item<CAP>((N + tile - 1) / tile, a.last_first);
    if (t < 0) return;
    const int64_t n0 = t * tile;
    process_tile<CAP, G, COV, WIN, true>(g, dg, q, n0, (int)min((int64_t)tile, N - n0), a, rho0, idx, d2, cov);
}

// Outputs in mapped host memory off 128-byte lines (k <= 32): scans packed one
// after another, a slice of a larger array.  Bounded by the host link (186 GB/s
// of plain copies).  A warp's own rows, stored 128 bytes at a time, run at its
// rate where those are whole lines and far below where each one straddles two,
// so there a block of four warps answers HOST_WARPS units (32 queries, or 16
// with eight lanes each), stages their rows in shared memory and writes each
// array's rows as one block of 16-byte vectors where the row base allows it,
// with one mark (k_knn_rest reads them back over the link).  us for 1M queries,
// 2M map, one scan starting on a line / one row after it, and 16 scans packed:
//   k = 20: one-warp units 1052 / 1739, 1437; staged 1058 / 1172, 1126
//   k = 10:                 794 / 1166, 1115;         777 /  994,  873
//   k = 32:                1563 / 1654, 1639;        1583 / 1611, 1601
// 131k queries, k = 20: 177 / 278, 232; 185 / 197, 186.  In a step of 1.45M
// points, blocks of 640, 1280 and 2560 bytes (one, two, four warps) reach 147,
// 156 and 162 GB/s; eight warps would not fit 48 KB.
constexpr int HOST_WARPS = 4;
__host__ __device__ constexpr size_t host_stage_bytes(int tile, int k) {
    return (size_t)tile * (2 * k + 6) * sizeof(uint32_t);
}

// n words from shared to global or host memory, by all threads of the block.
__device__ __forceinline__ void copy_rows(void* __restrict__ to, const uint32_t* __restrict__ from, int n) {
    uint32_t* const dst = static_cast<uint32_t*>(to);
    const int wide = ((reinterpret_cast<uintptr_t>(to) | reinterpret_cast<uintptr_t>(from)) & 15) == 0 ? n >> 2 : 0;
    for (int i = threadIdx.x; i < wide; i += blockDim.x)
        reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(from)[i];
    for (int i = 4 * wide + threadIdx.x; i < n; i += blockDim.x) dst[i] = from[i];
}

template <int CAP, int G, int COV, bool WIN>
__device__ __forceinline__ void host_tile(const Grid& g, const float* __restrict__ q, int64_t n0, int cnt,
                                          const TileArgs& a, float rho0, int32_t* __restrict__ idx,
                                          float* __restrict__ d2, float* __restrict__ cov) {
    constexpr int WQ = 32 / G, TILE = HOST_WARPS * WQ;
    __shared__ __align__(16) unsigned char smem[HOST_WARPS][group_warp_smem(CAP, G)];
    extern __shared__ __align__(16) uint32_t stage[];  // idx rows, d2 rows, covariances of the tile
    const int w = threadIdx.x >> 5, k = a.k, first = w * WQ;
    uint32_t* const sd = stage + TILE * k;
    uint32_t* const sc = sd + TILE * k;
    const bool left = group_unit<CAP, G, COV, WIN, false, 2>(
        g, g, q + 3 * (n0 + first), min(max(cnt - first, 0), WQ), a, rho0, reinterpret_cast<int32_t*>(stage) + first * k,
        reinterpret_cast<float*>(sd) + first * k, cov ? reinterpret_cast<float*>(sc) + 6 * first : nullptr, smem[w]);
    if (__syncthreads_or(left) && threadIdx.x == 0) sd[0] |= UNIT_FLAG;  // copied by thread 0
    copy_rows(idx + n0 * k, stage, cnt * k);
    copy_rows(d2 + n0 * k, sd, cnt * k);
    if (COV && cov != nullptr) copy_rows(cov + 6 * n0, sc, cnt * 6);
}

constexpr int host_blocks(int cap) { return cap == 32 ? 8 : 5; }  // what shared memory and 64 (102) registers allow

template <int CAP, int G, int COV, bool WIN>
__global__ void __launch_bounds__(32 * HOST_WARPS, host_blocks(CAP))
    k_knn_host(Grid g, const float* __restrict__ q, int64_t N, int tile, TileArgs a, float rho0,
               int32_t* __restrict__ idx, float* __restrict__ d2, float* __restrict__ cov) {
    const int64_t t = work_item<CAP>((N + tile - 1) / tile, a.last_first);
    if (t < 0) return;
    const int64_t n0 = t * tile;
    host_tile<CAP, G, COV, WIN>(g, q, n0, (int)min((int64_t)tile, N - n0), a, rho0, idx, d2, cov);
}

template <int CAP, int G, int COV, bool WIN>
__global__ void __launch_bounds__(32 * HOST_WARPS, host_blocks(CAP))
    k_knn_host_batch(Grid g, const ScanDesc* __restrict__ scans, int nscans, int64_t total_tiles, int tile, TileArgs a,
                     float rho0) {
    const int64_t item = work_item<CAP>(total_tiles, a.last_first);
    if (item < 0) return;
    const ScanDesc sd = scans[scan_of_item(scans, nscans, item)];
    const int64_t n0 = (item - sd.tile0) * tile;
    host_tile<CAP, G, COV, WIN>(g, sd.q, n0, (int)min((int64_t)tile, sd.n - n0), a, rho0, sd.idx, sd.d2, sd.cov);
}

__global__ void k_cov(Grid g, const int32_t* __restrict__ idx, int64_t N, int k, float eps,
                      float* __restrict__ cov) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    cov_row(g, idx + n * k, 1, k, eps, cov + 6 * n, true);
}

// The search kernel of FORM (0 one scan, 1 batched, 2 union; into host memory,
// groups only: 3 and 4 ragged, 5 and 6 on lines) and WIN for mode
// = search_mode(k) and `group` lanes per query of the group search; cov 0 none,
// 1 plain, 2 weighted by a kernel descriptor.  (Weighted covariances have
// kernels of their own: the descriptors' code beside the plain sums cost the
// plain search 10 % in instruction fetches.)
template <int FORM, bool WIN, int CAP, int G, int COV>
void* form_kernel() {
    if constexpr (FORM == 0) return (void*)k_knn<CAP, G, COV, WIN>;
    else if constexpr (FORM == 1) return (void*)k_knn_batch<CAP, G, COV, WIN>;
    else if constexpr (FORM == 2) return (void*)k_knn_union<CAP, G, COV, WIN>;
    else if constexpr (FORM == 3) return (void*)k_knn_host<CAP, G, COV, WIN>;
    else if constexpr (FORM == 4) return (void*)k_knn_host_batch<CAP, G, COV, WIN>;
    else if constexpr (FORM == 5) return (void*)k_knn<CAP, G, COV, WIN, 1>;
    else return (void*)k_knn_batch<CAP, G, COV, WIN, 1>;
}
template <int FORM, bool WIN, int CAP, int G>
void* form_kernel(int cov) {
    if (cov == 0) return form_kernel<FORM < 5 ? FORM : FORM - 5, WIN, CAP, G, 0>();  // nothing to finish
    if (CAP == 0 || cov == 1) return form_kernel<FORM, WIN, CAP, G, 1>();
    return form_kernel<FORM, WIN, CAP, G, CAP == 0 ? 1 : 2>();
}
template <int FORM, bool WIN, int CAP>
void* form_kernel(int cov, int group) {
    return group == 4 ? form_kernel<FORM, WIN, CAP, 4>(cov) : form_kernel<FORM, WIN, CAP, 8>(cov);
}
template <int FORM, bool WIN>
void* knn_kernel(int mode, int cov, int group) {
    if constexpr (FORM < 3)
        if (mode == 2) return form_kernel<FORM, WIN, 0, 1>(cov);
    return mode == 0 ? form_kernel<FORM, WIN, 32>(cov, group) : form_kernel<FORM, WIN, 64>(cov, group);
}

}  // namespace
