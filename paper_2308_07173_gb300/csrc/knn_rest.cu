// The queries that the group search (k <= 32, knn_kernels.cuh) left
// unanswered: those whose k-th neighbour lies beyond the reach of its
// lane-parallel attempts (a scan's sparse rim, points off the map), and those
// with more equal distances than it sorts.  They come in clusters (32 in one
// tile, many adjacent tiles), and one such query costs a warp tens of
// microseconds, so answering them inside their own tile's warp, as the
// search did before, set the end of the launch: up to 0.9 ms on a scan whose
// other queries took 0.1 ms.
//
// Here every warp answers one query at a time.  A block reads the marks of
// 32 work items (units of up to 8 queries; into ragged host memory up to
// 32 queries with one mark), strided by the grid so that neighbouring ones fall to
// different blocks, and its 8 warps take a marked item's rows.  The grid fills
// the chip from 608 items on: leftovers, not marks, take the time (60k queries
// around 40 tight clusters into host memory: 22.2 ms with a block per 32 items,
// 5.6 with the staged search before groups, 3.6 now).
//
// First the block turns its units' covariances into C' = I - (1 - eps) n n^T
// (eps >= 0; done in the search into host memory), one query per lane.  Inside the search this ran on one warp of
// a block while the others idled, or on 8 of 32 lanes: 10 of 73 us of the
// 131k scan, k = 20.  Rows without a value (NAN_ROW) are left alone, among
// them the unanswered ones, which get theirs complete.
#include "knn_kernels.cuh"

namespace {

constexpr int REST_WARPS = 8;
constexpr int REST_BLOCKS = 608;  // 4 per SM

struct RestTile {
    const float* q;
    int32_t* idx;
    uint32_t* d2;  // bits of the squared distances
    float* cov;
    int64_t n0;
    int cnt;
};

template <bool DEL, typename F>
__device__ __forceinline__ void rest_body(const Grid& g, const Grid& dg, int64_t tiles, int64_t queries, const TileArgs& a,
                                          float rho0, F&& tile_at) {
    __shared__ u64 s_pend[REST_WARPS][64];
    __shared__ int32_t s_nb[REST_WARPS][32];
    __shared__ unsigned s_marked;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = a.k;
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&g.stats[0], (unsigned long long)queries);
    const bool regularise = a.eps >= 0.0f && !a.finish;
    cudaGridDependencySynchronize();  // the search's rows and marks are complete and visible
    for (int64_t base = blockIdx.x; base < tiles; base += (int64_t)32 * gridDim.x) {
        if (warp == 0) {
            const int64_t t = base + (int64_t)lane * gridDim.x;
            bool marked = false;
            if (t < tiles) {
                const RestTile r = tile_at(t);
                marked = (r.d2[r.n0 * k] & UNIT_FLAG) != 0u;
            }
            const unsigned b = __ballot_sync(FULL, marked);
            if (lane == 0) s_marked = b;
        }
        if (regularise) {
            const int64_t t = base + (int64_t)(threadIdx.x >> 3) * gridDim.x;
            if (t < tiles) {
                const RestTile r = tile_at(t);
                const int row = threadIdx.x & 7;
                if (row < r.cnt && r.cov != nullptr) {
                    float* const c = r.cov + 6 * (r.n0 + row);
                    float v[6];
                    bool some = false;
#pragma unroll
                    for (int j = 0; j < 6; ++j) {
                        v[j] = c[j];
                        some |= __float_as_uint(v[j]) != NAN_ROW;
                    }
                    if (some) {
                        cov_regularise(v, a.eps);
                        store6(c, v[0], v[1], v[2], v[3], v[4], v[5]);
                    }
                }
            }
        }
        __syncthreads();
        unsigned todo = s_marked;
        __syncthreads();
        while (todo) {
            const int j = __ffs(todo) - 1;
            todo &= todo - 1u;
            const RestTile r = tile_at(base + (int64_t)j * gridDim.x);
            for (int row = warp; row < r.cnt; row += REST_WARPS) {
                const int64_t n = r.n0 + row;
                const unsigned head = r.d2[n * k];
                __syncwarp();
                if (head != UNANSWERED) {
                    if (row == 0 && lane == 0) r.d2[n * k] = head & ~UNIT_FLAG;
                    continue;
                }
                const float qx = __ldg(r.q + 3 * n), qy = __ldg(r.q + 3 * n + 1), qz = __ldg(r.q + 3 * n + 2);
                const float rho1 = rho0 * (g.exhaustive ? START : LIMITED_START);
                float rho = rho1;
                if (!g.exhaustive && a.probe_c > 0.0f)
                    rho = LIMITED_START * probe_radius<32, true>(g, true, qx, qy, qz, k, a.probe_c, lane);
                SearchState<1> S;
                state_reset(S);
                const int sr = g.exhaustive
                                   ? knn_search<1, DEL>(g, dg, qx, qy, qz, k, rho, S, s_pend[warp], lane)
                                   : knn_search<1, DEL, true>(g, dg, qx, qy, qz, k, rho, S, s_pend[warp], lane, rho1);
                const bool ok = sr == SEARCH_OK;
                if (!ok && lane == 0) atomicOr(g.status, sr == SEARCH_SHORT ? ST_SHORT : ST_SEARCH_LIMIT);
                if (lane < k) {
                    const int32_t i = ok ? (int32_t)(uint32_t)S.L[0] : -1;
                    s_nb[warp][lane] = i;
                    r.idx[n * k + lane] = i;
                    r.d2[n * k + lane] = ok ? (uint32_t)(S.L[0] >> 32) : 0x7f800000u;
                }
                __syncwarp();
                if (r.cov != nullptr && lane == 0) cov_row_any<DEL>(g, dg, s_nb[warp], k, a, qx, qy, qz, r.cov + 6 * n);
                __syncwarp();
            }
        }
    }
}

template <bool DEL>
__global__ void __launch_bounds__(32 * REST_WARPS, 4) k_knn_rest(Grid g, Grid dg, const float* q, int64_t N, int tile,
                                                              TileArgs a, float rho0, int32_t* idx, float* d2,
                                                              float* cov) {
    rest_body<DEL>(g, dg, (N + tile - 1) / tile, N, a, rho0, [&](int64_t t) {
        const int64_t n0 = t * tile;
        return RestTile{q, idx, reinterpret_cast<uint32_t*>(d2), cov, n0, (int)min((int64_t)tile, N - n0)};
    });
}

__global__ void __launch_bounds__(32 * REST_WARPS, 4) k_knn_rest_batch(Grid g, const ScanDesc* __restrict__ scans,
                                                                    int nscans, int64_t total_tiles,
                                                                    int64_t queries, int tile, TileArgs a,
                                                                    float rho0) {
    rest_body<false>(g, g, total_tiles, queries, a, rho0, [&](int64_t t) {
        const ScanDesc sd = scans[scan_of_item(scans, nscans, t)];
        const int64_t n0 = (t - sd.tile0) * tile;
        return RestTile{sd.q, sd.idx, reinterpret_cast<uint32_t*>(sd.d2), sd.cov, n0, (int)min((int64_t)tile, sd.n - n0)};
    });
}

// Launched as a programmatic dependent of the search before it on the stream,
// so its blocks are in place when that ends.
template <typename... P>
cudaError_t launch(void (*kern)(P...), int64_t tiles, cudaStream_t s, P... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)std::min<int64_t>(tiles, REST_BLOCKS));
    c.blockDim = dim3(32 * REST_WARPS);
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, args...);
}

}  // namespace

cudaError_t pc_rest_prepare() {
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, k_knn_rest<false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, k_knn_rest<true>);
    return e == cudaSuccess ? cudaFuncGetAttributes(&at, k_knn_rest_batch) : e;
}

cudaError_t pc_launch_rest(const Grid& g, const Grid* dg, const float* q, int64_t N, int tile, const TileArgs& a,
                           float rho0, int32_t* idx, float* d2, float* cov, cudaStream_t s) {
    return launch<Grid, Grid, const float*, int64_t, int, TileArgs, float, int32_t*, float*, float*>(
        dg ? k_knn_rest<true> : k_knn_rest<false>, (N + tile - 1) / tile, s, g, dg ? *dg : g, q, N, tile, a, rho0, idx,
        d2, cov);
}

cudaError_t pc_launch_rest_batch(const Grid& g, const ScanDesc* scans_dev, int nscans, int64_t total_tiles,
                                 int64_t queries, int tile, const TileArgs& a, float rho0, cudaStream_t s) {
    return launch<Grid, const ScanDesc*, int, int64_t, int64_t, int, TileArgs, float>(
        k_knn_rest_batch, total_tiles, s, g, scans_dev, nscans, total_tiles, queries, tile, a, rho0);
}
