// Nearest-points search and neighbourhood covariance on sm_103a CUDA cores
// (Sec. III-C1 "Efficient registration method": the per-point covariances
// C_i of Eq. 19 need every point's k nearest neighbours and the covariance
// of that neighbourhood -- the step the paper moves from CPU to GPU).
//
// Exactness rests on one fact, certified_tau: for a box of cells around q,
// every target point outside the box has a binary32 d2 above a computable
// tau, so any radius t with t^2 <= tau that holds >= k points holds the k
// nearest.  Two searches use it:
//
// * Group search (k <= 32; group_unit): four or eight lanes per query walk
//   the rows of the box (one contiguous point range per row), keep the points
//   within the radius in shared memory, and sort the survivors by (d2, index).
// * Warp path (k > 32, and in knn_rest.cu the group search's leftovers;
//   knn_search): one query per warp, the rows of a widening box read one per
//   lane (cells through the hash where there is no row index), candidates 32
//   at a time, survivors merged into a register top-k by bitonic shuffles.
//
// The covariance is a two-pass binary32 mean/centred sum shifted by the
// nearest neighbour; for eps >= 0 a closed-form binary32 eigen-solve gives
// the normal n and C' = I - (1-eps) n n^T.  Nothing here changes a result bit
// with the tile, launch shape, radii, tile order or batching.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "knn_kernels.cuh"

// ---------------------------------------------------------------- host side
namespace {

// The search mode for k on this target: its tune may ask for 64 survivor
// slots (mode 1) for every k <= 32.
int target_mode(const pc_target_s* t, int k) {
    const int m = search_mode(k);
    return (m == 0 && t->tune.slots == 64) ? 1 : m;
}
int clamp_warps(int w) { return w <= 0 ? 4 : (w > 8 ? 8 : w); }

// Lanes per query of the group search.  Eight shorten a query's chain of
// dependent loads where a call cannot fill the chip; four do less work.
// Measured, us with 4 / 8 lanes at 6k, 20k, 48k queries: track map, k = 20
// 29 / 22, 32 / 29, 40 / 48; k = 10 27 / 21, 27 / 24, 34 / 37; k = 32 41 / 27,
// 42 / 33, 51 / 55; uniform box, k = 20 46 / 34, 53 / 50, 78 / 80.
int group_lanes(int64_t n) { return n <= 24576 ? 8 : 4; }

// The forms of pc_internal.h, as one scan (0) or batched (1) and where the outputs lie.
int host_form(int form, Out out, int mode) {
    return mode == 2 || out == Out::device ? form : form + (out == Out::host_ragged ? 3 : 5);
}
void* search_kernel(int form, bool windowed, int mode, int cov, int group) {
    if (form >= 3)
        return windowed ? pc_knn_kernel_host_win(form, mode, cov, group) : pc_knn_kernel_host(form, mode, cov, group);
    return windowed    ? pc_knn_kernel_win(form, mode, cov, group)
           : form == 2 ? pc_knn_kernel_union(mode, cov, group)
           : form == 1 ? pc_knn_kernel_batch(mode, cov, group)
                       : knn_kernel<0, false>(mode, cov, group);
}

// Launches the search kernel of (form, mode, covariance kind, window) over
// its work items: one per one-warp block of the group search, one per block of
// its host forms, one per warp of the warp path.
cudaError_t launch_form(int form, const Grid& g, int mode, int cov, int64_t tiles, int tile, int warps, int k,
                        void** args, cudaStream_t s) {
    if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
    const bool blocks = form == 3 || form == 4;
    const int group = mode < 2 ? 32 * (blocks ? HOST_WARPS : 1) / tile : 1;
    void* kern = search_kernel(form, g.windowed != 0, mode, cov, group);
    const int items = mode < 2 ? 1 : warps, threads = 32 * (mode == 2 ? warps : blocks ? HOST_WARPS : 1);
    return cudaLaunchKernel(kern, dim3((unsigned)((tiles + items - 1) / items)), dim3(threads), args,
                            blocks ? host_stage_bytes(tile, k) : 0, s);
}

int cov_kind(bool with_cov, const CovKernel& ck) { return !with_cov ? 0 : (ck.type == 0 ? 1 : 2); }

TileArgs tile_args(const pc_target_s* t, const CovKernel& ck, int k, float eps, Out out) {
    return TileArgs{k, eps, t->tune.order == 0 ? 1 : 0, ck, out == Out::device ? 0 : 1, pc_probe_c(t)};
}

}  // namespace

// A kernel that has not run yet is loaded by its first launch, which takes
// device memory (2 MB at a time) and 0.7 ms more: too late for the entries that
// promise not to allocate, and for the first scan served.
cudaError_t pc_knn_prepare() {
    static std::mutex mu;
    static uint64_t done = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done >> dev & 1) return cudaSuccess;
    cudaFuncAttributes at;
    for (int form = 0; form < 7; ++form)
        for (int win = 0; win < 2; ++win)
            for (int mode = 0; mode < (form < 3 ? 3 : 2); ++mode)
                for (int cov = 0; cov < (mode == 2 ? 2 : 3); ++cov)
                    for (int group = 4; group <= (mode == 2 ? 4 : 8); group += 4)
                        if ((e = cudaFuncGetAttributes(&at, search_kernel(form, win != 0, mode, cov, group))) !=
                            cudaSuccess)
                            return e;
    if ((e = pc_rest_prepare()) != cudaSuccess) return e;
    done |= 1ull << dev;
    return cudaSuccess;
}

// 32 warps an SM, of which 20 are resident at once (the warp path takes 92
// registers). 20k queries, k = 48 on a 300k map, with 20, 32, 48 warps an SM: 89,
// 84, 96 us; 40k: 154, 138, 142; 131k: 417, 381, 368.
constexpr int64_t WARP_PATH_WARPS = 152 * 32;

int pc_search_tile(const pc_target_s* t, int k, int64_t n, Out out) {
    if (target_mode(t, k) < 2) return 32 * (out == Out::host_ragged ? HOST_WARPS : 1) / group_lanes(n);
    // The warp path answers a tile's queries one after another on one warp
    // (each starts from the last one's radius): tiles shrink until a call has
    // WARP_PATH_WARPS.  20k queries, k = 48 on a 300k map, tiles of 32 (4 warps an
    // SM): 188 us, of 4: 84.
    // Not where the exact scan may not follow (exhaustive = 0): there the radius
    // a query starts from decides whether it is answered, and must not depend
    // on the size of the call.
    const int most = t->tune.tile <= 0 ? 32 : std::min(t->tune.tile, 32);
    if (!t->g.exhaustive) return most;
    return (int)std::max<int64_t>(1, std::min<int64_t>(most, n / WARP_PATH_WARPS));
}

// The covariance (plain, or weighted by the target's kernel descriptor) is
// fused into the search.  With appended points the main grid and the delta
// grid are searched as one map.
cudaError_t pc_launch_knn(const pc_target_s* t, const float* q, int64_t N, int k, float eps,
                          int32_t* idx, float* d2, float* cov, float rho0, cudaStream_t s,
                          Out out) {
    if (N == 0) return cudaSuccess;
    if (t->delta) out = Out::device;  // the union search has no host forms; its rows may lie anywhere
    const int mode = target_mode(t, k), warps = clamp_warps(t->tune.warps);
    const int tile = pc_search_tile(t, k, N, out);
    const int64_t tiles = (N + tile - 1) / tile;
    TileArgs a = tile_args(t, t->ck, k, eps, out);
    Grid g = t->g, dg = t->delta ? t->delta->g : t->g;
    cudaError_t e;
    if (t->delta) {
        void* args[] = {&g, &dg, (void*)&q, (void*)&N, (void*)&tile, &a, &rho0, &idx, &d2, &cov};
        e = launch_form(2, g, mode, cov_kind(cov != nullptr, t->ck), tiles, tile, warps, k, args, s);
    } else {
        void* args[] = {&g, (void*)&q, (void*)&N, (void*)&tile, &a, &rho0, &idx, &d2, &cov};
        e = launch_form(host_form(0, out, mode), g, mode, cov_kind(cov != nullptr, t->ck), tiles, tile, warps, k, args, s);
    }
    if (e != cudaSuccess || mode == 2) return e;
    return pc_launch_rest(g, t->delta ? &dg : nullptr, q, N, tile, a, rho0, idx, d2, cov, s);
}

cudaError_t pc_launch_cov(const pc_target_s* t, const int32_t* idx, int64_t N, int k, float eps,
                          float* cov, cudaStream_t s) {
    if (N == 0) return cudaSuccess;
    const int threads = 128;
    const int64_t blocks = (N + threads - 1) / threads;
    k_cov<<<(unsigned)blocks, threads, 0, s>>>(t->g, idx, N, k, eps, cov);
    return cudaGetLastError();
}

cudaError_t pc_launch_knn_batch(const pc_target_s* t, const Grid& gv, const CovKernel& ck,
                                const ScanDesc* scans_dev, int nscans, int64_t total_tiles, int64_t queries,
                                int tile, int warps, int k, float eps, bool with_cov, Out out, float rho0,
                                cudaStream_t s) {
    if (total_tiles == 0) return cudaSuccess;
    const int mode = target_mode(t, k);
    TileArgs a = tile_args(t, ck, k, eps, out);
    Grid g = gv;
    void* args[] = {&g, (void*)&scans_dev, &nscans, &total_tiles, &tile, &a, &rho0};
    const cudaError_t e =
        launch_form(host_form(1, out, mode), g, mode, cov_kind(with_cov, ck), total_tiles, tile, warps, k, args, s);
    if (e != cudaSuccess || mode == 2) return e;
    return pc_launch_rest_batch(g, scans_dev, nscans, total_tiles, queries, tile, a, rho0, s);
}
