// Host-side definitions shared by the library's translation units.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "pc.h"
#include "pc_device.cuh"

constexpr uint32_t PC_MAGIC_LIVE = 0x70637467u;  // "pctg"
constexpr uint32_t PC_MAGIC_DEAD = 0xdeadbeefu;

// Kernel-descriptor weights of the covariance (pc_set_cov_kernel), as the
// device sees them: s = sigma (RBF), 1 / (2 sigma^2) (Gaussian) or
// 1 / sigma (Laplacian); o = the target's bounding-box minimum.
struct CovKernel {
    int type;
    float s, alpha, c, d;
    float ox, oy, oz;
};

// Where a search's outputs lie: device memory, or mapped page-locked host memory
// with every array on a 128-byte line, or off one.
enum class Out { device, host_lines, host_ragged };

// What a search launch passes to its kernels besides the grid and buffers.
struct TileArgs {
    int k;
    float eps;
    int last_first;  // issue tiles from the end of the query array
    CovKernel ck;    // kernel-descriptor weights; type 0: the plain covariance
    int finish;      // group search: regularise in the search (outputs in host memory) instead of in k_knn_rest
    float probe_c;   // > 0: every query estimates its own starting radius (probe_radius)
};

// One scan of a batched launch, as the batched kernel reads it from the scan table.
struct ScanDesc {
    const float* q;
    int64_t n;
    int32_t* idx;
    float* d2;
    float* cov;     // may be null: no covariance for this scan
    int64_t tile0;  // first work item of this scan
};

struct pc_target_s {
    uint32_t magic;
    int device;
    pcdev::Grid g;        // kernel view; the pointers below back it
    pc_build_opts opts;
    pc_tune tune;
    float bbox_max[3];
    float rho_hint[64];
    int uneven;  // the calibration's k-th-neighbour distances spread widely (p90 / p25 > 1.55)
    int64_t table_cap;
    int64_t device_bytes;
    // owned device memory
    uint4* table;
    float4* pts;
    float4* xyz;
    unsigned long long* cell_keys;
    uint32_t* cell_start;
    uint32_t* dstart;
    uint2* xcut;  // sub-cell cut of the row index (Grid::xcut), or null
    int* status;  // 64 bytes: status word, then 4 u64 statistics counters at +32
    // staging for pc_knn_cov_host, grown on demand
    void* stage;
    size_t stage_bytes;
    CovKernel ck;  // covariance weights (type 0: none)
    // incremental updates (pc_target_append): the appended points, f32
    // [delta_m, 3] in append order, and a grid over them; their indices
    // follow the main map's (M + position)
    pc_target_s* delta;
    float* delta_xyz;
    int64_t delta_m, delta_cap;
    // the window of pc_set_window, kept to re-apply to a rebuilt delta grid
    pc_window win;
    int has_win;
};

struct pc_batch_s {
    uint32_t magic;
    pc_target_s* t;
    pcdev::Grid g;  // the target's view when planned (window included)
    CovKernel ck;   // and its covariance weights
    int n_scans;
    int k;
    float eps;
    bool with_cov;
    Out out;
    int tile;
    int warps;
    int64_t total_tiles;
    int64_t total_queries;
    ScanDesc* scans_dev;
    cudaGraph_t graph;
    cudaGraphExec_t exec;
    cudaStream_t captured_on;
};

// The whole grid as the search window (no point tests).
inline void pc_clear_window(pcdev::Grid& g) {
    g.windowed = 0;
    g.wlx = 0;
    g.whx = g.dimx - 1;
    g.wly = 0;
    g.why = g.dimy - 1;
    g.wlz = 0;
    g.whz = g.dimz - 1;
    g.tlx = g.thx = g.tly = g.thy = g.tlz = g.thz = -1;
    g.wlox = g.wloy = g.wloz = -INFINITY;
    g.whix = g.whiy = g.whiz = INFINITY;
}

// mem.cu: device memory of targets on the current device, ready for use in
// the order of stream s.  pc_dev_free: after the work queued on s.
cudaError_t pc_dev_alloc(void** out, size_t bytes, cudaStream_t s);
void pc_dev_free(void* ptr, cudaStream_t s);
// cudaMalloc that asks the pool for its unused memory before it fails.
cudaError_t pc_plain_alloc(void** out, size_t bytes);
// A target's fence, usable as memory; freeing it waits for the device.
// pc_dev_free_idle frees it and then the pool memory at ptrs, for any stream's
// users and while any thread captures.
cudaError_t pc_fence_alloc(void** out, size_t bytes);
void pc_dev_free_idle(void* fence, void* const* ptrs, int n);

// Calls that wait for the device, or allocate, leave captures in progress alone.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    RelaxedCapture(const RelaxedCapture&) = delete;
};

// grid_build.cu
pc_status pc_build_grid(const float* xyz, int64_t M, const pc_build_opts& o, cudaStream_t s,
                        pc_target_s* t);
void pc_free_grid(pc_target_s* t);
// Every (M / n)-th point of the target in caller order, to q [n, 3].
cudaError_t pc_launch_sample(const pc_target_s* t, int64_t n, float* q, cudaStream_t s);
// Over n <= 1024 rows of kc <= 64 squared distances: out[k] = the 75th
// percentile of column k's finite distances (0: none), out[64], out[65] = the
// 25th and 90th of column min(kc, 16) - 1.
cudaError_t pc_launch_rho_hints(const float* d2, int n, int kc, float* out, cudaStream_t s);
size_t pc_sort_temp_words(int64_t n);
cudaError_t pc_radix_sort_pairs(unsigned long long** keys, uint32_t** vals, unsigned long long* keys_alt,
                                uint32_t* vals_alt, int64_t n, int nbits, uint32_t* temp, cudaStream_t s);
size_t pc_scan_temp_words(int64_t n);
cudaError_t pc_scan_exclusive(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total_dev,
                              uint32_t* temp, cudaStream_t s);

// The search kernels' translation units (whole-map / window variants, with or
// without appended points): form 0 one scan, 1 batched, 2 union; k <= 32 into
// host memory: 3 one scan and 4 batched, ragged, 5 and 6 the same on lines;
// group: lanes per query of the group search (k <= 32).
void* pc_knn_kernel_win(int form, int mode, int cov, int group);
void* pc_knn_kernel_batch(int mode, int cov, int group);
void* pc_knn_kernel_batch_win(int mode, int cov, int group);
void* pc_knn_kernel_union(int mode, int cov, int group);
void* pc_knn_kernel_union_win(int mode, int cov, int group);
void* pc_knn_kernel_host(int host_form, int mode, int cov, int group);
void* pc_knn_kernel_host_win(int host_form, int mode, int cov, int group);

// knn_cov.cu
cudaError_t pc_launch_knn(const pc_target_s* t, const float* q, int64_t N, int k, float eps,
                          int32_t* idx, float* d2, float* cov, float rho0, cudaStream_t s, Out out = Out::device);
// Loads every search kernel on the current device (once; called by the first
// build, so that no search or capture is the first to launch one).
cudaError_t pc_knn_prepare();
cudaError_t pc_rest_prepare();
// Queries of one work item of a search over n queries (k <= 32: a unit of the
// group search, or a block's units into ragged host memory; else the tune's tile).
int pc_search_tile(const pc_target_s* t, int k, int64_t n, Out out);
cudaError_t pc_launch_cov(const pc_target_s* t, const int32_t* idx, int64_t N, int k, float eps,
                          float* cov, cudaStream_t s);
cudaError_t pc_launch_knn_batch(const pc_target_s* t, const pcdev::Grid& g, const CovKernel& ck,
                                const ScanDesc* scans_dev, int nscans, int64_t total_tiles, int64_t queries,
                                int tile, int warps, int k, float eps, bool with_cov, Out out, float rho0,
                                cudaStream_t s);

// knn_rest.cu: the queries that a group search (k <= 32) over the same
// arguments left unanswered; dg: the appended points' grid, or null.
cudaError_t pc_launch_rest(const pcdev::Grid& g, const pcdev::Grid* dg, const float* q, int64_t N, int tile,
                           const TileArgs& a, float rho0, int32_t* idx, float* d2, float* cov, cudaStream_t s);
cudaError_t pc_launch_rest_batch(const pcdev::Grid& g, const ScanDesc* scans_dev, int nscans, int64_t total_tiles,
                                 int64_t queries, int tile, const TileArgs& a, float rho0, cudaStream_t s);

// gicp.cu
size_t pc_gicp_work_size();
cudaError_t pc_launch_gicp_linearize(const pc_target_s* t, const float* map_cov, const float* src,
                                     int64_t n, const float* src_cov, const float* pose,
                                     float max_dist, double* out, int32_t* corr, void* work,
                                     float2 r0, float2 r0d, cudaStream_t s);
cudaError_t pc_launch_gicp_update(const double* lin, float lambda, float* pose, double* xi,
                                  cudaStream_t s);

// delta.cu: covariances and packing over the main grid plus the delta grid
cudaError_t pc_launch_cov_union(const pc_target_s* t, const int32_t* idx, int64_t N, int k, float eps,
                                float* cov, cudaStream_t s);
cudaError_t pc_launch_pack_xyz(const pc_target_s* t, float* out, cudaStream_t s);

// pc_api.cu
float pc_rho0(const pc_target_s* t, int k);
// The probe constant of the group search's per-query starting radius (0: off).
float pc_probe_c(const pc_target_s* t);
// Launch shape of a batched call over caller-provided scans.
struct BatchShape {
    int64_t tiles;  // work items (tiles of `tile` queries) over all scans; 0: nothing to do
    int tile, warps;
    int64_t queries;
    bool any_cov;   // some scan asks for covariances
    Out out;        // where some output lies that is not device memory
};
// Argument checks and scan table shared by pc_batch_plan,
// pc_batch_run_scratch and pc_batch_run_noalloc; fills table[0, n_scans)
// with the addresses kernels use (mapped host memory translated).
pc_status pc_batch_table(const pc_target_s* t, const pc_scan* scans, int n_scans, int k, float eps,
                         ScanDesc* table, BatchShape* shape);
pc_status pc_from_cuda(cudaError_t e);
bool pc_target_is_live(const pc_target_s* t);
bool pc_is_device_ptr(const void* p);
