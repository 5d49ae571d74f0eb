// Search kernels over a map grown by appended points (pc_target_append):
// the main grid and the appended-points grid searched as one map in the
// same lane and warp paths as the whole-map kernels (knn_kernels.cuh,
// DEL = true).  This unit holds the whole-map variant; knn_union_win.cu the
// window variant.  Both compile in parallel with the other search units.
#include "knn_kernels.cuh"

void* pc_knn_kernel_union(int mode, int cov, int group) { return knn_kernel<2, false>(mode, cov, group); }
