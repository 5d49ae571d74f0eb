// Batched search kernels, whole-map variant (knn_batch_win.cu: window variant).
#include "knn_kernels.cuh"

void* pc_knn_kernel_batch(int mode, int cov, int group) { return knn_kernel<1, false>(mode, cov, group); }
