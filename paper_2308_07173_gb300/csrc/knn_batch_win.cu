// Batched search kernels, window variant.
#include "knn_kernels.cuh"

void* pc_knn_kernel_batch_win(int mode, int cov, int group) {
    return knn_kernel<1, true>(mode, cov, group);
}
