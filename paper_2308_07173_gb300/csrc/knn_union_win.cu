// Window variant of the union search kernels (knn_union.cu): rows on the
// window's boundary cells of either grid test each point against the window.
#include "knn_kernels.cuh"

void* pc_knn_kernel_union_win(int mode, int cov, int group) {
    return knn_kernel<2, true>(mode, cov, group);
}
