// Window variant of the search kernels (pc_set_window): the same code as
// the whole-map kernels with WIN = true, so rows on the window's boundary
// cells test each point against the window box.
#include "knn_kernels.cuh"

void* pc_knn_kernel_win(int form, int mode, int cov, int group) {
    return form == 2   ? pc_knn_kernel_union_win(mode, cov, group)
           : form == 1 ? pc_knn_kernel_batch_win(mode, cov, group)
                       : knn_kernel<0, true>(mode, cov, group);
}
