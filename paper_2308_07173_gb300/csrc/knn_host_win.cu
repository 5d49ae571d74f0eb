// Window variant of the search kernels that write mapped host memory.
#include "knn_kernels.cuh"

void* pc_knn_kernel_host_win(int host_form, int mode, int cov, int group) {
    return host_form == 3 ? knn_kernel<3, true>(mode, cov, group) : knn_kernel<4, true>(mode, cov, group);
}
