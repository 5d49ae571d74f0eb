// Search kernels that write mapped host memory, window variant.
#include "knn_kernels.cuh"

void* pc_knn_kernel_host_win(int form, int mode, int cov, int group) {
    return form == 3   ? knn_kernel<3, true>(mode, cov, group)
           : form == 4 ? knn_kernel<4, true>(mode, cov, group)
           : form == 5 ? knn_kernel<5, true>(mode, cov, group)
                       : knn_kernel<6, true>(mode, cov, group);
}
