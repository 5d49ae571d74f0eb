// Search kernels that write mapped host memory, whole-map variant
// (knn_host_win.cu: window variant).
#include "knn_kernels.cuh"

void* pc_knn_kernel_host(int form, int mode, int cov, int group) {
    return form == 3   ? knn_kernel<3, false>(mode, cov, group)
           : form == 4 ? knn_kernel<4, false>(mode, cov, group)
           : form == 5 ? knn_kernel<5, false>(mode, cov, group)
                       : knn_kernel<6, false>(mode, cov, group);
}
