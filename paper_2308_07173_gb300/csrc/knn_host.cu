// Search kernels that write mapped host memory, whole-map variant
// (knn_host_win.cu: window variant).  host_form: 3 one scan, 4 batched.
#include "knn_kernels.cuh"

void* pc_knn_kernel_host(int host_form, int mode, int cov, int group) {
    return host_form == 3 ? knn_kernel<3, false>(mode, cov, group) : knn_kernel<4, false>(mode, cov, group);
}
