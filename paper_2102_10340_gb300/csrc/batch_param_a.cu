// batch_param_a.cu -- k_batch_param launchers, one halo lane, depths 1-4.
#include "batch_kernels.cuh"

RDK_INSTANTIATE_BATCH_PARAM(1, 1)
RDK_INSTANTIATE_BATCH_PARAM(2, 1)
RDK_INSTANTIATE_BATCH_PARAM(3, 1)
RDK_INSTANTIATE_BATCH_PARAM(4, 1)
