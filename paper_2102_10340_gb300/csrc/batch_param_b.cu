// batch_param_b.cu -- k_batch_param launchers, two halo lanes, depths 1-4.
#include "batch_kernels.cuh"

RDK_INSTANTIATE_BATCH_PARAM(1, 2)
RDK_INSTANTIATE_BATCH_PARAM(2, 2)
RDK_INSTANTIATE_BATCH_PARAM(3, 2)
RDK_INSTANTIATE_BATCH_PARAM(4, 2)
