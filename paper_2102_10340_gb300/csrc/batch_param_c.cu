// batch_param_c.cu -- k_batch_param launchers, two halo lanes, depths 5-6.
#include "batch_kernels.cuh"

RDK_INSTANTIATE_BATCH_PARAM(5, 2)
RDK_INSTANTIATE_BATCH_PARAM(6, 2)
