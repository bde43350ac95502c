// batch_param_d.cu -- k_batch_param launchers, two halo lanes, depths 7-8.
#include "batch_kernels.cuh"

RDK_INSTANTIATE_BATCH_PARAM(7, 2)
RDK_INSTANTIATE_BATCH_PARAM(8, 2)
