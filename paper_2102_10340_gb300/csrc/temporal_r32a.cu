// temporal_r32a.cu -- k_temporal launchers for FP32 planes with ragged rows, depths 1-4.
#include "temporal_launch.cuh"

RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 1)
RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 2)
RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 3)
RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 4)
