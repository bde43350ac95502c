// temporal_r32c.cu -- k_temporal launchers for FP32 planes with ragged rows, depths 7-8.
#include "temporal_launch.cuh"

RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 7)
RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 8)
