// temporal_r32b.cu -- k_temporal launchers for FP32 planes with ragged rows, depths 5-6.
#include "temporal_launch.cuh"

RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 5)
RDK_INSTANTIATE_TEMPORAL(rdk::Ragged<float>, 6)
