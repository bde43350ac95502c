// resident_v12.cu -- the cluster-resident kernel, 12 values per lane.
#include "resident_launch.cuh"

template RDK_RESIDENT_SIG(12);
