// resident_v8.cu -- the cluster-resident kernel, 8 values per lane.
#include "resident_launch.cuh"

template RDK_RESIDENT_SIG(8);
