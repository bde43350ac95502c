// resident_v2.cu -- the cluster-resident kernel, 2 values per lane.
#include "resident_launch.cuh"

template RDK_RESIDENT_SIG(2);
