// resident_v4.cu -- the cluster-resident kernel, 4 values per lane.
#include "resident_launch.cuh"

template RDK_RESIDENT_SIG(4);
