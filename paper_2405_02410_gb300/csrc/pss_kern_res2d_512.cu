// pss_kern_res2d_512.cu -- the cluster-resident 2D step for rows of 512 points
// (a translation unit per row length so that nvcc builds them in parallel).
#include "pss_resident2d.cuh"

namespace pss {
template cudaError_t launch_res2_nx<512>(const Res2Args &, int, cudaStream_t, int *);
}
