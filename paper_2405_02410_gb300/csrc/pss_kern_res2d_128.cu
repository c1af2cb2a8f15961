// pss_kern_res2d_128.cu -- the cluster-resident 2D step for rows of 128 points
// (a translation unit per row length so that nvcc builds them in parallel).
#include "pss_resident2d.cuh"

namespace pss {
template cudaError_t launch_res2_nx<128>(const Res2Args &, int, cudaStream_t, int *);
}
