// pss_kern_line_f32.cu -- FP32 instantiation of the 1D runs (k_line).
#include "pss_line.cuh"

namespace pss {
template cudaError_t launch_line<float>(const LineArgs<float> &, int, cudaStream_t);
}
