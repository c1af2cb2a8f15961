// pss_kern_line_f64.cu -- FP64 instantiation of the 1D runs (k_line).
#include "pss_line.cuh"

namespace pss {
template cudaError_t launch_line<double>(const LineArgs<double> &, int, cudaStream_t);
}
