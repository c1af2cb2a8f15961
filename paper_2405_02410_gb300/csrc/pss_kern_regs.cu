// pss_kern_regs.cu -- the register passes of FP32 2D and 3D systems.
#include <type_traits>

#include "pss_regs.cuh"

namespace pss {
cudaError_t launch_col3(const ColArgs<float> &a, int nslots, cudaStream_t st) {
    switch (a.sp.n_inner) {
        case 16: return launch_col3_n<16>(a, nslots, st);
        case 32: return launch_col3_n<32>(a, nslots, st);
        case 64: return launch_col3_n<64>(a, nslots, st);
        case 128: return launch_col3_n<128>(a, nslots, st);
        case 256: return launch_col3_n<256>(a, nslots, st);
        case 512: return launch_col3_n<512>(a, nslots, st);
        case 1024: return launch_col3_n<1024>(a, nslots, st);
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_mid3(const MidArgs<float> &a, int nslots, int ntiles, cudaStream_t st) {
    switch (a.sp.ny) {
        case 16: return launch_mid3_n<16>(a, nslots, ntiles, st);
        case 32: return launch_mid3_n<32>(a, nslots, ntiles, st);
        case 64: return launch_mid3_n<64>(a, nslots, ntiles, st);
        case 128: return launch_mid3_n<128>(a, nslots, ntiles, st);
        case 256: return launch_mid3_n<256>(a, nslots, ntiles, st);
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_row3(const RowArgs<float> &a, int nslots, cudaStream_t st) {
    switch (a.sp.nx) {
        case 16: return launch_row3_n<16>(a, nslots, st);
        case 32: return launch_row3_n<32>(a, nslots, st);
        case 64: return launch_row3_n<64>(a, nslots, st);
        case 128: return launch_row3_n<128>(a, nslots, st);
        case 256: return launch_row3_n<256>(a, nslots, st);
        case 512: return launch_row3_n<512>(a, nslots, st);
        case 1024: return launch_row3_n<1024>(a, nslots, st);
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_terms3(const TermArgs &a, int batch, cudaStream_t st) {
    switch (a.sp.nx) {
        case 16: return launch_terms3_n<16>(a, batch, st);
        case 32: return launch_terms3_n<32>(a, batch, st);
        case 64: return launch_terms3_n<64>(a, batch, st);
        case 128: return launch_terms3_n<128>(a, batch, st);
        case 256: return launch_terms3_n<256>(a, batch, st);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace pss
