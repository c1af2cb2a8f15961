// pss_kern_terms_f32.cu -- the row kernel of product terms (FP32, 1D and 2D).
#include "pss_terms.cuh"

namespace pss {
cudaError_t launch_terms(const TermArgs &a, int batch, cudaStream_t st) {
    switch (a.sp.nx) {
        case 4: return launch_terms_n<4>(a, batch, st);
        case 8: return launch_terms_n<8>(a, batch, st);
        case 16: return launch_terms_n<16>(a, batch, st);
        case 32: return launch_terms_n<32>(a, batch, st);
        case 64: return launch_terms_n<64>(a, batch, st);
        case 128: return launch_terms_n<128>(a, batch, st);
        case 256: return launch_terms_n<256>(a, batch, st);
        case 512: return launch_terms_n<512>(a, batch, st);
        case 1024: return launch_terms_n<1024>(a, batch, st);
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace pss
