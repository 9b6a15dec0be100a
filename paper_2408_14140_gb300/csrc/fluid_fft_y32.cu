// The y passes of the fluid step's spectral solves, FP32 fields.
#include "fluid_fft.cuh"

namespace gbib {

template <>
cudaError_t fft_y<Fp32>(bool inverse, const FftGrid<Fp32> &g, int ncomp, Spectrum<Fp32> sp, cudaStream_t s) {
    switch (g.log2n[1]) {
        case 4: return launch_y<Fp32, 4>(inverse, g, ncomp, sp, s);
        case 5: return launch_y<Fp32, 5>(inverse, g, ncomp, sp, s);
        case 6: return launch_y<Fp32, 6>(inverse, g, ncomp, sp, s);
        case 7: return launch_y<Fp32, 7>(inverse, g, ncomp, sp, s);
        case 8: return launch_y<Fp32, 8>(inverse, g, ncomp, sp, s);
        case 9: return launch_y<Fp32, 9>(inverse, g, ncomp, sp, s);
        default: return launch_y<Fp32, 10>(inverse, g, ncomp, sp, s);
    }
}

}  // namespace gbib
