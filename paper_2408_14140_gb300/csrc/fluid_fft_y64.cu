// The y passes of the fluid step's spectral solves, FP64 fields (64-bit block fixed point).
#include "fluid_fft.cuh"

namespace gbib {

template <>
cudaError_t fft_y<Fx64>(bool inverse, const FftGrid<Fx64> &g, int ncomp, Spectrum<Fx64> sp, cudaStream_t s) {
    switch (g.log2n[1]) {
        case 4: return launch_y<Fx64, 4>(inverse, g, ncomp, sp, s);
        case 5: return launch_y<Fx64, 5>(inverse, g, ncomp, sp, s);
        case 6: return launch_y<Fx64, 6>(inverse, g, ncomp, sp, s);
        case 7: return launch_y<Fx64, 7>(inverse, g, ncomp, sp, s);
        case 8: return launch_y<Fx64, 8>(inverse, g, ncomp, sp, s);
        case 9: return launch_y<Fx64, 9>(inverse, g, ncomp, sp, s);
        default: return launch_y<Fx64, 10>(inverse, g, ncomp, sp, s);
    }
}

}  // namespace gbib
