// The x passes of the fluid step's spectral solves, FP64 fields (64-bit block fixed point).
#include "fluid_fft.cuh"

namespace gbib {

template <>
cudaError_t fft_x<Fx64>(int mode, const FftGrid<Fx64> &g, int ncomp, const Fx64::Real *src, Spectrum<Fx64> sp, Fx64::Real *dst,
                        Fx64::Real *old, int *maxold, cudaStream_t s) {
    switch (g.log2n[0]) {
        case 4: return launch_x<Fx64, 4>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 5: return launch_x<Fx64, 5>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 6: return launch_x<Fx64, 6>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 7: return launch_x<Fx64, 7>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 8: return launch_x<Fx64, 8>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 9: return launch_x<Fx64, 9>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        default: return launch_x<Fx64, 10>(mode, g, ncomp, src, sp, dst, old, maxold, s);
    }
}

}  // namespace gbib
