// The x passes of the fluid step's spectral solves, the FP32 pressure solve in 64-bit block fixed point.
#include "fluid_fft.cuh"

namespace gbib {

template <>
cudaError_t fft_x<Fx64On32>(int mode, const FftGrid<Fx64On32> &g, int ncomp, const Fx64On32::Real *src, Spectrum<Fx64On32> sp, Fx64On32::Real *dst,
                        Fx64On32::Real *old, int *maxold, cudaStream_t s) {
    switch (g.log2n[0]) {
        case 4: return launch_x<Fx64On32, 4>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 5: return launch_x<Fx64On32, 5>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 6: return launch_x<Fx64On32, 6>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 7: return launch_x<Fx64On32, 7>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 8: return launch_x<Fx64On32, 8>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 9: return launch_x<Fx64On32, 9>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        default: return launch_x<Fx64On32, 10>(mode, g, ncomp, src, sp, dst, old, maxold, s);
    }
}

}  // namespace gbib
