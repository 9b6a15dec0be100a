// The x passes of the fluid step's spectral solves, FP32 fields.
#include "fluid_fft.cuh"

namespace gbib {

template <>
cudaError_t fft_x<Fp32>(int mode, const FftGrid<Fp32> &g, int ncomp, const Fp32::Real *src, Spectrum<Fp32> sp, Fp32::Real *dst,
                        Fp32::Real *old, int *maxold, cudaStream_t s) {
    switch (g.log2n[0]) {
        case 4: return launch_x<Fp32, 4>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 5: return launch_x<Fp32, 5>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 6: return launch_x<Fp32, 6>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 7: return launch_x<Fp32, 7>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 8: return launch_x<Fp32, 8>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        case 9: return launch_x<Fp32, 9>(mode, g, ncomp, src, sp, dst, old, maxold, s);
        default: return launch_x<Fp32, 10>(mode, g, ncomp, src, sp, dst, old, maxold, s);
    }
}

}  // namespace gbib
