// The z passes of the fluid step's spectral solves, FP64 fields (64-bit block fixed point).
#include "fluid_fft.cuh"

namespace gbib {

template <>
cudaError_t fft_z<Fx64>(const FftGrid<Fx64> &g, int ncomp, Spectrum<Fx64> sp, const SymbolArgs &sy, cudaStream_t s) {
    switch (g.log2n[2]) {
        case 4: return launch_z<Fx64, 4>(g, ncomp, sp, sy, s);
        case 5: return launch_z<Fx64, 5>(g, ncomp, sp, sy, s);
        case 6: return launch_z<Fx64, 6>(g, ncomp, sp, sy, s);
        case 7: return launch_z<Fx64, 7>(g, ncomp, sp, sy, s);
        case 8: return launch_z<Fx64, 8>(g, ncomp, sp, sy, s);
        case 9: return launch_z<Fx64, 9>(g, ncomp, sp, sy, s);
        default: return launch_z<Fx64, 10>(g, ncomp, sp, sy, s);
    }
}

}  // namespace gbib
