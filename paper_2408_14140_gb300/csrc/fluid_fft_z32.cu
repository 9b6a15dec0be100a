// The z passes of the fluid step's spectral solves, FP32 fields.
#include "fluid_fft.cuh"

namespace gbib {

template <>
cudaError_t fft_z<Fp32>(const FftGrid<Fp32> &g, int ncomp, Spectrum<Fp32> sp, const SymbolArgs &sy, cudaStream_t s) {
    switch (g.log2n[2]) {
        case 4: return launch_z<Fp32, 4>(g, ncomp, sp, sy, s);
        case 5: return launch_z<Fp32, 5>(g, ncomp, sp, sy, s);
        case 6: return launch_z<Fp32, 6>(g, ncomp, sp, sy, s);
        case 7: return launch_z<Fp32, 7>(g, ncomp, sp, sy, s);
        case 8: return launch_z<Fp32, 8>(g, ncomp, sp, sy, s);
        case 9: return launch_z<Fp32, 9>(g, ncomp, sp, sy, s);
        default: return launch_z<Fp32, 10>(g, ncomp, sp, sy, s);
    }
}

}  // namespace gbib
