// Radix plan 2: the per-axis spectral passes with the radices of plan 0, m* + i w* in one row.
#include "fft_kernels.cuh"

namespace sipf {

cudaError_t axis_dispatch_p2(int H, const SpecRun& run, int pass, int device, cudaStream_t s) {
    switch (H) {
        case 64: return axis_pass<64, 0, true>(run, pass, device, s);
        case 128: return axis_pass<128, 0, true>(run, pass, device, s);
        case 256: return axis_pass<256, 0, true>(run, pass, device, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sipf
