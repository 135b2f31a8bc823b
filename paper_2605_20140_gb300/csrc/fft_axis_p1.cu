// Per-axis spectral passes (H > 128) with radix plan 1.
#include "fft_kernels.cuh"

namespace sipf {

cudaError_t axis_dispatch_p1(int H, const SpecRun& run, int pass, int device, cudaStream_t s) {
    switch (H) {
        case 144: return axis_pass<144, 1, false>(run, pass, device, s);
        case 192: return axis_pass<192, 1, false>(run, pass, device, s);
        case 216: return axis_pass<216, 1, false>(run, pass, device, s);
        case 256: return axis_pass<256, 1, false>(run, pass, device, s);
        case 288: return axis_pass<288, 1, false>(run, pass, device, s);
        case 384: return axis_pass<384, 1, false>(run, pass, device, s);
        case 432: return axis_pass<432, 1, false>(run, pass, device, s);
        case 512: return axis_pass<512, 1, false>(run, pass, device, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sipf
