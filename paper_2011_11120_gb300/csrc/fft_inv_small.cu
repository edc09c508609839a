// Inverse transforms of 64, 128 and 256 samples.
#include "fft_inv.cuh"

namespace mdc {
template bool irfft4_launch<8, 8>(mdc_plan*, const IrfftArgs&, cudaStream_t);
template bool irfft4_launch<16, 8>(mdc_plan*, const IrfftArgs&, cudaStream_t);
template bool irfft4_launch<16, 16>(mdc_plan*, const IrfftArgs&, cudaStream_t);
}  // namespace mdc
