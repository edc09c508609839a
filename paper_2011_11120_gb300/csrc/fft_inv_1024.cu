// Inverse transforms of 1024 samples.
#include "fft_inv.cuh"

namespace mdc {
template bool irfft4_launch<32, 32>(mdc_plan*, const IrfftArgs&, cudaStream_t);
}  // namespace mdc
