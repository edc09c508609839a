// Inverse transforms of 512 samples.
#include "fft_inv.cuh"

namespace mdc {
template bool irfft4_launch<32, 16>(mdc_plan*, const IrfftArgs&, cudaStream_t);
}  // namespace mdc
