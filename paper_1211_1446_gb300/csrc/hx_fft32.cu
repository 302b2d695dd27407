// FFT passes of H' x in FP32 (complex64 blocks).
#include "hx_fft.cuh"

namespace dks {

unsigned debug_take_fft32() { return debug_take_unit(); }
template int fft_local<float2, float2>(dks_ctx*, const KPoint&, const float2*, float2*, int, int, float2*, void*, double, double,
                   cudaStream_t);

}  // namespace dks
