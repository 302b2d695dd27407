// FFT passes of H' x in native FP64 (complex128 blocks).
#include "hx_fft.cuh"

namespace dks {

unsigned debug_take_fft64() { return debug_take_unit(); }
template int fft_local<double2, double2>(dks_ctx*, const KPoint&, const double2*, double2*, int, int, double2*, void*, double, double,
                   cudaStream_t);

}  // namespace dks
