// Double-float stick-forward kernels of H' x (see hx_fftdf.cu).
#include "hx_fft.cuh"

namespace dks {

unsigned debug_take_fftdf_fwd() { return debug_take_unit(); }
template int launch_stick_forward<double2, cdp, false>(dks_ctx*, const KPoint&, const ExecPlan&, const ctw*, const cdp*,
                                                        const double2*, double2*, int, double, double, cudaStream_t);
template int launch_stick_forward<double2, cdp, true>(dks_ctx*, const KPoint&, const ExecPlan&, const ctw*, const cdp*,
                                                        const double2*, double2*, int, double, double, cudaStream_t);

}  // namespace dks
