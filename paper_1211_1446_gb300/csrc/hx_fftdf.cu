// FFT passes of H' x in double-float (complex128 blocks, emulated FP64): the driver, the stick-inverse
// and the plane kernels without merged radices.  The other kernels are instantiated in
// hx_fftdf_plane.cu, hx_fftdf_bare.cu and hx_fftdf_fwd.cu: the double-float butterflies take the compiler a minute
// per group.
#include "hx_fft.cuh"

namespace dks {

extern template int launch_plane<cdp, true>(dks_ctx*, const KPoint&, const ExecPlan&, const ExecPlan&, const ctw*, const ctw*,
                                       const dfl*, cdp*, cdp*, int, cudaStream_t);
extern template int launch_plane_bare<cdp>(dks_ctx*, const KPoint&, const ExecPlan&, const ExecPlan&, const ctw*, const ctw*,
                                       const dfl*, cdp*, int, cudaStream_t);
extern template int launch_stick_forward<double2, cdp, false>(dks_ctx*, const KPoint&, const ExecPlan&, const ctw*, const cdp*,
                                                        const double2*, double2*, int, double, double, cudaStream_t);
extern template int launch_stick_forward<double2, cdp, true>(dks_ctx*, const KPoint&, const ExecPlan&, const ctw*, const cdp*,
                                                        const double2*, double2*, int, double, double, cudaStream_t);
unsigned debug_take_fftdf_plane();
unsigned debug_take_fftdf_bare();
unsigned debug_take_fftdf_fwd();
unsigned debug_take_fftdf() {
  unsigned first = 0u;
  for (unsigned v : {debug_take_unit(), debug_take_fftdf_plane(), debug_take_fftdf_bare(), debug_take_fftdf_fwd()})
    if (!first) first = v;
  return first;
}
template int fft_local<double2, cdp>(dks_ctx*, const KPoint&, const double2*, double2*, int, int, cdp*, void*, double, double,
                   cudaStream_t);

}  // namespace dks
