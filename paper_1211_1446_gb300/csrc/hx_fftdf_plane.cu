// Double-float plane kernels of H' x with merged radices (see hx_fftdf.cu).
#include "hx_fft.cuh"

namespace dks {

unsigned debug_take_fftdf_plane() { return debug_take_unit(); }
template int launch_plane<cdp, true>(dks_ctx*, const KPoint&, const ExecPlan&, const ExecPlan&, const ctw*, const ctw*,
                                       const dfl*, cdp*, cdp*, int, cudaStream_t);

}  // namespace dks
