// Double-float plane kernel of H' x with its twiddles in global memory (see hx_fftdf.cu).
#include "hx_fft.cuh"

namespace dks {

unsigned debug_take_fftdf_bare() { return debug_take_unit(); }
template int launch_plane_bare<cdp>(dks_ctx*, const KPoint&, const ExecPlan&, const ExecPlan&, const ctw*, const ctw*,
                                       const dfl*, cdp*, int, cudaStream_t);

}  // namespace dks
