// Electron density (Eq. density) from the stick and plane passes of H' x, in native FP64.
#include "hx_fft.cuh"

namespace dks {

unsigned debug_take_density() { return debug_take_unit(); }

// density from the split plane: after B1, per (p3, column block) the inverse FFT along axis 1 of
// every field it owns and the weighted sum of |psi|^2, added into the DIF-ordered planes
template <bool BIG>
__global__ void __launch_bounds__(256) k_plane_cols_density(const double2* __restrict__ pbuf, ExecPlan e1, int ld,
                                                            int n2, int n3, const double2* __restrict__ tw1,
                                                            const double* __restrict__ wfield, int nf, int fper,
                                                            int cpb, int ls1, unsigned mcpb, unsigned mlast,
                                                            double* __restrict__ rho_perm) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n1 = e1.n;
  const int z = blockIdx.x, c0 = blockIdx.y * cpb, f0 = blockIdx.z * fper, f1 = min(nf, f0 + fper);
  const int ncl = min(cpb, n2 - c0);
  double2* cols = reinterpret_cast<double2*>(smem_raw);
  double2* tw = cols + (size_t)cpb * ls1;
  double* acc = reinterpret_cast<double*>(tw + e1.ntw);
  load_twiddles(tw, tw1, e1.ntw);
  const unsigned mc = ncl == cpb ? mcpb : mlast;
  for (int e = threadIdx.x; e < n1 * ncl; e += blockDim.x) acc[e] = 0.0;
  for (int f = f0; f < f1; ++f) {
    const double2* pl = pbuf + ((size_t)f * n3 + z) * (size_t)n1 * ld;
    for (int e = threadIdx.x; e < n1 * ncl; e += blockDim.x) {
      const int i = mdiv(e, mc), c = e - i * ncl;
      cols[c * ls1 + i] = pl[(size_t)i * ld + c0 + c];
    }
    __syncthreads();
    fft_axis<double2, BIG>(cols, Lines{nullptr, ls1, 1, ncl, mc}, e1, tw, false);
    const double w = wfield[f];
    for (int e = threadIdx.x; e < n1 * ncl; e += blockDim.x) {
      const int i = mdiv(e, mc), c = e - i * ncl;
      const double2 v = cols[c * ls1 + i];
      acc[e] = fma(w, fma(v.x, v.x, v.y * v.y), acc[e]);
    }
    __syncthreads();
  }
  double* out = rho_perm + (size_t)z * n1 * ld;
  for (int e = threadIdx.x; e < n1 * ncl; e += blockDim.x) {
    const int i = mdiv(e, mc), c = e - i * ncl;
    if (acc[e] != 0.0) atomicAdd(out + (size_t)i * ld + c0 + c, acc[e]);
  }
}

// ---------------------------------------------------------------------------
// electron density (Eq. density): pass A as above, then per plane the inverse 2D FFT of
// every field and the weighted sum of |psi|^2 over the fields, FP64 throughout.  The sum
// stays in shared memory across the fields a CTA owns; the planes are in the DIF-permuted
// order of the potential ([p3][p1*LD + p2]).  As in k_plane, axis 2 runs over the rows that hold
// a stick.
// ---------------------------------------------------------------------------
template <bool BIG>
__global__ void __launch_bounds__(512) k_plane_density(const double2* __restrict__ t, int nsticks,
                                                       const int* __restrict__ stick_plane,
                                                       const int* __restrict__ plane_rows, int nrows, unsigned mrows,
                                                       ExecPlan e1, ExecPlan e2, int ld, unsigned mcols, int n3,
                                                       const double2* __restrict__ tw1,
                                                       const double2* __restrict__ tw2,
                                                       const double* __restrict__ wfield, int nf, int fper,
                                                       double* __restrict__ rho_perm) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int np = e1.n * ld;
  double2* plane = reinterpret_cast<double2*>(smem_raw);
  double2* stw1 = plane + np;
  double2* stw2 = stw1 + e1.ntw;
  double* acc = reinterpret_cast<double*>(stw2 + e2.ntw);
  int* rows = reinterpret_cast<int*>(acc + np);
  load_twiddles(stw1, tw1, e1.ntw);
  load_twiddles(stw2, tw2, e2.ntw);
  for (int e = threadIdx.x; e < nrows; e += blockDim.x) rows[e] = plane_rows[e];
  const int z = blockIdx.x;
  const int f0 = blockIdx.y * fper, f1 = min(nf, f0 + fper);
  for (int e = threadIdx.x; e < np; e += blockDim.x) acc[e] = 0.0;
  for (int f = f0; f < f1; ++f) {
    for (int e = threadIdx.x; e < np; e += blockDim.x) plane[e] = double2{0.0, 0.0};
    __syncthreads();
    const double2* row = t + ((size_t)f * n3 + z) * nsticks;
    for (int s = threadIdx.x; s < nsticks; s += blockDim.x) {
      const int at = stick_plane[s];
      if (dks_ok(at >= 0 && at < np, kChkPlaneDensity | (s & 0xffffff))) stage_elem(plane + at, row + s);
    }
    stage_wait_all();
    __syncthreads();
    fft_axis<double2, BIG>(plane, Lines{rows, 0, 1, nrows, mrows}, e2, stw2, false);
    fft_axis<double2, BIG>(plane, Lines{nullptr, 1, ld, e2.n, mcols}, e1, stw1, false);
    const double w = wfield[f];
    for (int e = threadIdx.x; e < np; e += blockDim.x) {
      const double2 v = plane[e];
      acc[e] = fma(w, fma(v.x, v.x, v.y * v.y), acc[e]);
    }
    __syncthreads();
  }
  double* out = rho_perm + (size_t)z * np;
  for (int e = threadIdx.x; e < np; e += blockDim.x)
    if (acc[e] != 0.0) atomicAdd(out + e, acc[e]);
}

// rho[(i1 N2 + i2) N3 + i3] += scale * rho_perm[(p3[i3] N1 + p1[i1]) LD + p2[i2]]
__global__ void k_unpermute_add(const double* __restrict__ rho_perm, double* __restrict__ rho, int n1, int n2,
                                int n3, int ld, const int* __restrict__ p1, const int* __restrict__ p2,
                                const int* __restrict__ p3, double scale) {
  const size_t ng = (size_t)n1 * n2 * n3;
  for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < ng; n += (size_t)gridDim.x * blockDim.x) {
    const int i3 = (int)(n % n3);
    const size_t r = n / n3;
    const int i2 = (int)(r % n2), i1 = (int)(r / n2);
    const size_t at = ((size_t)p3[i3] * n1 + p1[i1]) * ld + p2[i2];
    if (dks_ok(at < (size_t)n3 * n1 * ld, kChkUnpermute | (unsigned)(n & 0xffffff))) rho[n] += scale * rho_perm[at];
  }
}

int density_accumulate(dks_ctx* ctx, int ik, const double2* x, int nb, const double* occ, double* rho,
                       cudaStream_t st) {
  if (nb <= 0) return DKS_OK;
  KPoint& kp = ctx->k[ik];
  Exec& ex = exec0(ctx);
  const int npw = kp.npw, nc = ctx->ncomp;
  const int n1 = ctx->grid[0], n2 = ctx->grid[1], n3 = ctx->grid[2], ld = ctx->plane_ld;
  const size_t field_elems = (size_t)kp.nsticks * n3;
  const size_t np = (size_t)n1 * ld;
  const ExecPlan &e1 = ctx->exec64[0], &e2 = ctx->exec64[1], &e3 = ctx->exec64[2];
  const size_t sm_b = np * (sizeof(double2) + sizeof(double)) + (e1.ntw + e2.ntw) * sizeof(double2) + n1 * sizeof(int);
  // one plane per CTA (the plane and its |psi|^2 sum in shared memory), or the split form: rows
  // by k_plane_rows_inv into the buffer P, then columns by k_plane_cols_density
  const bool split = ctx->plane_split || sm_b > 227 * 1024;
  const size_t plane_elems = split ? (size_t)n3 * np : 0;
  int chunk = (int)std::max<size_t>(1, ctx->chunk_budget / (nc * (field_elems + plane_elems) * sizeof(double2)));
  chunk = std::min(chunk, nb);
  const size_t perm_bytes = ((n3 * np * sizeof(double) + 255) / 256) * 256;
  const size_t w_bytes = ((nc * (size_t)nb * sizeof(double) + 255) / 256) * 256;
  const size_t t_bytes = ((nc * (size_t)chunk * field_elems * sizeof(double2) + 255) / 256) * 256;
  DKS_TRY(grow(ex.ws_h, perm_bytes + w_bytes + t_bytes + nc * (size_t)chunk * plane_elems * sizeof(double2)));
  double* rho_perm = reinterpret_cast<double*>(ex.ws_h.ptr);
  double* wf = reinterpret_cast<double*>(reinterpret_cast<char*>(ex.ws_h.ptr) + perm_bytes);
  double2* tbuf = reinterpret_cast<double2*>(reinterpret_cast<char*>(ex.ws_h.ptr) + perm_bytes + w_bytes);
  double2* pbuf = reinterpret_cast<double2*>(reinterpret_cast<char*>(ex.ws_h.ptr) + perm_bytes + w_bytes + t_bytes);
  const int ls1 = n1 | 1;
  const int rpb = lines_per_cta(n1, ld, sizeof(double2));
  const int cpb = lines_per_cta(n2, ls1, sizeof(double2), (size_t)n1 * sizeof(double));
  const size_t sm_r = (size_t)rpb * ld * sizeof(double2) + twiddle_bytes<double2>(e2.ntw);
  const size_t sm_cd = (size_t)cpb * (ls1 * sizeof(double2) + n1 * sizeof(double)) + e1.ntw * sizeof(double2);
  std::vector<double> wh((size_t)nc * nb);
  for (int b = 0; b < nb; ++b)
    for (int c = 0; c < nc; ++c) wh[(size_t)b * nc + c] = occ[b];
  DKS_CUDA_TRY(cudaMemcpyAsync(wf, wh.data(), wh.size() * sizeof(double), cudaMemcpyHostToDevice, st));
  DKS_CUDA_TRY(cudaMemsetAsync(rho_perm, 0, n3 * np * sizeof(double), st));
  const bool big = e1.big || e2.big;
  auto rows_inv = big ? k_plane_rows_inv<double2, true> : k_plane_rows_inv<double2, false>;
  auto cols_density = big ? k_plane_cols_density<true> : k_plane_cols_density<false>;
  auto plane_density = big ? k_plane_density<true> : k_plane_density<false>;
  if (split) {
    DKS_TRY(allow_smem((const void*)rows_inv));
    DKS_TRY(allow_smem((const void*)cols_density));
  } else {
    DKS_TRY(allow_smem((const void*)plane_density));
  }
  const int tb_plane = pick_plane_threads(e1, e2, kp.nrows, sm_b, 512);
  for (int b0 = 0; b0 < nb; b0 += chunk) {
    const int nbc = std::min(chunk, nb - b0);
    const int nf = nc * nbc;
    const double es = sizeof(double2), tb = (double)nf * field_elems * es;
    {
      Prof pr(P_STICK_INV, st, (double)nf * npw * es + tb, 5.0 * n3 * std::log2((double)n3) * kp.nsticks * nf);
      const double2* xb = x + (size_t)b0 * nc * npw;
      if (e3.big) DKS_TRY((launch_stick_inverse<double2, double2, true>(kp, e3, ctx->etw64[2], xb, tbuf, nf, st)));
      else DKS_TRY((launch_stick_inverse<double2, double2, false>(kp, e3, ctx->etw64[2], xb, tbuf, nf, st)));
    }
    {
      // split the fields of a plane over enough CTAs to fill the GPU twice; atomics combine them
      const int nsplit = std::max(1, std::min(nf, (2 * ctx->num_sms + n3 - 1) / n3));
      const int fper = (nf + nsplit - 1) / nsplit;
      const double nn = (double)n1 * n2;
      Prof pr(P_SCF, st, tb + 2.0 * n3 * np * sizeof(double), nf * n3 * (5.0 * nn * std::log2(nn) + 3.0 * nn));
      if (split) {
        pr.count(1);
        const dim3 g1(n3, nf, (n1 + rpb - 1) / rpb);
        rows_inv<<<g1, 256, sm_r, st>>>(tbuf, pbuf, kp.nsticks, kp.stick_plane, e2, ld, n1, n3, ctx->etw64[1], rpb,
                                        magic(rpb), magic(n1 - (n1 - 1) / rpb * rpb));
        const dim3 g2(n3, (n2 + cpb - 1) / cpb, (nf + fper - 1) / fper);
        cols_density<<<g2, 256, sm_cd, st>>>(pbuf, e1, ld, n2, n3, ctx->etw64[0], wf + (size_t)b0 * nc, nf, fper, cpb,
                                             ls1, magic(cpb), magic(n2 - (n2 - 1) / cpb * cpb), rho_perm);
      } else {
        dim3 gb(n3, (nf + fper - 1) / fper);
        plane_density<<<gb, tb_plane, sm_b, st>>>(tbuf, kp.nsticks, kp.stick_plane, kp.plane_rows, kp.nrows,
                                                  magic(kp.nrows), e1, e2, ld, magic(n2), n3, ctx->etw64[0],
                                                  ctx->etw64[1], wf + (size_t)b0 * nc, nf, fper, rho_perm);
      }
    }
  }
  {
    const size_t ng = (size_t)ctx->ng;
    Prof pr(P_SCF, st, 3.0 * ng * sizeof(double), 2.0 * ng);
    const int blocks = (int)std::min<size_t>((ng + 255) / 256, (size_t)ctx->num_sms * 8);
    k_unpermute_add<<<blocks, 256, 0, st>>>(rho_perm, rho, n1, n2, n3, ld, ctx->posd[0], ctx->posd[1], ctx->posd[2],
                                            1.0 / ctx->volume);
  }
  DKS_CUDA_TRY(cudaGetLastError());
  return DKS_OK;
}


}  // namespace dks
