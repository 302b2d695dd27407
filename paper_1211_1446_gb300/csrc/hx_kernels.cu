// H' x for the shifted valence DKS operator (Eq. vDKS): the terms without a grid, the projector
// contractions around the FFT passes (hx_fft.cuh), and kinetic balance.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "dks_internal.h"
#include "dks_kernels.cuh"
#include "fft_device.cuh"

namespace dks {

template <typename Vg, typename Vs>
int fft_local(dks_ctx* ctx, const KPoint& kp, const Vg* x, Vg* out, int nb, int chunk, Vs* tbuf, void* pbufv,
              double shift, double scale, cudaStream_t st);
extern template int fft_local<float2, float2>(dks_ctx*, const KPoint&, const float2*, float2*, int, int, float2*, void*, double, double,
                   cudaStream_t);
extern template int fft_local<double2, double2>(dks_ctx*, const KPoint&, const double2*, double2*, int, int, double2*, void*, double, double,
                   cudaStream_t);
extern template int fft_local<double2, cdp>(dks_ctx*, const KPoint&, const double2*, double2*, int, int, cdp*, void*, double, double,
                   cudaStream_t);
unsigned debug_take_fft32();
unsigned debug_take_fft64();
unsigned debug_take_fftdf();
unsigned debug_take_density();

__device__ __forceinline__ void dirac4(const double2 xv[4], double qx, double qy, double qz, double c,
                                       double diag_small, double shift, double2 h[4]) {
  // [[0, c s.q], [c s.q, -2c^2]] x - shift x ;  s.q = [[qz, qx - i qy], [qx + i qy, -qz]]
  const double2 qm = {c * qx, -c * qy};   // c (qx - i qy)
  const double2 qp = {c * qx, c * qy};    // c (qx + i qy)
  const double cz = c * qz;
  double2 a = cmul(qm, xv[3]);
  h[0] = {cz * xv[2].x + a.x - shift * xv[0].x, cz * xv[2].y + a.y - shift * xv[0].y};
  a = cmul(qp, xv[2]);
  h[1] = {a.x - cz * xv[3].x - shift * xv[1].x, a.y - cz * xv[3].y - shift * xv[1].y};
  a = cmul(qm, xv[1]);
  h[2] = {cz * xv[0].x + a.x + (diag_small - shift) * xv[2].x,
          cz * xv[0].y + a.y + (diag_small - shift) * xv[2].y};
  a = cmul(qp, xv[0]);
  h[3] = {a.x - cz * xv[1].x + (diag_small - shift) * xv[3].x,
          a.y - cz * xv[1].y + (diag_small - shift) * xv[3].y};
}

// KSSO kinetic term alone (no local potential on the grid): fields of npw planewaves
template <typename V>
__global__ void k_kinetic_only(const V* __restrict__ x, V* __restrict__ out, int npw, int nfields,
                               const double* __restrict__ ek, double shift, double scale) {
  const size_t total = (size_t)nfields * npw;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int p = (int)(e % npw);
    const double k = scale * (ek[p] - shift);
    const double2 xv = to_d2(x[e]);
    out[e] = from_d2<V>({k * xv.x, k * xv.y});
  }
}

// Dirac term alone (no local potential on the grid)
template <typename V>
__global__ void k_dirac_only(const V* __restrict__ x, V* __restrict__ out, int npw, int nb,
                             const double* __restrict__ q, double c, double shift, double scale) {
  const size_t total = (size_t)nb * npw;
  const double diag_small = -2.0 * c * c;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t b = e / npw;
    const int p = (int)(e - b * npw);
    const size_t fo = b * 4 * npw;
    double2 xv[4], h[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) xv[a] = to_d2(x[fo + (size_t)a * npw + p]);
    dirac4(xv, q[3 * p], q[3 * p + 1], q[3 * p + 2], c, diag_small, shift, h);
#pragma unroll
    for (int a = 0; a < 4; ++a)
      out[fo + (size_t)a * npw + p] = from_d2<V>({scale * h[a].x, scale * h[a].y});
  }
}

// Eq. (RKB) in the planewave basis (p -> q = k+G, m = 1): small = (sigma.q) large / (2c).
// Complex128 data: FP64 arithmetic with q; complex64 data: FP32 arithmetic with the leading
// parts of c q (scaled by 1 / (2 c^2)).
__device__ __forceinline__ void kb_spinor(double qx, double qy, double qz, double2 u, double2 d, double2& s0,
                                          double2& s1) {
  s0 = double2{qz * u.x + qx * d.x + qy * d.y, qz * u.y + qx * d.y - qy * d.x};
  s1 = double2{qx * u.x - qy * u.y - qz * d.x, qx * u.y + qy * u.x - qz * d.y};
}
__device__ __forceinline__ void kb_spinor(float qx, float qy, float qz, float2 u, float2 d, float2& s0,
                                          float2& s1) {
  s0 = float2{qz * u.x + qx * d.x + qy * d.y, qz * u.y + qx * d.y - qy * d.x};
  s1 = float2{qx * u.x - qy * u.y - qz * d.x, qx * u.y + qy * u.x - qz * d.y};
}
__global__ void k_kinetic_balance64(double2* __restrict__ x, int npw, int nb, const double* __restrict__ q,
                                    double c) {
  const size_t total = (size_t)nb * npw;
  const double h = 0.5 / c;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const size_t b = e / npw;
    const int p = (int)(e - b * npw);
    double2* xb = x + b * 4 * npw + p;
    double2 s0, s1;
    kb_spinor(h * q[3 * p], h * q[3 * p + 1], h * q[3 * p + 2], xb[0], xb[npw], s0, s1);
    xb[2 * (size_t)npw] = s0;
    xb[3 * (size_t)npw] = s1;
  }
}
__global__ void k_kinetic_balance32(float2* __restrict__ x, int npw, int nb, const float* __restrict__ cq,
                                    float h) {
  const size_t total = (size_t)nb * npw;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const size_t b = e / npw;
    const int p = (int)(e - b * npw);
    float2* xb = x + b * 4 * npw + p;
    float2 s0, s1;
    kb_spinor(h * cq[6 * p], h * cq[6 * p + 2], h * cq[6 * p + 4], xb[0], xb[npw], s0, s1);
    xb[2 * (size_t)npw] = s0;
    xb[3 * (size_t)npw] = s1;
  }
}

template <typename V>
int apply_h(dks_ctx* ctx, Exec& ex, int ik, const V* x, V* out, int nb, double shift, double scale,
            cudaStream_t st) {
  if (nb <= 0) return DKS_OK;
  KPoint& kp = ctx->k[ik];
  const int npw = kp.npw;
  const bool fp64 = sizeof(V) == sizeof(double2);
  const int n3 = ctx->grid[2];
  const int nc = ctx->ncomp;
  const int ncol = nb * nc / 2;   // projector columns x~: two-spinors of 2 npw rows
  const size_t zp_elems = (size_t)ctx->nproj * ncol;
  const size_t field_elems = (size_t)kp.nsticks * n3;
  // split pass B: one N1 x LD plane per (field, p3) in the buffer P (the arithmetic type of the
  // transforms has the size of V: complex128 and double-float pairs are both 16 bytes)
  const size_t plane_elems = split_plane(ctx, sizeof(V)) ? (size_t)n3 * ctx->grid[0] * ctx->plane_ld : 0;
  // chunk of bands whose intermediates stay within the L2-resident budget
  int chunk = (int)std::max<size_t>(1, ctx->chunk_budget / (nc * (field_elems + plane_elems) * sizeof(V)));
  chunk = std::min(chunk, nb);
  const size_t zp_bytes = ((zp_elems * sizeof(double2) + 255) / 256) * 256;
  const size_t t_bytes = ctx->has_v ? ((nc * chunk * field_elems * sizeof(V) + 255) / 256) * 256 : 0;
  const size_t p_bytes = ctx->has_v ? nc * chunk * plane_elems * sizeof(V) : 0;
  DKS_TRY(grow(ex.ws_h, zp_bytes + t_bytes + p_bytes + 256));
  double2* zp = reinterpret_cast<double2*>(ex.ws_h.ptr);
  V* tbuf = reinterpret_cast<V*>(reinterpret_cast<char*>(ex.ws_h.ptr) + zp_bytes);
  void* pbuf = p_bytes ? reinterpret_cast<char*>(ex.ws_h.ptr) + zp_bytes + t_bytes : nullptr;
  const V* bt = nullptr;
  // refinement phase with DKS_TC_FP64: both projector contractions from exact integer slices of
  // x~ (made here) and of the projector table (made once per k-point)
  const bool ozp = fp64 && ex.df_gemm && ctx->nproj && tc_enabled(TC_FP64) && projector_slices(ctx, ik, st);
  OzBlock bto;
  if (ozp) DKS_TRY(oz_layout(kp.btoz, 2 * npw, ctx->nproj, &bto));
  if (ctx->nproj) {
    bt = fp64 ? reinterpret_cast<const V*>(kp.bt64) : reinterpret_cast<const V*>(kp.bt32);
    DKS_CUDA_TRY(cudaMemsetAsync(zp, 0, zp_elems * sizeof(double2), st));
    // Z = B^H x~ : (nproj x 2npw) (2npw x 2nb)
    if (ozp) {
      // x~ (2 npw x ncol) as the A operand, the table as B: Z = (x~^H B)^H
      DKS_TRY(grow(ex.ws_oz, oz_bytes(2 * npw, ncol)));
      OzBlock xo;
      DKS_TRY(oz_layout(ex.ws_oz.ptr, 2 * npw, ncol, &xo));
      DKS_TRY(oz_split((const double2*)x, 2 * npw, ncol, xo, st));
      DKS_TRY(oz_gemm_hn(xo, ncol, bto, ctx->nproj, zp, ctx->nproj, true, st, P_PROJ_HN));
    } else if (fp64 && ex.df_gemm)
      DKS_TRY(gemm_hn_df(kp.btdf, 2 * npw, (const double2*)x, 2 * npw, 2 * npw, ctx->nproj, ncol, zp, st,
                         P_PROJ_HN));
    else
      DKS_TRY(gemm_hn<V>(bt, 2 * npw, x, 2 * npw, 2 * npw, ctx->nproj, ncol, zp, st, P_PROJ_HN, 0, false,
                         ctx->tc_proj));
  }
  if (ctx->has_v) {
    bool done = false;
    if constexpr (std::is_same<V, double2>::value) {
      if (ex.df_gemm) {
        DKS_TRY((fft_local<double2, cdp>(ctx, kp, x, out, nb, chunk, reinterpret_cast<cdp*>(tbuf), pbuf, shift, scale, st)));
        done = true;
      }
    }
    if (!done) DKS_TRY((fft_local<V, V>(ctx, kp, x, out, nb, chunk, tbuf, pbuf, shift, scale, st)));
  } else if (nc == 4) {
    const int blocks = std::max(1, std::min(ctx->num_sms * 8, (int)(((size_t)nb * npw + 255) / 256)));
    Prof pr(P_DIRAC + (fp64 ? 0 : kProf32), st, 8.0 * nb * npw * sizeof(V) + 24.0 * npw, 64.0 * nb * npw);
    k_dirac_only<V><<<blocks, 256, 0, st>>>(x, out, npw, nb, kp.q, ctx->c, shift, scale);
  } else {
    const int blocks = std::max(1, std::min(ctx->num_sms * 8, (int)(((size_t)2 * nb * npw + 255) / 256)));
    Prof pr(P_DIRAC + (fp64 ? 0 : kProf32), st, 4.0 * nb * npw * sizeof(V) + 8.0 * npw, 8.0 * nb * npw);
    k_kinetic_only<V><<<blocks, 256, 0, st>>>(x, out, npw, 2 * nb, kp.ek, shift, scale);
  }
  DKS_CUDA_TRY(cudaGetLastError());
  if (ctx->nproj) {
    // out~ += B (scale D Z)
    if (ozp)
      DKS_TRY(oz_rotate(bto, 0, ctx->nproj, zp, ctx->nproj, ncol, (double2*)out, 2 * npw, 1.0, st, scale,
                        ctx->dvec_dev, P_PROJ_NN));
    else if (fp64 && ex.df_gemm)
      DKS_TRY(gemm_nn_df(kp.btdf, 2 * npw, 2 * npw, ctx->nproj, zp, ctx->nproj, ctx->dvec_dev, ncol,
                         (double2*)out, 2 * npw, 1.0, st, scale, P_PROJ_NN));
    else
      DKS_TRY(gemm_nn<V>(bt, 2 * npw, 2 * npw, ctx->nproj, zp, ctx->nproj, ctx->dvec_dev, ncol, out, 2 * npw,
                         1.0, st, scale, P_PROJ_NN, ctx->tc_proj));
  }
  return DKS_OK;
}

// the first failed index check of the FFT kernels since the last call, then cleared (debug build; 0 in
// the product build)
unsigned debug_check_take() {
  unsigned first = 0u;
  for (unsigned v : {debug_take_fft32(), debug_take_fft64(), debug_take_fftdf(), debug_take_density()})
    if (!first) first = v;
  return first;
}

int kinetic_balance(dks_ctx* ctx, int ik, void* x, int nb, bool fp64, cudaStream_t st) {
  const KPoint& kp = ctx->k[ik];
  const size_t total = (size_t)nb * kp.npw;
  if (!total) return DKS_OK;
  const int blocks = (int)std::min<size_t>((total + 255) / 256, (size_t)ctx->num_sms * 8);
  Prof pr(P_MISC, st, 2.0 * total * 2 * (fp64 ? 16.0 : 8.0) + 24.0 * kp.npw, 16.0 * total);
  if (fp64)
    k_kinetic_balance64<<<blocks, 256, 0, st>>>((double2*)x, kp.npw, nb, kp.q, ctx->c);
  else
    k_kinetic_balance32<<<blocks, 256, 0, st>>>((float2*)x, kp.npw, nb, kp.cq32, (float)(0.5 / (ctx->c * ctx->c)));
  DKS_CUDA_TRY(cudaGetLastError());
  return DKS_OK;
}

template int apply_h<double2>(dks_ctx*, Exec&, int, const double2*, double2*, int, double, double, cudaStream_t);
template int apply_h<float2>(dks_ctx*, Exec&, int, const float2*, float2*, int, double, double, cudaStream_t);

}  // namespace dks
