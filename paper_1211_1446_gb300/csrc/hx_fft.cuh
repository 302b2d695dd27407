// H' x for the shifted valence DKS operator (Eq. vDKS, Sec. 3.1 "matrix-free Hx").
//
//   H' x = [[0, c s.q], [c s.q, -2c^2]] x          free Dirac term per planewave (Eq. 2)
//        + FFT^-1 . V(r) . FFT x                     local potential, one grid per component
//        + (I2 (x) B D B^H) x                         spin-orbit projectors (Eq. HGH)
//
// GPU layout.  x[band][comp][pw] with planewaves in canonical order, so each
// (m1, m2) "stick" along the third axis is a contiguous run of planewaves.  The
// 3D transform of one field (band, comp) runs in three passes that keep all
// intermediates in a stick-compressed buffer T[field][p3][stick] sized to stay
// resident in the 129 MB L2:
//   pass A  the stick's consecutive planewaves, and zeros, into a length-N3 line in shared memory,
//           inverse FFT along axis 3 (DIF, natural in -> digit-reversed out) whose last pass stores to T
//   pass B  one (field, plane) per CTA: scatter the sticks into an N1 x N2 plane
//           in shared memory, inverse 2D FFT (DIF), multiply by V/Ng stored in
//           the same digit-reversed order, forward 2D FFT (DIT, digit-reversed in
//           -> natural out), gather the sticks back (in place in T, as swapped data: real and
//           imaginary part exchanged, see fft_device.cuh)
//   pass C  four components of one band per CTA: forward FFT along axis 3 (DIT),
//           gather to the sphere, add the Dirac 4x4 term computed in FP64 and the
//           optional filter shift, scale, store
// Pairing DIF for the inverse with DIT for the forward transform removes every
// digit-reversal permutation: the real-space planes simply live in permuted
// order, and V is uploaded in that order.
// The projector term is two tall-skinny contractions over 2*npw rows with
// x viewed as [2*nb][2*npw] (large and small two-spinors as separate columns).
//
// Kernels and launchers of the three passes, as templates over the storage and the arithmetic type;
// hx_fft32.cu, hx_fft64.cu, hx_fftdf*.cu and hx_density.cu instantiate them (separate translation
// units, compiled in parallel), hx_kernels.cu holds the rest of H' x.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <string>
#include <type_traits>

#include "dks_internal.h"
#include "dks_kernels.cuh"
#include "fft_device.cuh"

namespace dks {

// ---------------------------------------------------------------------------
// pass A: sphere -> stick lines, inverse FFT along axis 3
// ---------------------------------------------------------------------------
// twiddles follow the data in shared memory, 16-byte aligned (twiddle_bytes leaves room for that)
template <typename V>
__device__ __forceinline__ typename TwOf<V>::T* twiddle_space(V* end) {
  return reinterpret_cast<typename TwOf<V>::T*>((reinterpret_cast<uintptr_t>(end) + 15) & ~(uintptr_t)15);
}
// asynchronous copy of one element into shared memory (many loads in flight, no registers held)
template <typename V>
__device__ __forceinline__ void stage_elem(V* dst, const V* src) {
  if constexpr (sizeof(V) == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
// double2 -> cdp: copied as it is; the thread that copied an element converts it after its wait
__device__ __forceinline__ void stage_elem(cdp* dst, const double2* src) {
  stage_elem(reinterpret_cast<double2*>(dst), src);
}
__device__ __forceinline__ void stage_wait_all() { asm volatile("cp.async.wait_all;\n" ::); }

// The planewaves of a stick are consecutive frequencies (the sphere is convex), so the line of stick
// s holds x[start .. start + count) from position `first` on, modulo N3, and zeros elsewhere: one
// warp per line reads it with coalesced loads and no index tables.  T holds the arithmetic type V
// (cdp in the emulated-FP64 mode), so only x is converted; the last pass stores straight to T.
template <typename Vg, typename V, bool BIG>
__global__ void __launch_bounds__(256, sizeof(V) == sizeof(float2) ? 5 : 3) k_stick_inverse(
    const Vg* __restrict__ x, V* __restrict__ t, int npw, int nsticks, const int* __restrict__ stick_start,
    const int* __restrict__ stick_first, const __grid_constant__ ExecPlan e3,
    const typename TwOf<V>::T* __restrict__ tw3, int lspb, int ls, unsigned mlines) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int spb = 1 << lspb;
  V* line = reinterpret_cast<V*>(smem_raw);   // spb lines of stride ls (odd)
  auto* tw = twiddle_space<V>(line + spb * ls);
  const int n3 = e3.n;
  const int s0 = blockIdx.x * spb;
  const int ns = min(spb, nsticks - s0);
  const int f = blockIdx.y;
  load_twiddles(tw, tw3, e3.ntw);
  const Vg* xf = x + (size_t)f * npw;
  for (int s = threadIdx.x >> 5; s < ns; s += blockDim.x >> 5) {
    const int q = stick_start[s0 + s], count = stick_start[s0 + s + 1] - q, first = stick_first[s0 + s];
    for (int z = threadIdx.x & 31; z < n3; z += 32) {
      const int k = z - first + (z < first ? n3 : 0);
      V* dst = line + s * ls + z;
      if (k < count && dks_ok(k >= 0 && q + k < npw, kChkStickInverse | ((q + k) & 0xffffff))) stage_elem(dst, xf + q + k);
      else *dst = vzero<V>();
    }
  }
  stage_wait_all();
  if constexpr (!std::is_same<Vg, V>::value) {
    for (int s = threadIdx.x >> 5; s < ns; s += blockDim.x >> 5) {
      const int count = stick_start[s0 + s + 1] - stick_start[s0 + s], first = stick_first[s0 + s];
      for (int z = threadIdx.x & 31; z < n3; z += 32) {
        if (z - first + (z < first ? n3 : 0) >= count) continue;   // stays a zero pair
        V* dst = line + s * ls + z;
        *dst = cdp_split(*reinterpret_cast<const double2*>(dst));
      }
    }
  }
  __syncthreads();
  fft_axis_store<V, BIG>(line, Lines{nullptr, ls, 1, spb, mlines}, e3, tw,
                         StickBuf<V>{t + (size_t)f * n3 * nsticks + s0, nsticks, ns, lspb, 0});
}

// ---------------------------------------------------------------------------
// pass B: one plane of one field: 2D inverse FFT, x V/Ng, 2D forward FFT
// ---------------------------------------------------------------------------
// resident threads per SM of k_plane, i.e. the bound its registers are compiled for: 64 per thread
// for 8-byte elements, 80 with merged radices, 128 for 16-byte elements.  (60 x 60 x 216, 104
// columns: 64 / 80 / 128 registers 1.79 / 1.76 / 1.90 ms; double-float 48 x 48 x 56, 40 columns: 80 /
// 96 / 128 registers 0.683 / 0.682 / 0.662 ms.)
__host__ __device__ constexpr int plane_max_threads(size_t elem, bool big) {
  return elem == sizeof(float2) ? (big ? 768 : 1024) : 512;
}

// Per CTA: zero plane, sticks scattered into it (coalesced reads), then 2 (passes of axis 2) + 2
// (passes of axis 1) - 1 passes, the last inverse and the first forward pass of axis 1 and the
// product with V being one.  Axis 2 runs over the rows that hold a stick only (29 of 60 for a grid
// twice as fine as the sphere needs); the others are zero before and unused after.
// TWS: the twiddles and the row table in shared memory after the plane; planes that leave no room for
// them read both through L1, which beats the three-kernel form (4 columns, us: 160 x 180 x 12 complex64
// 191 against 342, 120 x 120 x 12 double-float 301 against 360; 16 columns on 120 x 120 x 216 24.1 against 29.3 ms).
template <typename V, bool BIG, bool TWS>
__global__ void __launch_bounds__(plane_max_threads(sizeof(V), BIG), 1)
    k_plane(V* __restrict__ t, int nsticks, const int* __restrict__ stick_plane, const int* __restrict__ plane_rows,
            int nrows, unsigned mrows, const __grid_constant__ ExecPlan e1,
            const __grid_constant__ ExecPlan e2, int ld, unsigned mcols, int n3, const typename TwOf<V>::T* __restrict__ tw1, const typename TwOf<V>::T* __restrict__ tw2,
            const typename RealOf<V>::T* __restrict__ vperm) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* plane = reinterpret_cast<V*>(smem_raw);   // n1 rows of stride ld (odd), position i1*ld + i2
  const int np = e1.n * ld;
  const typename TwOf<V>::T *ptw1 = tw1, *ptw2 = tw2;
  const int* rows = plane_rows;
  const int z = blockIdx.x, f = blockIdx.y;
  for (int e = threadIdx.x; e < np; e += blockDim.x) plane[e] = vzero<V>();
  if constexpr (TWS) {
    auto* stw1 = twiddle_space<V>(plane + np);
    auto* stw2 = stw1 + e1.ntw;
    int* srows = reinterpret_cast<int*>(stw2 + e2.ntw);
    load_twiddles(stw1, tw1, e1.ntw);
    load_twiddles(stw2, tw2, e2.ntw);
    for (int e = threadIdx.x; e < nrows; e += blockDim.x) srows[e] = plane_rows[e];
    ptw1 = stw1;
    ptw2 = stw2;
    rows = srows;
  }
  __syncthreads();
  V* row = t + ((size_t)f * n3 + z) * nsticks;
  for (int s = threadIdx.x; s < nsticks; s += blockDim.x) {
    const int at = stick_plane[s];
    if (dks_ok(at >= 0 && at < np, kChkPlane | (s & 0xffffff))) stage_elem(plane + at, row + s);
  }
  stage_wait_all();
  __syncthreads();
  const typename RealOf<V>::T* vz = vperm + (size_t)z * np;
  const int a = e2.nst, b = a + e1.nst, c = b + e1.nst - 1, steps = c + e2.nst;
#pragma unroll 1
  for (int i = 0; i < steps; ++i) {
    const bool ax2 = i < a || i >= c, dit = i >= b;
    const int k = i < a ? i : i < b ? i - a : i < c ? e1.nst - 2 - (i - b) : e2.nst - 1 - (i - c);
    const ExecPass& p = ax2 ? e2.p[k] : e1.p[k];
    const Lines ln{ax2 ? rows : nullptr, 1, ax2 ? 1 : ld, ax2 ? nrows : e2.n, ax2 ? mrows : mcols};
    fft_step<V, BIG>(plane, ln, p, ax2 ? e2.n : e1.n, (ax2 ? ptw2 : ptw1) + p.tw, dit, i == b - 1 ? vz : nullptr);
  }
  for (int s = threadIdx.x; s < nsticks; s += blockDim.x) {
    const int at = stick_plane[s];
    if (dks_ok(at >= 0 && at < np, kChkPlane | (s & 0xffffff))) row[s] = plane[at];
  }
}

// ---------------------------------------------------------------------------
// pass B split in three kernels, for planes too large for one CTA's shared memory (N1 LD
// sizeof(Vs) above the 227 KB limit, e.g. 120 x 121 complex128) or when chosen by the tuner.
// The plane of one (field, p3) goes through an L2-resident buffer P[field][p3][i1][LD] (rows in
// natural i1 order before the column transform, in DIF position order after it); every pass is the
// one of k_plane, so the results are the same bit for bit.
//   B1  rows r0 .. r0+nr-1: scatter their sticks, inverse FFT along axis 2     -> P
//   B2  columns c0 .. c0+nc-1 (DIF positions along axis 2): inverse FFT along axis 1,
//       x V/Ng, forward FFT along axis 1                                       -> P (swapped data)
//   B3  rows: forward FFT along axis 2, gather the sticks                      -> T
// ---------------------------------------------------------------------------
template <typename Vs, bool BIG>
__global__ void __launch_bounds__(256) k_plane_rows_inv(const Vs* __restrict__ t, Vs* __restrict__ pbuf, int nsticks,
                                                        const int* __restrict__ stick_plane, ExecPlan e2, int ld,
                                                        int n1, int n3, const typename TwOf<Vs>::T* __restrict__ tw2, int rpb,
                                                        unsigned mrpb, unsigned mlast) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Vs* rows = reinterpret_cast<Vs*>(smem_raw);   // rpb rows of stride ld
  auto* tw = twiddle_space<Vs>(rows + rpb * ld);
  load_twiddles(tw, tw2, e2.ntw);
  const int z = blockIdx.x, f = blockIdx.y, r0 = blockIdx.z * rpb;
  const int nr = min(rpb, n1 - r0);
  for (int e = threadIdx.x; e < nr * ld; e += blockDim.x) rows[e] = vzero<Vs>();
  __syncthreads();
  const Vs* src = t + ((size_t)f * n3 + z) * nsticks;
  const int lo = r0 * ld, hi = (r0 + nr) * ld;   // stick_plane = i1 LD + i2
  for (int s = threadIdx.x; s < nsticks; s += blockDim.x) {
    const int pos = stick_plane[s];
    if (pos >= lo && pos < hi) rows[pos - lo] = src[s];
  }
  __syncthreads();
  fft_axis<Vs, BIG>(rows, Lines{nullptr, ld, 1, nr, nr == rpb ? mrpb : mlast}, e2, tw, false);
  Vs* out = pbuf + (((size_t)f * n3 + z) * n1 + r0) * ld;
  for (int e = threadIdx.x; e < nr * ld; e += blockDim.x) out[e] = rows[e];
}

template <typename Vs, bool BIG>
__global__ void __launch_bounds__(256) k_plane_cols_v(Vs* __restrict__ pbuf, ExecPlan e1, int ld, int n2, int n3,
                                                      const typename TwOf<Vs>::T* __restrict__ tw1,
                                                      const typename RealOf<Vs>::T* __restrict__ vperm, int cpb,
                                                      int ls1, unsigned mcpb, unsigned mlast) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Vs* cols = reinterpret_cast<Vs*>(smem_raw);   // cpb lines of stride ls1 (odd), element i1
  const int n1 = e1.n;
  auto* tw = twiddle_space<Vs>(cols + cpb * ls1);
  load_twiddles(tw, tw1, e1.ntw);
  const int z = blockIdx.x, f = blockIdx.y, c0 = blockIdx.z * cpb;
  const int ncl = min(cpb, n2 - c0);
  Vs* pl = pbuf + ((size_t)f * n3 + z) * (size_t)n1 * ld;
  const unsigned mc = ncl == cpb ? mcpb : mlast;
  for (int e = threadIdx.x; e < n1 * ncl; e += blockDim.x) {
    const int i = mdiv(e, mc), c = e - i * ncl;
    cols[c * ls1 + i] = pl[(size_t)i * ld + c0 + c];
  }
  __syncthreads();
  const Lines ln{nullptr, ls1, 1, ncl, mc};
  fft_axis<Vs, BIG>(cols, ln, e1, tw, false);
  const typename RealOf<Vs>::T* vz = vperm + (size_t)z * n1 * ld;
  for (int e = threadIdx.x; e < n1 * ncl; e += blockDim.x) {
    const int i = mdiv(e, mc), c = e - i * ncl;
    cols[c * ls1 + i] = cswap(cscale(cols[c * ls1 + i], vz[(size_t)i * ld + c0 + c]));
  }
  __syncthreads();
  fft_axis<Vs, BIG>(cols, ln, e1, tw, true);
  for (int e = threadIdx.x; e < n1 * ncl; e += blockDim.x) {
    const int i = mdiv(e, mc), c = e - i * ncl;
    pl[(size_t)i * ld + c0 + c] = cols[c * ls1 + i];
  }
}

template <typename Vs, bool BIG>
__global__ void __launch_bounds__(256) k_plane_rows_fwd(Vs* __restrict__ t, const Vs* __restrict__ pbuf, int nsticks,
                                                        const int* __restrict__ stick_plane, ExecPlan e2, int ld,
                                                        int n1, int n3, const typename TwOf<Vs>::T* __restrict__ tw2, int rpb,
                                                        unsigned mrpb, unsigned mlast) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Vs* rows = reinterpret_cast<Vs*>(smem_raw);
  auto* tw = twiddle_space<Vs>(rows + rpb * ld);
  load_twiddles(tw, tw2, e2.ntw);
  const int z = blockIdx.x, f = blockIdx.y, r0 = blockIdx.z * rpb;
  const int nr = min(rpb, n1 - r0);
  const Vs* in = pbuf + (((size_t)f * n3 + z) * n1 + r0) * ld;
  for (int e = threadIdx.x; e < nr * ld; e += blockDim.x) rows[e] = in[e];
  __syncthreads();
  fft_axis<Vs, BIG>(rows, Lines{nullptr, ld, 1, nr, nr == rpb ? mrpb : mlast}, e2, tw, true);
  Vs* dst = t + ((size_t)f * n3 + z) * nsticks;
  const int lo = r0 * ld, hi = (r0 + nr) * ld;
  for (int s = threadIdx.x; s < nsticks; s += blockDim.x) {
    const int pos = stick_plane[s];
    if (pos >= lo && pos < hi) dst[s] = rows[pos - lo];
  }
}

// ---------------------------------------------------------------------------
// pass C: forward FFT along axis 3, gather, Dirac term (FP64), shift, scale
// ---------------------------------------------------------------------------
// (hu, hd) += (c s.q) (u, d), c q = (cx, cy, cz)
__device__ __forceinline__ void sq_acc(double cx, double cy, double cz, double2 u, double2 d, double2& hu,
                                       double2& hd) {
  hu.x = fma(cy, d.y, fma(cx, d.x, fma(cz, u.x, hu.x)));
  hu.y = fma(-cy, d.x, fma(cx, d.y, fma(cz, u.y, hu.y)));
  hd.x = fma(-cz, d.x, fma(-cy, u.y, fma(cx, u.x, hd.x)));
  hd.y = fma(-cz, d.y, fma(cy, u.x, fma(cx, u.y, hd.y)));
}

// sum_k c_k x_k for four double-float constants c_k = (h, l) and FP32 values x_k: exact FP32
// products with their rounding errors, two-sum of the leading parts; result as (hi, lo)
__device__ __forceinline__ dfl dsum4(float c1h, float c1l, float x1, float c2h, float c2l, float x2, float c3h,
                                     float c3l, float x3, float c4h, float c4l, float x4) {
  float s = c1h * x1;
  float r = fmaf(c1l, x1, fmaf(c1h, x1, -s));
  auto add = [&](float ch, float cl, float x) {
    const float p = ch * x;
    const float e = fmaf(cl, x, fmaf(ch, x, -p));
    const float t = s + p;
    const float bb = t - s;
    r += ((s - (t - bb)) + (p - bb)) + e;
    s = t;
  };
  add(c2h, c2l, x2);
  add(c3h, c3l, x3);
  add(c4h, c4l, x4);
  return dfl{s, r};
}

// The lines of NC components of one band: forward FFT along axis 3 from T (swapped data after pass B)
// into shared memory; line_val reads an element of the result
template <typename V> __device__ __forceinline__ V line_val(const V* line, int at) { return cswap(line[at]); }
template <typename V, bool BIG, int NC>
__device__ __forceinline__ void stick_lines_forward(const V* __restrict__ t, V* line, int nsticks, int s0, int ns,
                                                    int lspb, int ls, unsigned mlines, const ExecPlan& e3,
                                                    const typename TwOf<V>::T* __restrict__ tw3) {
  auto* tw = twiddle_space<V>(line + ((NC * ls) << lspb));
  load_twiddles(tw, tw3, e3.ntw);   // the first DIT pass has none; the barrier after it publishes them
  fft_axis_load<V, BIG>(line, Lines{nullptr, ls, 1, NC << lspb, mlines}, e3, tw,
                        StickBuf<V>{const_cast<V*>(t) + s0, nsticks, ns, lspb, (size_t)e3.n * nsticks});
}

template <typename Vg, typename V, bool BIG>
__global__ void __launch_bounds__(256) k_stick_forward(
    const V* __restrict__ t, const Vg* __restrict__ x, Vg* __restrict__ out, int npw, int nsticks,
    const int* __restrict__ stick_start, const int* __restrict__ pw_at, const __grid_constant__ ExecPlan e3,
    const typename TwOf<V>::T* __restrict__ tw3, const double* __restrict__ cq64, const float* __restrict__ cq32,
    double c, double shift, double scale, int lspb, int ls, unsigned mlines) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* line = reinterpret_cast<V*>(smem_raw);   // 4*spb lines of stride ls (odd)
  const int spb = 1 << lspb;
  const int s0 = blockIdx.x * spb;
  const int ns = min(spb, nsticks - s0);
  const int b = blockIdx.y, n3 = e3.n;
  stick_lines_forward<V, BIG, 4>(t + (size_t)b * 4 * n3 * nsticks, line, nsticks, s0, ns, lspb, ls, mlines, e3, tw3);
  const size_t fo = (size_t)b * 4 * npw;
  const int q0 = stick_start[s0], q1 = stick_start[s0 + ns];
  if constexpr (std::is_same<Vg, float2>::value && std::is_same<V, float2>::value) {
    // FP32 blocks: the large components in FP32; the small components, where c s.q x_L and
    // (2c^2 + shift) x_S nearly cancel, as double-float sums of exact products
    const double kd = 2.0 * c * c + shift;
    const float kh = (float)kd, kl = (float)(kd - (double)kh), sh = (float)shift, sc = (float)scale;
    for (int p = q0 + threadIdx.x; p < q1; p += blockDim.x) {
      const int at = pw_at[p], s = (at >> 8) - s0, iz = at & 255;
      if (!dks_ok(s >= 0 && s < ns && iz >= 0 && iz < n3, kChkStickForward | (p & 0xffffff))) continue;
      const float2 x0 = x[fo + p], x1 = x[fo + (size_t)npw + p], x2 = x[fo + 2 * (size_t)npw + p],
                   x3 = x[fo + 3 * (size_t)npw + p];
      const float* cq = cq32 + 6 * (size_t)p;
      const float cxh = cq[0], cxl = cq[1], cyh = cq[2], cyl = cq[3], czh = cq[4], czl = cq[5];
      float2 h[4];
      h[0] = float2{czh * x2.x + cxh * x3.x + cyh * x3.y - sh * x0.x, czh * x2.y + cxh * x3.y - cyh * x3.x - sh * x0.y};
      h[1] = float2{cxh * x2.x - cyh * x2.y - czh * x3.x - sh * x1.x, cxh * x2.y + cyh * x2.x - czh * x3.y - sh * x1.y};
      const dfl h2r = dsum4(czh, czl, x0.x, cxh, cxl, x1.x, cyh, cyl, x1.y, -kh, -kl, x2.x);
      const dfl h2i = dsum4(czh, czl, x0.y, cxh, cxl, x1.y, -cyh, -cyl, x1.x, -kh, -kl, x2.y);
      const dfl h3r = dsum4(cxh, cxl, x0.x, -cyh, -cyl, x0.y, -czh, -czl, x1.x, -kh, -kl, x3.x);
      const dfl h3i = dsum4(cxh, cxl, x0.y, cyh, cyl, x0.x, -czh, -czl, x1.y, -kh, -kl, x3.y);
      const float2 l2 = line_val(line, (2 * spb + s) * ls + iz), l3 = line_val(line, (3 * spb + s) * ls + iz);
      h[2] = float2{h2r.h + (h2r.l + l2.x), h2i.h + (h2i.l + l2.y)};
      h[3] = float2{h3r.h + (h3r.l + l3.x), h3i.h + (h3i.l + l3.y)};
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const float2 loc = line_val(line, (a * spb + s) * ls + iz);
        h[a] = float2{h[a].x + loc.x, h[a].y + loc.y};
      }
#pragma unroll
      for (int a = 0; a < 4; ++a) out[fo + (size_t)a * npw + p] = float2{sc * h[a].x, sc * h[a].y};
    }
    return;
  }
  // FP64: the local term starts each sum, then c s.q and the diagonal as fused multiply-adds (28 of
  // them per planewave and band for a plain H'; the FP64 unit is what this epilogue waits for)
  const double kl = -shift, ks = -2.0 * c * c - shift;
  for (int p = q0 + threadIdx.x; p < q1; p += blockDim.x) {
    const int at = pw_at[p], s = (at >> 8) - s0, iz = at & 255;
    if (!dks_ok(s >= 0 && s < ns && iz >= 0 && iz < n3, kChkStickForward | (p & 0xffffff))) continue;
    double2 xv[4], h[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      xv[a] = to_d2(x[fo + (size_t)a * npw + p]);
      h[a] = to_d2(line_val(line, (a * spb + s) * ls + iz));
    }
    const double cx = cq64[3 * (size_t)p], cy = cq64[3 * (size_t)p + 1], cz = cq64[3 * (size_t)p + 2];
    sq_acc(cx, cy, cz, xv[2], xv[3], h[0], h[1]);
    sq_acc(cx, cy, cz, xv[0], xv[1], h[2], h[3]);
#pragma unroll
    for (int a = 2; a < 4; ++a) h[a] = double2{fma(ks, xv[a].x, h[a].x), fma(ks, xv[a].y, h[a].y)};
    if (shift != 0.0) {
#pragma unroll
      for (int a = 0; a < 2; ++a) h[a] = double2{fma(kl, xv[a].x, h[a].x), fma(kl, xv[a].y, h[a].y)};
    }
    if (scale != 1.0) {
#pragma unroll
      for (int a = 0; a < 4; ++a) h[a] = double2{scale * h[a].x, scale * h[a].y};
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) out[fo + (size_t)a * npw + p] = from_d2<Vg>(h[a]);
  }
}

// KSSO two-spinors: forward z-transform of the V psi sticks of both components, gathered onto
// the sphere, plus the kinetic term: out = scale ((|k+G|^2/2 - shift) x + V psi)
template <typename Vg, typename V, bool BIG>
__global__ void __launch_bounds__(256) k_stick_forward_ks(
    const V* __restrict__ t, const Vg* __restrict__ x, Vg* __restrict__ out, int npw, int nsticks,
    const int* __restrict__ stick_start, const int* __restrict__ pw_at, const __grid_constant__ ExecPlan e3,
    const typename TwOf<V>::T* __restrict__ tw3, const double* __restrict__ ek, double shift, double scale, int lspb,
    int ls, unsigned mlines) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* line = reinterpret_cast<V*>(smem_raw);   // 2*spb lines of stride ls (odd)
  const int spb = 1 << lspb;
  const int s0 = blockIdx.x * spb;
  const int ns = min(spb, nsticks - s0);
  const int b = blockIdx.y, n3 = e3.n;
  stick_lines_forward<V, BIG, 2>(t + (size_t)b * 2 * n3 * nsticks, line, nsticks, s0, ns, lspb, ls, mlines, e3, tw3);
  const size_t fo = (size_t)b * 2 * npw;
  const int q0 = stick_start[s0], q1 = stick_start[s0 + ns];
  for (int p = q0 + threadIdx.x; p < q1; p += blockDim.x) {
    const int at = pw_at[p], s = (at >> 8) - s0, iz = at & 255;
    if (!dks_ok(s >= 0 && s < ns && iz >= 0 && iz < n3, kChkStickForwardKs | (p & 0xffffff))) continue;
    if constexpr (std::is_same<Vg, float2>::value && std::is_same<V, float2>::value) {
      const float kin = (float)(ek[p] - shift), sc = (float)scale;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const float2 xv = x[fo + (size_t)a * npw + p], loc = line_val(line, (a * spb + s) * ls + iz);
        out[fo + (size_t)a * npw + p] = float2{sc * fmaf(kin, xv.x, loc.x), sc * fmaf(kin, xv.y, loc.y)};
      }
    } else {
      const double kin = ek[p] - shift;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const double2 xv = to_d2(x[fo + (size_t)a * npw + p]), loc = to_d2(line_val(line, (a * spb + s) * ls + iz));
        out[fo + (size_t)a * npw + p] = from_d2<Vg>({scale * fma(kin, xv.x, loc.x), scale * fma(kin, xv.y, loc.y)});
      }
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// lets fn take up to a whole SM's shared memory.  Always the same bound: concurrent solve workers
// launch one kernel with different sizes, and a worker must not lower the bound another relies on
static int allow_smem(const void* fn) {
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e != cudaSuccess) return fail(DKS_ERR_CUDA, std::string("smem attribute: ") + cudaGetErrorString(e));
  return DKS_OK;
}

// sticks per CTA of the stick kernels, as a power of two 2^l <= 32, so that the lines of
// lines_per_stick components stay within `target` bytes of shared memory
static int pick_lspb(int ls, size_t elem, int lines_per_stick, size_t target) {
  int l = 5;
  while (l > 0 && ((size_t)ls * elem * lines_per_stick << l) > target) --l;
  return l;
}

// CTA size of the one-plane kernels: the fewest rounds of butterflies per plane (each round costs
// about a radix), for as many planes per SM as shared memory and `max_threads` resident threads
// allow -- the passes are separated by barriers, so a plane's time is its number of rounds and
// other planes fill the SM meanwhile.  Whole multiples of four warps only, which load the SM's four
// schedulers evenly (48 x 48 complex64 planes: 96 / 128 / 160 / 192 threads 176 / 168 / 176 / 183 us),
// or two warps for small planes.
static int pick_plane_threads(const ExecPlan& e1, const ExecPlan& e2, int nrows, size_t smem, int max_threads) {
  int best = 64;
  double best_cost = 0.0;
  for (int t : {64, 128, 256, 384, 512}) {
    const int res = std::min((int)(228 * 1024 / (smem + 1024)), std::min(32, max_threads / t));
    if (res < 1) break;
    double cost = 0.0;
    for (int i = 0; i < e1.nst; ++i) cost += 2.0 * e1.p[i].R * ((e2.n * (e1.n / e1.p[i].R) + t - 1) / t);
    for (int i = 0; i < e2.nst; ++i) cost += 2.0 * e2.p[i].R * ((nrows * (e2.n / e2.p[i].R) + t - 1) / t);
    cost /= res;
    if (t == 64 || cost < best_cost) {
      best = t;
      best_cost = cost;
    }
  }
  return best;
}
// rows (or columns) of a plane per CTA in the split form: about 64 KB of shared memory
static inline int lines_per_cta(int nlines, int line_stride, size_t elem, size_t extra_per_line = 0) {
  return std::max(1, std::min(nlines, (int)((64 * 1024) / (line_stride * elem + extra_per_line))));
}

template <typename Vg, typename Vs, bool BIG3>
int launch_stick_inverse(const KPoint& kp, const ExecPlan& e3, const typename TwOf<Vs>::T* tw3, const Vg* x, Vs* t,
                                int nf, cudaStream_t st) {
  const int ls = e3.n | 1;                    // odd line stride: conflict-free shared memory
  const int l = pick_lspb(ls, sizeof(Vs), 1, 32 * 1024);
  const size_t sm = ((size_t)ls << l) * sizeof(Vs) + twiddle_bytes<Vs>(e3.ntw);
  DKS_TRY(allow_smem((const void*)k_stick_inverse<Vg, Vs, BIG3>));
  const dim3 g((kp.nsticks + (1 << l) - 1) >> l, nf);
  k_stick_inverse<Vg, Vs, BIG3><<<g, 256, sm, st>>>(x, t, kp.npw, kp.nsticks, kp.stick_start, kp.stick_first, e3, tw3,
                                                    l, ls, magic(1 << l));
  return DKS_OK;
}

template <typename Vg, typename Vs, bool BIG3>
int launch_stick_forward(dks_ctx* ctx, const KPoint& kp, const ExecPlan& e3, const typename TwOf<Vs>::T* tw3, const Vs* t,
                                const Vg* x, Vg* out, int nbc, double shift, double scale, cudaStream_t st) {
  const int ls = e3.n | 1, nc = ctx->ncomp;
  const int l = pick_lspb(ls, sizeof(Vs), nc, 64 * 1024);
  const size_t sm = ((size_t)ls * nc << l) * sizeof(Vs) + twiddle_bytes<Vs>(e3.ntw);
  const void* fn = nc == 4 ? (const void*)k_stick_forward<Vg, Vs, BIG3> : (const void*)k_stick_forward_ks<Vg, Vs, BIG3>;
  DKS_TRY(allow_smem(fn));
  const dim3 g((kp.nsticks + (1 << l) - 1) >> l, nbc);
  const unsigned ml = magic(nc << l);
  if (nc == 4)
    k_stick_forward<Vg, Vs, BIG3><<<g, 256, sm, st>>>(t, x, out, kp.npw, kp.nsticks, kp.stick_start, kp.pw_at, e3,
                                                      tw3, kp.cq64, kp.cq32, ctx->c, shift, scale, l, ls, ml);
  else
    k_stick_forward_ks<Vg, Vs, BIG3><<<g, 256, sm, st>>>(t, x, out, kp.npw, kp.nsticks, kp.stick_start, kp.pw_at, e3,
                                                         tw3, kp.ek, shift, scale, l, ls, ml);
  return DKS_OK;
}

// shared memory of pass B in one kernel: the plane, its twiddles and its row table
template <typename Vs>
static size_t plane_smem(const dks_ctx* ctx, const KPoint& kp, const ExecPlan& e1, const ExecPlan& e2) {
  return (size_t)e1.n * ctx->plane_ld * sizeof(Vs) + twiddle_bytes<Vs>(e1.ntw + e2.ntw) + kp.nrows * sizeof(int);
}

// pass B of nfi fields, in one kernel or split through pbuf
template <typename Vs, bool BIG>
int launch_plane(dks_ctx* ctx, const KPoint& kp, const ExecPlan& e1, const ExecPlan& e2,
                        const typename TwOf<Vs>::T* tw1, const typename TwOf<Vs>::T* tw2,
                        const typename RealOf<Vs>::T* vp, Vs* tbuf, Vs* pbuf, int nfi, cudaStream_t st) {
  const int n1 = e1.n, n2 = e2.n, n3 = ctx->grid[2], ld = ctx->plane_ld, ls1 = n1 | 1;
  if (split_plane(ctx, sizeof(Vs))) {
    if (!pbuf) return fail(DKS_ERR_INVALID_ARG, "split plane FFT without its buffer");
    const int rpb = lines_per_cta(n1, ld, sizeof(Vs)), cpb = lines_per_cta(n2, ls1, sizeof(Vs));
    const size_t sm_r = (size_t)rpb * ld * sizeof(Vs) + twiddle_bytes<Vs>(e2.ntw),
                 sm_cv = (size_t)cpb * ls1 * sizeof(Vs) + twiddle_bytes<Vs>(e1.ntw);
    DKS_TRY(allow_smem((const void*)k_plane_rows_inv<Vs, BIG>));
    DKS_TRY(allow_smem((const void*)k_plane_cols_v<Vs, BIG>));
    DKS_TRY(allow_smem((const void*)k_plane_rows_fwd<Vs, BIG>));
    const dim3 g1(n3, nfi, (n1 + rpb - 1) / rpb), g2(n3, nfi, (n2 + cpb - 1) / cpb);
    const unsigned mr = magic(rpb), mrl = magic(n1 - (n1 - 1) / rpb * rpb), mc = magic(cpb),
                   mcl = magic(n2 - (n2 - 1) / cpb * cpb);
    k_plane_rows_inv<Vs, BIG><<<g1, 256, sm_r, st>>>(tbuf, pbuf, kp.nsticks, kp.stick_plane, e2, ld, n1, n3, tw2,
                                                         rpb, mr, mrl);
    k_plane_cols_v<Vs, BIG><<<g2, 256, sm_cv, st>>>(pbuf, e1, ld, n2, n3, tw1, vp, cpb, ls1, mc, mcl);
    k_plane_rows_fwd<Vs, BIG><<<g1, 256, sm_r, st>>>(tbuf, pbuf, kp.nsticks, kp.stick_plane, e2, ld, n1, n3, tw2,
                                                         rpb, mr, mrl);
    return DKS_OK;
  }
  const size_t sm = plane_smem<Vs>(ctx, kp, e1, e2);
  const int tb = ctx->plane_threads > 0
                     ? ctx->plane_threads
                     : pick_plane_threads(e1, e2, kp.nrows, sm, plane_max_threads(sizeof(Vs), BIG));
  DKS_TRY(allow_smem((const void*)k_plane<Vs, BIG, true>));
  k_plane<Vs, BIG, true><<<dim3(n3, nfi), tb, sm, st>>>(tbuf, kp.nsticks, kp.stick_plane, kp.plane_rows, kp.nrows,
                                                        magic(kp.nrows), e1, e2, ld, magic(n2), n3, tw1, tw2, vp);
  return DKS_OK;
}

// pass B of planes that fit shared memory without their twiddles only
template <typename Vs>
int launch_plane_bare(dks_ctx* ctx, const KPoint& kp, const ExecPlan& e1, const ExecPlan& e2,
                      const typename TwOf<Vs>::T* tw1, const typename TwOf<Vs>::T* tw2,
                      const typename RealOf<Vs>::T* vp, Vs* tbuf, int nfi, cudaStream_t st) {
  const int n3 = ctx->grid[2], ld = ctx->plane_ld;
  const size_t sm = (size_t)e1.n * ld * sizeof(Vs);
  const int tb = ctx->plane_threads > 0
                     ? ctx->plane_threads
                     : pick_plane_threads(e1, e2, kp.nrows, sm, plane_max_threads(sizeof(Vs), true));
  DKS_TRY(allow_smem((const void*)k_plane<Vs, true, false>));
  k_plane<Vs, true, false><<<dim3(n3, nfi), tb, sm, st>>>(tbuf, kp.nsticks, kp.stick_plane, kp.plane_rows, kp.nrows,
                                                          magic(kp.nrows), e1, e2, ld, magic(e2.n), n3, tw1, tw2, vp);
  return DKS_OK;
}

// The three FFT passes over chunks of bands.  Vg is the type of x and out, Vs the arithmetic type of
// the transforms and of the intermediates T and P: the same type, or double-float (cdp) for
// complex128 data in the emulated-FP64 mode.
template <typename Vg, typename Vs>
int fft_local(dks_ctx* ctx, const KPoint& kp, const Vg* x, Vg* out, int nb, int chunk, Vs* tbuf, void* pbufv,
                     double shift, double scale, cudaStream_t st) {
  const bool fp64 = sizeof(Vg) == sizeof(double2);
  const bool df = !std::is_same<Vg, Vs>::value;
  const int npw = kp.npw, n3 = ctx->grid[2];
  const size_t field_elems = (size_t)kp.nsticks * n3;
  using TW = typename TwOf<Vs>::T;
  const TW* tw1 = df ? (const TW*)ctx->etwdf[0] : fp64 ? (const TW*)ctx->etw64[0] : (const TW*)ctx->etw32[0];
  const TW* tw2 = df ? (const TW*)ctx->etwdf[1] : fp64 ? (const TW*)ctx->etw64[1] : (const TW*)ctx->etw32[1];
  const TW* tw3 = df ? (const TW*)ctx->etwdf[2] : fp64 ? (const TW*)ctx->etw64[2] : (const TW*)ctx->etw32[2];
  const ExecPlan* ep = sizeof(Vs) == sizeof(float2) ? ctx->exec32 : ctx->exec64;
  using VR = typename RealOf<Vs>::T;
  const VR* vp = df ? (const VR*)ctx->vpermdf : fp64 ? (const VR*)ctx->vperm64 : (const VR*)ctx->vperm32;
  const int nc = ctx->ncomp;                   // fields per band: 4 (DKS) or 2 (KSSO)
  const int cat32 = fp64 ? 0 : kProf32;
  const bool split = split_plane(ctx, sizeof(Vs));
  for (int b0 = 0; b0 < nb; b0 += chunk) {
    const int nbc = std::min(chunk, nb - b0);
    const Vg* xb = x + (size_t)b0 * nc * npw;
    Vg* ob = out + (size_t)b0 * nc * npw;
    const double nf = (double)nc * nbc, es = (double)sizeof(Vg);
    const double tb = nf * (double)field_elems * es;          // one pass over the stick buffer
    const double f3 = 5.0 * n3 * std::log2((double)n3) * kp.nsticks * nf;
    {
      Prof pr(P_STICK_INV + cat32, st, nf * npw * es + tb, f3);
      if (ep[2].big) DKS_TRY((launch_stick_inverse<Vg, Vs, true>(kp, ep[2], tw3, xb, tbuf, nc * nbc, st)));
      else DKS_TRY((launch_stick_inverse<Vg, Vs, false>(kp, ep[2], tw3, xb, tbuf, nc * nbc, st)));
    }
    {
      const double nn = (double)ctx->grid[0] * ctx->grid[1];
      Prof pr(P_PLANE + cat32, st, 2.0 * tb + (double)ctx->ng * es / 2,
              nf * n3 * (10.0 * nn * std::log2(nn) + 2.0 * nn));
      if (split) pr.count(2);
      Vs* pbuf = reinterpret_cast<Vs*>(pbufv);
      if (!split && plane_smem<Vs>(ctx, kp, ep[0], ep[1]) > kPlaneSmem)
        DKS_TRY((launch_plane_bare<Vs>(ctx, kp, ep[0], ep[1], tw1, tw2, vp, tbuf, nc * nbc, st)));
      else if (ep[0].big || ep[1].big)
        DKS_TRY((launch_plane<Vs, true>(ctx, kp, ep[0], ep[1], tw1, tw2, vp, tbuf, pbuf, nc * nbc, st)));
      else
        DKS_TRY((launch_plane<Vs, false>(ctx, kp, ep[0], ep[1], tw1, tw2, vp, tbuf, pbuf, nc * nbc, st)));
    }
    {
      Prof pr(P_STICK_FWD + cat32, st, tb + 2.0 * nf * npw * es + 24.0 * npw,
              f3 + (nc == 4 ? 64.0 : 8.0) * nbc * npw);
      if (ep[2].big) DKS_TRY((launch_stick_forward<Vg, Vs, true>(ctx, kp, ep[2], tw3, tbuf, xb, ob, nbc, shift, scale, st)));
      else DKS_TRY((launch_stick_forward<Vg, Vs, false>(ctx, kp, ep[2], tw3, tbuf, xb, ob, nbc, shift, scale, st)));
    }
  }
  DKS_CUDA_TRY(cudaGetLastError());
  return DKS_OK;
}

// the first failed index check of this translation unit's kernels since the last call, then cleared
// (debug build; 0 in the product build)
static unsigned debug_take_unit() {
#ifdef DKS_DEBUG
  unsigned v = 0u, z = 0u;
  if (cudaMemcpyFromSymbol(&v, g_dks_check, sizeof(v)) != cudaSuccess) return 0xffffffffu;
  cudaMemcpyToSymbol(g_dks_check, &z, sizeof(z));
  return v;
#else
  return 0u;
#endif
}

}  // namespace dks
