// Mixed-radix FFT passes over lines held in shared memory (radices 2..8 and the merged radices 9,
// 10, 12, 14, 15, 16).
//
// A pass of radix R over a block length L (sub-length S = L / R) combines the R elements
// j, j + S, ..., j + (R-1) S of every length-L block.  The decimation-in-frequency (DIF) pass
// applies the small DFT and then multiplies output m by w^(j m N/L); the decimation-in-time
// (DIT) pass multiplies input r by w^(j r N/L) first.  Running the DIF passes with L = N, N/R0,
// ... leaves the spectrum in mixed-radix digit-reversed order, and the DIT passes in the
// opposite order take that order back to natural order, so a DIF inverse transform followed by
// a DIT forward transform needs no permutation at all.
//
// Only the inverse sign (+) exists in the device code.  The forward transform of z is the swapped
// inverse transform of swap(z) (swap exchanges the real and imaginary parts), so the forward
// phase keeps its data swapped: the swap costs nothing where the data is multiplied by V or loaded
// from global memory, and one copy of every butterfly serves both directions (the double-float
// butterflies are thousands of instructions; four copies of each overflowed the instruction cache).
//
// The small DFTs use fixed butterflies with the roots of unity as compile-time constants: the
// odd radices pair inputs r and R-r (R=3, 5, 7), composite radices are a two-factor split with
// constant inner twiddles.  Only the inter-pass twiddles come from a table.
//
// Execution passes (ExecPlan) merge two neighbouring passes (Ra, Rb) of an AxisPlan into one of
// radix Ra Rb where the product is at most 16 (10 for the 16-byte types): one trip through shared
// memory and one set of twiddles less.  A merged DIF pass stores output m at sub-block
// (m mod Ra) Rb + m / Ra, so the digit-reversed order of the axis plan is unchanged.
//
// Thread mapping: consecutive threads take consecutive lines (same butterfly position), so a
// warp touches addresses one line stride apart; callers give lines an odd stride (contiguous
// lines) or a unit stride (strided lines), which keeps shared-memory accesses free of bank
// conflicts for 8- and 16-byte elements, and makes the twiddle reads broadcasts.  Positions come
// from one multiply-high per division (ExecPass::mS, magic()); twiddles are laid out [j][r] per
// pass, so a butterfly's factors are at constant offsets from one address.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "dks_internal.h"
#include "dks_kernels.cuh"

namespace dks {

// ------------------------------------------------------------------ constants
// cos and sin of 2 pi t / 5040 (every root of unity of the radices is one of these): reduced to
// the first octant in integers, then a correctly rounded literal
__host__ __device__ constexpr double root_octant(int t, bool sine) {
  switch (t) {
    case 84: return sine ? 0.1045284632676534713998 : 0.9945218953682733369227;
    case 140: return sine ? 0.1736481776669303488517 : 0.9848077530122080593667;
    case 168: return sine ? 0.2079116908177593371017 : 0.9781476007338056379286;
    case 180: return sine ? 0.2225209339563144042889 : 0.9749279121818236070181;
    case 252: return sine ? 0.3090169943749474241023 : 0.9510565162951535721164;
    case 280: return sine ? 0.3420201433256687330441 : 0.9396926207859083840541;
    case 315: return sine ? 0.3826834323650897717285 : 0.9238795325112867561282;
    case 336: return sine ? 0.406736643075800207754 : 0.9135454576426008955021;
    case 360: return sine ? 0.4338837391175581204758 : 0.9009688679024191262361;
    case 420: return sine ? 0.5 : 0.8660254037844386467637;
    case 504: return sine ? 0.5877852522924731291687 : 0.8090169943749474241023;
    case 540: return sine ? 0.623489801858733530525 : 0.7818314824680298087084;
    case 560: return sine ? 0.6427876096865393263226 : 0.7660444431189780352024;
    case 588: return sine ? 0.6691306063588582138263 : 0.7431448254773942350147;
    case 630: return sine ? 0.7071067811865475244008 : 0.7071067811865475244008;
    default: return sine ? 0.0 : 1.0;   // t = 0
  }
}
__host__ __device__ constexpr double root_cs(int t, bool sine) {
  if (t > 2520) return sine ? -root_cs(5040 - t, true) : root_cs(5040 - t, false);
  if (t > 1260) return sine ? root_cs(2520 - t, true) : -root_cs(2520 - t, false);
  return t > 630 ? root_octant(1260 - t, !sine) : root_octant(t, sine);
}
// cos(2 pi k / R), sin(2 pi k / R)
__host__ __device__ constexpr double root_cos(int R, int k) { return root_cs(k % R * (5040 / R), false); }
__host__ __device__ constexpr double root_sin(int R, int k) { return root_cs(k % R * (5040 / R), true); }

// ------------------------------------------------------------------ arithmetic types
// float2, double2, and cdp: a complex double-float value stored as the pair of leading parts and the
// pair of trailing parts, so that one packed instruction (add, mul, fma .f32x2) does the real and
// the imaginary part of a step.  The packed forms run at the same FP32 rate (39 T lane operations/s
// either way), but issue and instruction fetch halve, which is what the double-float butterflies
// (thousands of instructions each) are bound by.  Every operation rounds as its scalar form.
struct __align__(16) cdp {
  float2 h, l;
};
template <> struct RealOf<cdp> { using T = dfl; };

__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __ffma2_rn(b, float2{-1.f, -1.f}, a); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return p_add(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return p_sub(a, b); }
// a + i b and a - i b
template <typename V> __device__ __forceinline__ V cadd_i(V a, V b) { return V{a.x - b.y, a.y + b.x}; }
template <typename V> __device__ __forceinline__ V csub_i(V a, V b) { return V{a.x + b.y, a.y - b.x}; }

// (s + e) renormalised, as in df_add: h = s + e, l = e - (h - s)
__device__ __forceinline__ cdp p_renorm(float2 s, float2 e) {
  const float2 h = p_add(s, e);
  return cdp{h, p_sub(e, p_sub(h, s))};
}
// df_add on both parts
__device__ __forceinline__ cdp cadd(cdp a, cdp b) {
  const float2 s = p_add(a.h, b.h);
  const float2 bb = p_sub(s, a.h);
  const float2 e = p_add(p_sub(a.h, p_sub(s, bb)), p_sub(b.h, bb));
  return p_renorm(s, p_add(e, p_add(a.l, b.l)));
}
// df_add(a, -b)
__device__ __forceinline__ cdp csub(cdp a, cdp b) {
  const float2 s = p_sub(a.h, b.h);
  const float2 bb = p_sub(s, a.h);   // close to -b.h
  const float2 e = p_sub(p_sub(a.h, p_sub(s, bb)), p_add(b.h, bb));
  return p_renorm(s, p_add(e, p_sub(a.l, b.l)));
}
// df_mul of both parts by a real double-float pair, whose parts are given duplicated and negated
__device__ __forceinline__ cdp p_dmul(cdp a, float2 ch, float2 nch, float2 ncl) {
  const float2 p = p_mul(a.h, ch);
  float2 ne = p_fma(a.h, nch, p);    // -(error of p), exact
  ne = p_fma(a.h, ncl, ne);
  ne = p_fma(a.l, nch, ne);
  const float2 h = p_sub(p, ne);
  return cdp{h, p_sub(p_sub(p, h), ne)};
}
__device__ __forceinline__ cdp cscale(cdp a, dfl s) {
  return p_dmul(a, float2{s.h, s.h}, float2{-s.h, -s.h}, float2{-s.l, -s.l});
}
__device__ __forceinline__ cdp mul_i(cdp a) { return cdp{float2{-a.h.y, a.h.x}, float2{-a.l.y, a.l.x}}; }
__device__ __forceinline__ cdp cadd_i(cdp a, cdp b) { return cadd(a, mul_i(b)); }
__device__ __forceinline__ cdp csub_i(cdp a, cdp b) { return csub(a, mul_i(b)); }
// a twiddle as the tables hold it: for cdp the duplicated and negated parts p_dmul multiplies by
struct __align__(16) ctw {
  float2 rh, nrh, nrl, ih, nih, nil;   // re: h, -h, -l; im: h, -h, -l
};
static_assert(sizeof(ctw) == kTwDfFloats * sizeof(float), "layout of the uploaded table");
template <typename V> struct TwOf { using T = V; };
template <> struct TwOf<cdp> { using T = ctw; };
// a w = w_re a + w_im (i a)
__device__ __forceinline__ cdp cmul(cdp a, const ctw& w) {
  return cadd(p_dmul(a, w.rh, w.nrh, w.nrl), p_dmul(mul_i(a), w.ih, w.nih, w.nil));
}
__device__ __forceinline__ cdp cdp_split(double2 v) {
  const dfl re = df_split_rn(v.x), im = df_split_rn(v.y);
  return cdp{float2{re.h, im.h}, float2{re.l, im.l}};
}
__device__ __forceinline__ double2 to_d2(cdp v) {
  return double2{df_to_double_any(v.h.x, v.l.x), df_to_double_any(v.h.y, v.l.y)};
}
template <typename V> __device__ __forceinline__ V vzero() { return V{0, 0}; }
template <> __device__ __forceinline__ cdp vzero<cdp>() { return cdp{{0.f, 0.f}, {0.f, 0.f}}; }
template <typename V> __device__ __forceinline__ V cswap(V a) { return V{a.y, a.x}; }
template <> __device__ __forceinline__ cdp cswap<cdp>(cdp a) {
  return cdp{float2{a.h.y, a.h.x}, float2{a.l.y, a.l.x}};
}

// a real constant in the three arithmetic types: double, float, and a double-float pair
struct RK {
  double d;
  float h, l;
};
__host__ __device__ constexpr RK rk(double x) { return RK{x, (float)x, (float)(x - (double)(float)x)}; }

__device__ __forceinline__ float2 rmul(float2 a, RK c) { return p_mul(a, float2{c.h, c.h}); }
__device__ __forceinline__ double2 rmul(double2 a, RK c) { return double2{a.x * c.d, a.y * c.d}; }
__device__ __forceinline__ cdp rmul(cdp a, RK c) { return cscale(a, dfl{c.h, c.l}); }

// acc + c a and acc - c a: fused for float2 and double2 (one rounding per part)
__device__ __forceinline__ float2 racc(float2 acc, float2 a, RK c) { return p_fma(a, float2{c.h, c.h}, acc); }
__device__ __forceinline__ double2 racc(double2 acc, double2 a, RK c) {
  return double2{fma(a.x, c.d, acc.x), fma(a.y, c.d, acc.y)};
}
__device__ __forceinline__ cdp racc(cdp acc, cdp a, RK c) { return cadd(acc, rmul(a, c)); }
// c a + i s a
__device__ __forceinline__ float2 rrot(float2 a, RK c, RK s) {
  const float2 t = p_mul(a, float2{s.h, s.h});
  return float2{fmaf(a.x, c.h, -t.y), fmaf(a.y, c.h, t.x)};
}
__device__ __forceinline__ double2 rrot(double2 a, RK c, RK s) {
  return double2{fma(a.x, c.d, -s.d * a.y), fma(a.y, c.d, s.d * a.x)};
}
__device__ __forceinline__ cdp rrot(cdp a, RK c, RK s) { return cadd_i(rmul(a, c), rmul(a, s)); }

// a * exp(i 2 pi k / R)
template <int R, int K, typename V>
__device__ __forceinline__ V mul_root(V a) {
  static_assert(5040 % R == 0, "radix without tabulated roots");
  if constexpr (K == 0) {
    return a;
  } else if constexpr (4 * K == R) {
    return mul_i(a);
  } else {
    constexpr RK c = rk(root_cos(R, K)), s = rk(root_sin(R, K));
    return rrot(a, c, s);
  }
}

// compile-time loop
template <int I, int N, typename F>
__device__ __forceinline__ void sfor(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    sfor<I + 1, N>(f);
  }
}

// ------------------------------------------------------------------ small DFTs, y = DFT_R(x)
template <typename V, int R>
__device__ __forceinline__ void dft(const V* x, V* y);

// odd R: pairs a_r = x_r + x_{R-r}, b_r = x_r - x_{R-r};
// y_m, y_{R-m} = x_0 + sum_r a_r cos(2 pi r m / R) +- i sum_r b_r sin(2 pi r m / R)
template <typename V, int R>
__device__ __forceinline__ void dft_odd(const V* x, V* y) {
  constexpr int H = (R - 1) / 2;
  V a[H], b[H];
  V y0 = x[0];
  sfor<1, H + 1>([&](auto rc) {
    constexpr int r = decltype(rc)::value;
    a[r - 1] = cadd(x[r], x[R - r]);
    b[r - 1] = csub(x[r], x[R - r]);
    y0 = cadd(y0, a[r - 1]);
  });
  sfor<1, H + 1>([&](auto mc) {
    constexpr int m = decltype(mc)::value;
    V re = x[0], im;
    sfor<1, H + 1>([&](auto rc) {
      constexpr int r = decltype(rc)::value;
      constexpr int k = (r * m) % R;
      constexpr int kk = k <= H ? k : R - k;
      constexpr RK c = rk(root_cos(R, kk));
      re = racc(re, a[r - 1], c);
      constexpr RK sk = rk(k <= H ? root_sin(R, kk) : -root_sin(R, kk));
      im = r == 1 ? rmul(b[r - 1], sk) : racc(im, b[r - 1], sk);
    });
    y[m] = cadd_i(re, im);
    y[R - m] = csub_i(re, im);
  });
  y[0] = y0;
}

// R = P Q, n = Q n1 + n2, k = k1 + P k2:
// y[k1 + P k2] = sum_n2 w_Q^(n2 k2) [ w_R^(n2 k1) sum_n1 x[Q n1 + n2] w_P^(n1 k1) ]
template <typename V, int P, int Q>
__device__ __forceinline__ void dft_split(const V* x, V* y) {
  constexpr int R = P * Q;
  V a[Q][P];
  sfor<0, Q>([&](auto n2c) {
    constexpr int n2 = decltype(n2c)::value;
    V in[P];
    sfor<0, P>([&](auto n1c) { in[decltype(n1c)::value] = x[Q * decltype(n1c)::value + n2]; });
    dft<V, P>(in, a[n2]);
    sfor<1, P>([&](auto k1c) {
      constexpr int k1 = decltype(k1c)::value;
      a[n2][k1] = mul_root<R, n2 * k1>(a[n2][k1]);
    });
  });
  sfor<0, P>([&](auto k1c) {
    constexpr int k1 = decltype(k1c)::value;
    V in[Q], out[Q];
    sfor<0, Q>([&](auto n2c) { in[decltype(n2c)::value] = a[decltype(n2c)::value][k1]; });
    dft<V, Q>(in, out);
    sfor<0, Q>([&](auto k2c) { y[k1 + P * decltype(k2c)::value] = out[decltype(k2c)::value]; });
  });
}

template <typename V, int R>
__device__ __forceinline__ void dft(const V* x, V* y) {
  if constexpr (R == 1) {
    y[0] = x[0];
  } else if constexpr (R == 2) {
    y[0] = cadd(x[0], x[1]);
    y[1] = csub(x[0], x[1]);
  } else if constexpr (R == 4) {
    const V a = cadd(x[0], x[2]), b = csub(x[0], x[2]);
    const V c = cadd(x[1], x[3]), d = csub(x[1], x[3]);
    y[0] = cadd(a, c);
    y[2] = csub(a, c);
    y[1] = cadd_i(b, d);
    y[3] = csub_i(b, d);
  } else if constexpr (R == 6) {
    dft_split<V, 2, 3>(x, y);
  } else if constexpr (R == 8) {
    dft_split<V, 2, 4>(x, y);
  } else {
    static_assert(R == 3 || R == 5 || R == 7, "unsupported radix");
    dft_odd<V, R>(x, y);
  }
}

template <typename V, int P, int Q>
__device__ __forceinline__ void dft_pq(const V* x, V* y) {
  if constexpr (Q == 1) dft<V, P>(x, y);
  else dft_split<V, P, Q>(x, y);
}

// ------------------------------------------------------------------ passes
// a / d for 0 <= a < 65536 by m = magic(d) = ceil(2^32 / d) (0 stands for d = 1)
__device__ __forceinline__ int mdiv(int a, unsigned m) { return m ? (int)__umulhi((unsigned)a, m) : a; }

// the n lines a pass runs over: line l starts at rows[l] (a table in shared memory) or at l * lstride;
// its element i is es elements further per unit.  mN = magic(n)
struct Lines {
  const int* rows;
  int lstride, es, n;
  unsigned mN;
};

// Where a pass reads and writes: shared memory in place; or the last DIF pass storing straight to
// the stick buffer T; or the first DIT pass loading straight from it (T[component][position][stick],
// consecutive lines of a component are consecutive sticks, so both are coalesced).  The stick
// kernels save a trip through shared memory, a barrier and a loop that way.
enum PassIO { kInPlace, kStoreT, kLoadT };
template <typename V>
struct StickBuf {
  V* t;             // T at the CTA's first stick
  int nsticks, ns;  // stick count (the stride of a position), sticks of this CTA
  int lspb;         // log2 of the lines per component in shared memory
  size_t comp;      // stride of a component
};

// one execution pass of radix R = P Q (P then Q of the axis plan; Q = 1: a plain radix).
//   DIF: x[r] from sub-block r, y[m] w^(j m) to sub-block sigma(m) = (m mod P) Q + m / P
//   DIT (swapped data): x[r] w^(j r) from sub-block sigma(r), y[m] to sub-block m
//   vmid (only where S = 1): the last DIF pass of an inverse transform, the product with the real
//   factors vmid[offset] and the first DIT pass of the forward transform in one, without a trip
//   through shared memory between them; the result is swapped data
//   DIR: 0 DIF, 1 DIT, 2 as dit_rt says
template <typename V, int P, int Q, PassIO IO, int DIR>
__device__ __forceinline__ void fft_pass_dir(V* __restrict__ buf, const Lines& ln, const ExecPass& p, int n,
                                         const typename TwOf<V>::T* __restrict__ tw, bool dit_rt,
                                         const typename RealOf<V>::T* __restrict__ vmid, const StickBuf<V>& sb) {
  constexpr int R = P * Q;
  const bool dit = DIR == 2 ? dit_rt : DIR == 1;
  const int S = p.S;
  const int total = ln.n * (n / R);
  const int se = S * ln.es;
#pragma unroll 1
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int u = mdiv(t, ln.mN);
    const int line = t - u * ln.n;
    const int blk = mdiv(u, p.mS);
    const int j = u - blk * S;
    const int pos = blk * p.L + j;
    V* base = buf + (ln.rows ? ln.rows[line] : line * ln.lstride) + pos * ln.es;
    V* gbase = nullptr;
    if constexpr (IO != kInPlace) {
      const int s = line & ((1 << sb.lspb) - 1);
      if (s >= sb.ns) continue;   // beyond the last stick
      gbase = sb.t + (size_t)(line >> sb.lspb) * sb.comp + (size_t)pos * sb.nsticks + s;
    }
    const int gse = S * sb.nsticks;
    V x[R], y[R];
    sfor<0, R>([&](auto rc) {
      constexpr int r = decltype(rc)::value, sr = (r % P) * Q + r / P;
      const int slot = Q > 1 && dit ? sr : r;
      if constexpr (IO == kLoadT) x[r] = gbase[(size_t)slot * gse];
      else x[r] = base[slot * se];
    });
    if (dit && j) {
      const typename TwOf<V>::T* w = tw + j * R;
      sfor<1, R>([&](auto rc) { x[decltype(rc)::value] = cmul(x[decltype(rc)::value], w[decltype(rc)::value]); });
    }
    if (DIR != 1 && vmid) {
      const typename RealOf<V>::T* vb = vmid + (base - buf);
      typename RealOf<V>::T vv[R];
      sfor<0, R>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        vv[r] = vb[((r % P) * Q + r / P) * se];
      });
#pragma unroll 1
      for (int rep = 0;; ++rep) {
        dft_pq<V, P, Q>(x, y);
        if (rep) break;
        sfor<0, R>([&](auto rc) { x[decltype(rc)::value] = cswap(cscale(y[decltype(rc)::value], vv[decltype(rc)::value])); });
      }
    } else {
      dft_pq<V, P, Q>(x, y);
    }
    if (!dit && j) {
      const typename TwOf<V>::T* w = tw + j * R;
      sfor<1, R>([&](auto rc) { y[decltype(rc)::value] = cmul(y[decltype(rc)::value], w[decltype(rc)::value]); });
    }
    sfor<0, R>([&](auto rc) {
      constexpr int r = decltype(rc)::value, sr = (r % P) * Q + r / P;
      const int slot = Q > 1 && !dit && !vmid ? sr : r;
      if constexpr (IO == kStoreT) gbase[(size_t)slot * gse] = y[r];
      else base[slot * se] = y[r];
    });
  }
}

// One copy of a pass for both directions costs FP32 types little and keeps the double-float butterflies in
// the instruction cache; in native FP64 the factors of the other direction would still take their slots of
// the FP64 unit as predicated-off instructions (27 % more of them for 100 x 100 planes), so there each
// direction has its copy.
template <typename V, int P, int Q, PassIO IO>
__device__ __forceinline__ void fft_pass(V* __restrict__ buf, const Lines& ln, const ExecPass& p, int n,
                                         const typename TwOf<V>::T* __restrict__ tw, bool dit,
                                         const typename RealOf<V>::T* __restrict__ vmid, const StickBuf<V>& sb) {
  if constexpr (std::is_same<V, double2>::value) {
    if (dit) fft_pass_dir<V, P, Q, IO, 1>(buf, ln, p, n, tw, dit, vmid, sb);
    else fft_pass_dir<V, P, Q, IO, 0>(buf, ln, p, n, tw, dit, vmid, sb);
  } else {
    fft_pass_dir<V, P, Q, IO, 2>(buf, ln, p, n, tw, dit, vmid, sb);
  }
}

// one pass of any radix, and the barrier after it.  BIG: plans with merged radices (more registers)
template <typename V, bool BIG, PassIO IO = kInPlace>
__device__ __forceinline__ void fft_step(V* buf, const Lines& ln, const ExecPass& p, int n,
                                         const typename TwOf<V>::T* tw, bool dit, const typename RealOf<V>::T* vmid,
                                         const StickBuf<V>& sb = {}) {
  switch (p.R) {
    case 1: fft_pass<V, 1, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    case 2: fft_pass<V, 2, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    case 3: fft_pass<V, 3, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    case 4: fft_pass<V, 4, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    case 5: fft_pass<V, 5, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    case 6: fft_pass<V, 6, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    case 7: fft_pass<V, 7, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    case 8: fft_pass<V, 8, 1, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
    default:
      if constexpr (BIG) {
        switch (p.R) {
          case 9: fft_pass<V, 3, 3, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
          case 10: fft_pass<V, 5, 2, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
          default:
            if constexpr (sizeof(V) == sizeof(float2)) {
              switch (p.R) {
                case 12: fft_pass<V, 6, 2, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
                case 14: fft_pass<V, 7, 2, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
                case 15: fft_pass<V, 5, 3, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
                default: fft_pass<V, 8, 2, IO>(buf, ln, p, n, tw, dit, vmid, sb); break;
              }
            }
        }
      }
  }
  __syncthreads();
}

// all passes of one axis: DIF passes in plan order, DIT passes in reverse order
template <typename V, bool BIG>
__device__ __forceinline__ void fft_axis(V* buf, const Lines& ln, const ExecPlan& e, const typename TwOf<V>::T* tw,
                                         bool dit) {
#pragma unroll 1
  for (int i = 0; i < e.nst; ++i) {
    const int s = dit ? e.nst - 1 - i : i;
    fft_step<V, BIG>(buf, ln, e.p[s], e.n, tw + e.p[s].tw, dit, nullptr);
  }
}

// the inverse transform of the lines of axis 3 in shared memory, its last pass storing to T, and the
// forward transform from T, its first pass loading from there
template <typename V, bool BIG>
__device__ __forceinline__ void fft_axis_store(V* buf, const Lines& ln, const ExecPlan& e,
                                               const typename TwOf<V>::T* tw, const StickBuf<V>& sb) {
#pragma unroll 1
  for (int i = 0; i + 1 < e.nst; ++i) fft_step<V, BIG>(buf, ln, e.p[i], e.n, tw + e.p[i].tw, false, nullptr);
  const ExecPass& p = e.p[e.nst - 1];
  fft_step<V, BIG, kStoreT>(buf, ln, p, e.n, tw + p.tw, false, nullptr, sb);
}
template <typename V, bool BIG>
__device__ __forceinline__ void fft_axis_load(V* buf, const Lines& ln, const ExecPlan& e,
                                              const typename TwOf<V>::T* tw, const StickBuf<V>& sb) {
  const ExecPass& p = e.p[e.nst - 1];
  fft_step<V, BIG, kLoadT>(buf, ln, p, e.n, tw + p.tw, true, nullptr, sb);
#pragma unroll 1
  for (int i = e.nst - 2; i >= 0; --i) fft_step<V, BIG>(buf, ln, e.p[i], e.n, tw + e.p[i].tw, true, nullptr);
}

// copies n twiddles into shared memory (the caller's next barrier publishes them)
template <typename TW>
__device__ __forceinline__ void load_twiddles(TW* dst, const TW* __restrict__ src, int n) {
  for (int e = threadIdx.x; e < n; e += blockDim.x) dst[e] = src[e];
}

// shared memory of n twiddles, with room for their alignment
template <typename V>
static size_t twiddle_bytes(int n) {
  return n * sizeof(typename TwOf<V>::T) + 16;
}
}  // namespace dks
