// CUDA kernels of the FC spectral ISPH hot path (sm_103a).
//
// Data layout (HBM).  Real fields f[b][c][j] (j = y, contiguous; c = x index,
// or x * nz + z on a 3D grid).  Spectra after the y transform are stored
// transposed, S[b][field][ky][c] (c contiguous), so that the x pass reads
// whole rows (3D: x lines at stride nz, after a z pass over contiguous runs).
// The FC-extended grid is never materialised in HBM on the hot path: the
// continuation is computed in shared memory inside the transform kernels.
//
// Transform kernels run 32, 64 or 128 threads per CTA (one warp, whose
// barriers are warp barriers, for full batches; more where a pass has few
// lines or long ones), the threads of a CTA sharing its lines.  Column
// kernels (y direction) handle
// 2*Pp adjacent columns of one instance: two real columns are packed into
// one complex line (a + i b), transformed together, and separated with the
// Hermitian split
//   A_k = (Z_k + conj Z_{-k}) / 2,  B_k = (Z_k - conj Z_{-k}) / (2i).
// Row kernels (x direction) handle Rr x lines of one instance.  Outputs are
// formed and inverted together as far as shared memory leaves 12 warps per SM.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <type_traits>

#include "fcsph_ip.cuh"
#include "fcsph_warpfft.cuh"
#include "fcsph_regfft.cuh"
#include "fcsph_tma.cuh"
#include "fcsph_internal.h"

using namespace fcsph;

namespace {

constexpr int kThreads = 256;
// FFT kernels are launched with 32, 64 or 128 threads, which share the lines of
// their CTA, and are built three times: for plans of radices up to 9 (RM = 9), up
// to 17 (RM = 17) and for every plan (RM = 31: the large prime radices too).  The
// FP32-pair butterfly of 17 points holds 68 registers of data alone; without the
// radices above 9 the register allocator needs no spills at 128 registers (8
// bytes at 96), so more warps are resident to hide the latency of the dependent
// pair operations, shared-memory and table loads.  The large prime radices'
// code cost the others time where it stood between them: pressure solves of
// 256^2, length 510, 403 us with it and 397 without.
// Minimum resident 128-thread CTAs per SM asked of the register allocator.
template <typename T, int RM> struct MinCtas { static constexpr int v = RM <= 9 ? 4 : 3; };
template <int RM> struct MinCtas<float, RM> { static constexpr int v = RM <= 9 ? 8 : 4; };
// The line operator keeps its outputs' symbols live beside the transforms.
template <typename T, int RM> struct LineMinCtas { static constexpr int v = MinCtas<T, RM>::v; };
template <int RM> struct LineMinCtas<float, RM> { static constexpr int v = 4; };
constexpr int kMaxThreads = 128;
constexpr int kTeamsLine = 1;  // teams per CTA of the register line operator
// Calls f(std::integral_constant<int, RM>) for the largest radix of the plans.
template <typename F> cudaError_t with_rm(int rmax, F&& f) {
  if (rmax <= 9) return f(std::integral_constant<int, 9>{});
  if (rmax <= 17) return f(std::integral_constant<int, 17>{});
  return f(std::integral_constant<int, 31>{});
}

// A field value in the compute type (FP32 pairs: converted on the integer units).
template <typename T, typename U> __device__ __forceinline__ T to_t(U x) {
  if constexpr (std::is_same<T, ff>::value && std::is_same<U, double>::value) return ff_from(x);
  else return (T)x;
}

template <typename T> struct PoolOf;
template <> struct PoolOf<double> { static const double2* get(const fcsph_ctx* c) { return c->pool64; } };
template <> struct PoolOf<float> { static const float2* get(const fcsph_ctx* c) { return c->pool32; } };
template <> struct PoolOf<ff> { static const ff2* get(const fcsph_ctx* c) { return static_cast<const ff2*>(c->poolff); } };

// Loads of the spectra and fields a pass streams through go past L1 (each
// value is read once by its CTA): L1, what shared memory leaves of it, then
// keeps the roots, kernel transforms and index tables every line reads again.
__device__ __forceinline__ double2 ld_stream(const double2* p) { return __ldcg(p); }
__device__ __forceinline__ float2 ld_stream(const float2* p) { return __ldcg(p); }
__device__ __forceinline__ ff2 ld_stream(const ff2* p) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
  ff2 r;
  r.h = make_float2(v.x, v.y);
  r.l = make_float2(v.z, v.w);
  return r;
}
__device__ __forceinline__ double ld_stream(const double* p) { return __ldcg(p); }
__device__ __forceinline__ float ld_stream(const float* p) { return __ldcg(p); }

// for (k = threadIdx.x; k < n; k += blockDim.x) in batches of U indices: load(u,
// k) for all of them, then use(u, k) for all of them.  The loads of a batch
// are in flight together; in a plain loop the stores of one index (to shared
// or global memory the compiler cannot tell from what the next index reads)
// hold back the loads of the next.
template <int U, typename L, typename F> __device__ __forceinline__ void batched(int n, L load, F use) {
  for (int k0 = threadIdx.x; k0 < n; k0 += U * blockDim.x) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u * (int)blockDim.x < n) load(u, k0 + u * (int)blockDim.x);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u * (int)blockDim.x < n) use(u, k0 + u * (int)blockDim.x);
  }
}

__device__ __forceinline__ size_t fidx(const GridDev& g, int b, int i, int j) {
  return ((size_t)b * g.ncol + i) * g.ny + j;
}

// ---------------------------------------------------------------------------
// Compensated dot product for the FC continuation sum_m E[m] b[m]: the table
// entries reach ~1e4 while the result is O(|b|), so each product is split
// exactly (p + e = a*b via fma) and the terms are added with TwoSum; the
// result is accurate to a few ulps of the result instead of ulps of the terms.
struct Dot2 {
  double s = 0.0, c = 0.0;
  __device__ __forceinline__ void add(double a, double b) {
    const double p = __dmul_rn(a, b);
    join(p, fma(a, b, -p));
  }
  // the first product: what add() gives on an empty sum, 8 operations fewer
  __device__ __forceinline__ void start(double a, double b) {
    s = __dmul_rn(a, b);
    c = fma(a, b, -s);
  }
  // + t + e, e smaller than t's rounding errors
  __device__ __forceinline__ void join(double t, double e) {
    const double sum = s + t;
    const double bp = sum - s;
    c += (s - (sum - bp)) + (t - bp) + e;
    s = sum;
  }
  __device__ __forceinline__ double value() const { return s + c; }
};

// FC continuation sum of one line component: compensated FP64 (Dot2, table
// in double) for FP64 transforms; FP32-pair arithmetic (table in FP32 pairs)
// for FP32x2 and FP32 transforms.  For FP32 the pair sum (error ~2^-48 of
// sum |E b|) rounds to the same FP32 value an FP64 sum would, on the FP32
// units: the sum needs more than FP32 because the terms reach ~1e3-1e4 |b|.
template <typename T> struct FcTab { typedef double t; };
template <> struct FcTab<ff> { typedef ff t; };
template <> struct FcTab<float> { typedef ff t; };

// acc += e * x for both components of a complex line value.
template <typename T> struct FcAcc {
  Dot2 x, y;
  __device__ __forceinline__ void add(double e, double2 v) {
    x.add(e, v.x);
    y.add(e, v.y);
  }
  __device__ __forceinline__ double2 value() const { return make_double2(x.value(), y.value()); }
};
template <> struct FcAcc<ff> {
  ff2 a = ff2_make(ff(), ff());
  __device__ __forceinline__ void add(ff e, ff2 v) { a = cadd(a, cscale_l(e, v)); }
  __device__ __forceinline__ ff2 value() const { return a; }
};
template <> struct FcAcc<float> {
  ff2 a = ff2_make(ff(), ff());
  __device__ __forceinline__ void add(ff e, float2 v) {  // both components at once
    const float2 eh = dup2(e.h), p = mul2(eh, v);
    const float2 er = fma2(dup2(e.l), v, fma2(eh, v, neg2(p)));
    float2 sum, t;
    two_sum2(a.h, p, sum, t);
    a = norm2(sum, add2(t, add2(a.l, er)));
  }
  __device__ __forceinline__ float2 value() const { return add2(a.h, a.l); }
};

// The FP64 form of fc_append: one component per thread, since the compensated sums
// are the longest serial chain of a pass with few lines (20 terms of 10 FP64
// operations).  Each wall's half is summed by itself and the low half joined to
// the high one (the sum and its error), so that wide, two threads sharing a sum,
// does the same operations: rounding the joined pair does not make up for another
// order of summation.  A function of its own: inside the column pass of the large
// prime radices, which spills at 168 registers, its two sums moved the spills into
// the pass's loops (momentum pass of 32 boxes of 161^2 1863 us before, 2184 inline,
// 1842 so, with one pair of loads at a time in the fused forward).
template <typename Slot>
__device__ __noinline__ void fc_append_f64(double2* lines, int nl, int ls, int n, int C, int d,
                                           const double* __restrict__ E, Slot slot, int wide) {
  auto half_sum = [&](const double* e, const double2* L, int w, int k0) {
    auto at = [&](int m) { return reinterpret_cast<const double*>(L + slot(k0 + m))[w]; };
    Dot2 a;
    if (d > 0) a.start(e[0], at(0));
#pragma unroll 1
    for (int m = 1; m < d; ++m) a.add(e[m], at(m));
    return a;
  };
  const int sh = wide ? 1 : 0, total = (2 * nl * C) << sh;
  // whole warps go round together and tasks past the end repeat the last one:
  // every lane reaches the shuffle, whatever the compiler makes of the branches
  for (int t0 = threadIdx.x & ~31; t0 < total; t0 += blockDim.x) {
    const int t1 = t0 + (threadIdx.x & 31), t = min(t1, total - 1);
    const int half = t & sh, tt = t >> sh;
    const int w = tt & 1, p = (tt >> 1) / C, c = (tt >> 1) - p * C;
    double2* L = lines + (size_t)p * ls;
    const double* Er = E + c * 2 * d;
    Dot2 a = half_sum(half ? Er + d : Er, L, w, half ? 0 : n - d), lo;
    if (wide) {
      lo.s = __shfl_xor_sync(0xffffffffu, a.s, 1);
      lo.c = __shfl_xor_sync(0xffffffffu, a.c, 1);
    } else {
      lo = half_sum(Er + d, L, w, 0);
    }
    a.join(lo.s, lo.c);
    if (t1 < total && !half) reinterpret_cast<double*>(L + slot(n + c))[w] = a.value();
  }
}

// Appends the C continuation values of nl lines (stride ls, data in [0, n)):
// line[n + c] = sum_m E[c][m] line[n - d + m] + E[c][d + m] line[m], element k
// of a line in slot slot(k).  The (line, c) pairs are dealt to the threads.
template <typename T, typename Slot>
__device__ __forceinline__ void fc_append(typename CT<T>::t* lines, int nl, int ls, int n, int C, int d,
                                          const typename FcTab<T>::t* __restrict__ E, Slot slot, int wide = 0) {
  typedef typename CT<T>::t V;
  if constexpr (std::is_same<T, double>::value) {
    fc_append_f64(lines, nl, ls, n, C, d, E, slot, wide);
  } else {
    for (int t = threadIdx.x; t < nl * C; t += blockDim.x) {
      const int p = t / C, c = t - p * C;
      V* L = lines + (size_t)p * ls;
      const typename FcTab<T>::t* Er = E + c * 2 * d;
      FcAcc<T> a;
      for (int m = 0; m < d; ++m) {
        a.add(Er[m], L[slot(n - d + m)]);
        a.add(Er[d + m], L[slot(m)]);
      }
      L[slot(n + c)] = a.value();
    }
  }
}
struct NatSlot {
  __device__ __forceinline__ int operator()(int k) const { return k; }
};
template <typename T> struct InSlot {
  const IpPlan& P;
  __device__ __forceinline__ int operator()(int k) const { return in_slot<T>(P, k); }
};

// ---------------------------------------------------------------------------
// Half spectrum (or, dct = 1, the ny real DCT-I coefficients as (c, 0)) of
// the Pp transformed packed column pairs in R (stride ls, length n, output k
// in slot slot(k)) into spec[ky][i] of columns i0 + 2p, i0 + 2p + 1.
template <typename T, typename Slot>
__device__ __forceinline__ void col_store_spectrum(const typename CT<T>::t* R, int Pp, int ls, const GridDev& g, int i0,
                                                   int n, int dct, typename CT<T>::t* __restrict__ spec, Slot slot) {
  typedef typename CT<T>::t V;
  const int ny = g.ny;
  const int nk = dct ? ny : g.hy;
  for (int p = 0; p < Pp; ++p) {
    const int i = i0 + 2 * p;
    const V* L = R + (size_t)p * ls;
    V z_[2], zm_[2];
    batched<2>(nk, [&](int u, int k) {
      z_[u] = L[slot(k)];
      zm_[u] = L[slot(k == 0 ? 0 : n - k)];
    }, [&](int u, int k) {
      const V z = z_[u], zm = zm_[u];
      V a, b;  // columns i and i + 1
      if (dct) {
        const V h = chalf(cadd(z, zm));
        a = mk<V>(cre(h), (T)0.0);
        b = mk<V>(cim(h), (T)0.0);
      } else {
        a = chalf(cadd(z, cconj(zm)));
        b = rot<V, false>(chalf(csub(z, cconj(zm))));
      }
      V* S = spec + (size_t)k * g.ncol + i;
      if (i < g.ncol) S[0] = a;
      if (i + 1 < g.ncol) S[1] = b;
    });
  }
}
template <typename T> struct OutSlot {
  const IpPlan& P;
  __device__ __forceinline__ int operator()(int k) const { return out_slot<T>(P, k); }
};

// Forward transform of packed column pairs held in shared memory.
// lines: nf fields of Pp lines each (stride ls, field f's from line f Pp),
// line p has column i0+2p in the real and i0+2p+1 in the imaginary part for
// j < ny (element j in slot in_slot(j)).  dct = 0: FC-extend to my with table
// E ([C][2d], FP64 accumulation, FP32 pairs for FP32x2) and FFT (length my);
// dct = 1: even extension to 2(ny-1) and FFT (DCT-I, Eq. 31).  Stores the half
// spectrum (or the ny real DCT coefficients as (c, 0)) of field f into
// spec[f fstride + ky ncol + i].
template <typename T, int RM>
__device__ void col_forward_store(typename CT<T>::t* lines, typename CT<T>::t* scratch, int nf, int Pp, int ls,
                                  const GridDev& g, int i0, const typename FcTab<T>::t* __restrict__ E,
                                  const IpPlan& P, const typename CT<T>::t* __restrict__ pool, int dct,
                                  typename CT<T>::t* __restrict__ spec, size_t fstride) {
  const int ny = g.ny;
  if (!dct) {
    fc_append<T>(lines, nf * Pp, ls, ny, g.n_cont, g.n_match, E, InSlot<T>{P}, P.wide);
  } else {
    const int M = 2 * (ny - 1);
    for (int p = 0; p < nf * Pp; ++p)
      for (int jj = 1 + threadIdx.x; jj <= ny - 2; jj += blockDim.x)
        lines[(size_t)p * ls + in_slot<T>(P, M - jj)] = lines[(size_t)p * ls + in_slot<T>(P, jj)];
  }
  __syncthreads();
  fft_ip<T, RM>(lines, nf * Pp, ls, P, pool, scratch);
  for (int f = 0; f < nf; ++f)
    col_store_spectrum<T>(lines + (size_t)f * Pp * ls, Pp, ls, g, i0, P.n, dct, spec + f * fstride, OutSlot<T>{P});
}

// Gathers one half spectrum (rows ky < hy) of the column pairs into full-length
// packed lines Z_k = A_k + i B_k and Z_{n-k} = conj(A_k) + i conj(B_k); DC and
// Nyquist keep only the real parts.  put(L, k, z) stores element k.
template <typename T, typename Put>
__device__ __forceinline__ void col_gather_hermitian(typename CT<T>::t* lines, int Pp, int ls, const GridDev& g, int i0,
                                                     const typename CT<T>::t* spec, int n, Put put) {
  typedef typename CT<T>::t V;
  const int hy = g.hy;
  for (int p = 0; p < Pp; ++p) {
    const int ia = i0 + 2 * p, ib = ia + 1;
    V* L = lines + (size_t)p * ls;
    V A_[2], B_[2];
    batched<2>(hy, [&](int u, int k) {
      const V* S = spec + (size_t)k * g.ncol;
      A_[u] = B_[u] = mk<V>((T)0.0, (T)0.0);
      if (ia < g.ncol) A_[u] = ld_stream(S + ia);
      if (ib < g.ncol) B_[u] = ld_stream(S + ib);
    }, [&](int u, int k) {
      const V A = A_[u], B = B_[u];
      if (k == 0 || 2 * k == n) {
        put(L, k, mk<V>(cre(A), cre(B)));
      } else {
        put(L, k, cadd(A, rot<V, true>(B)));
        put(L, n - k, cconj(cadd(A, rot<V, false>(B))));
      }
    });
  }
}

// Packed DCT-I coefficient pairs (real parts of spec rows l < ny) into lines.
template <typename T>
__device__ void col_gather_dct(typename CT<T>::t* lines, int Pp, int ls, const GridDev& g, int i0,
                               const typename CT<T>::t* spec, const IpPlan& P) {
  typedef typename CT<T>::t V;
  const int ny = g.ny, M = 2 * (ny - 1);
  for (int p = 0; p < Pp; ++p) {
    const int ia = i0 + 2 * p, ib = ia + 1;
    V* L = lines + (size_t)p * ls;
    V z_[2];
    batched<2>(ny, [&](int u, int l) {
      const V* S = spec + (size_t)l * g.ncol;
      T a = (T)0.0, b = (T)0.0;
      if (ia < g.ncol) a = cre(ld_stream(S + ia));
      if (ib < g.ncol) b = cre(ld_stream(S + ib));
      z_[u] = mk<V>(a, b);
    }, [&](int u, int l) {
      L[in_slot<T>(P, l)] = z_[u];
      if (l >= 1 && l <= ny - 2) L[in_slot<T>(P, M - l)] = z_[u];
    });
  }
}

// ---------------------------------------------------------------------------
// Column forward: load nf real fields, FC (or DCT) + FFT, store spectra.
template <typename T, typename U, int RM>
__device__ __forceinline__ void col_fwd_body(const GridDev& g, const U* f0, const U* f1, const U* f2,
                                             const typename FcTab<T>::t* E, const IpPlan& P,
                                             const typename CT<T>::t* pool, int dct, typename CT<T>::t* spec,
                                             size_t fstride, size_t bstride, int Pp, int ls, int bx, int by, int bz) {
  typedef typename CT<T>::t V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* lines = reinterpret_cast<V*>(smem_raw);
  const int b = bz + g.b0, f = by;
  if (inactive(g, b)) return;
  const int i0 = bx * 2 * Pp;
  const U* src = f == 0 ? f0 : (f == 1 ? f1 : f2);
  const int ny = g.ny;
  for (int p = 0; p < Pp; ++p) {
    const int i = i0 + 2 * p;
    const U* c0 = src + ((size_t)b * g.ncol + i) * ny;
    const bool in0 = i < g.ncol, in1 = i + 1 < g.ncol;
    V* L = lines + (size_t)p * ls;
    U x_[4], y_[4];
    batched<4>(ny, [&](int u, int j) {
      x_[u] = in0 ? ld_stream(c0 + j) : (U)0;
      y_[u] = in1 ? ld_stream(c0 + ny + j) : (U)0;
    }, [&](int u, int j) { L[in_slot<T>(P, j)] = mk<V>(to_t<T>(x_[u]), to_t<T>(y_[u])); });
  }
  __syncthreads();
  col_forward_store<T, RM>(lines, lines + (size_t)Pp * ls, 1, Pp, ls, g, i0, E, P, pool, dct,
                       spec + b * bstride + f * fstride, fstride);
}

template <typename T, typename U, int RM>
__global__ void __launch_bounds__(kMaxThreads, MinCtas<T, RM>::v) k_col_fwd(const __grid_constant__ GridDev g, const U* __restrict__ f0, const U* __restrict__ f1, const U* __restrict__ f2,
                                                         const typename FcTab<T>::t* __restrict__ E, const __grid_constant__ IpPlan P,
                                                      const typename CT<T>::t* __restrict__ pool, int dct,
                                                      typename CT<T>::t* __restrict__ spec, size_t fstride,
                                                      size_t bstride, int Pp, int ls) {
  col_fwd_body<T, U, RM>(g, f0, f1, f2, E, P, pool, dct, spec, fstride, bstride, Pp, ls, blockIdx.x, blockIdx.y, blockIdx.z);
}

// ---------------------------------------------------------------------------
// Symbols (Eq. 16 reading): W_hat(s) = e^{-s} sum_{m<n} s^m/m!, s = |k|^2 h^2/4;
// DX = i kx W_hat, DY = i ky W_hat, DZ = i kz W_hat (each zero on its own
// axis' Nyquist plane), LAP = -|k|^2 W_hat, W = W_hat (kz = 0 in 2D).
// Products and sums of the wavenumbers use round-to-nearest intrinsics, which the compiler never
// contracts into FMAs: every CTA width then evaluates the same expression.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float div_rn(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double div_rn(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ ff mul_rn(ff a, ff b) { return a * b; }
__device__ __forceinline__ ff add_rn(ff a, ff b) { return a + b; }
__device__ __forceinline__ ff div_rn(ff a, ff b) { return a / b; }

// A symbol is real or purely imaginary: s or (imag) i s.
template <typename T>
__device__ __forceinline__ T symbol(int op, T kx, T ky, T kz, T kyy, T kzz, bool d3, bool nyq_x, bool nyq_y, bool nyq_z,
                                    T What, bool& imag) {
  imag = op == SYM_DX || op == SYM_DY || op == SYM_DZ;
  switch (op) {
    case SYM_W: return What;
    case SYM_DX: return nyq_x ? (T)0.0 : mul_rn(kx, What);
    case SYM_DY: return nyq_y ? (T)0.0 : mul_rn(ky, What);
    case SYM_DZ: return nyq_z ? (T)0.0 : mul_rn(kz, What);
    case SYM_LAP: {
      T k2 = add_rn(mul_rn(kx, kx), kyy);
      if (d3) k2 = add_rn(k2, kzz);
      return -mul_rn(k2, What);
    }
    case SYM_ONE: return (T)1.0;
    default: {  // projection terms: g = (i kx W_hat, i ky W_hat) up to the common factor i W_hat
      const T gx = nyq_x ? (T)0.0 : kx, gy = nyq_y ? (T)0.0 : ky;
      const T g2 = add_rn(mul_rn(gx, gx), mul_rn(gy, gy));
      if (!(static_cast<float>(g2) > 0.f)) return (T)0.0;
      const T num = op == SYM_NPXX ? mul_rn(gx, gx) : op == SYM_NPXY ? mul_rn(gx, gy) : mul_rn(gy, gy);
      return -div_rn(num, g2);
    }
  }
}
// s x or i s x, rounded as a product (never contracted with a later sum: the
// same result at every CTA width)
template <typename V, typename T> __device__ __forceinline__ V sym_mul(T s, bool imag, V x) {
  if (imag) x = rot<V, true>(x);
  if constexpr (std::is_same<T, ff>::value) return cscale_l(s, x);
  else return mk<V>(mul_rn(s, x.x), mul_rn(s, x.y));
}
template <typename V> __device__ __forceinline__ V cadd_rn(V a, V b) {
  if constexpr (std::is_same<V, ff2>::value) return cadd(a, b);
  else return mk<V>(add_rn(a.x, b.x), add_rn(a.y, b.y));
}

// sum_{m<n} s^m / m! (n = family) in Horner form with constant coefficients:
// W_hat = e^{-s} times this.
template <typename T> __device__ __forceinline__ T kernel_poly(int family, T s) {
  const T one = (T)1.0;
  switch (family) {
    case 1: return one;
    case 2: return one + s;
    case 3: return one + s * (one + s * (T)0.5);
    case 4: return one + s * (one + s * ((T)0.5 + s * (T)(1.0 / 6.0)));
    default: return one + s * (one + s * ((T)0.5 + s * ((T)(1.0 / 6.0) + s * (T)(1.0 / 24.0))));
  }
}

// Row (x) pass over the x lines of the y half-spectra: line q of an instance
// is the ky = q / nz row at z index kq = q % nz (3D: the spectra are already
// transformed in z; 2D: nz = 1, line q = row ky), its nx elements at stride
// nz.  For Rr lines of one instance: load nin input lines, FC-extend in x
// (walled x), FFT (length mx); then, `ob` outputs at a time, form
// sum_t S_t * F_t times `scale`, inverse FFT, truncate to nx and store.
// The symbols S_t are W_hat (Wt: the context's [hy nz][mx] table of Eq. 16 in
// the transform type) times 1, i kx, i ky, i kz or -|k|^2.
// Shared memory: the nin Rr input lines (their spectra after the transform)
// and `ob` Rr lines, in which ob outputs at a time are formed and inverted
// together (more butterflies per stage to deal to the lanes), plus the scratch
// line of a plan with a large prime radix.
template <typename T, int RM>
__device__ __forceinline__ void row_sym_body(const GridDev& g, const typename CT<T>::t* sp_in, typename CT<T>::t* sp_out,
                                             size_t fstride_in, size_t bstride_in, size_t fstride_out,
                                             size_t bstride_out, const RowOps& ops, const typename FcTab<T>::t* E,
                                             const IpPlan& P, const typename CT<T>::t* pool, const T* Wt,
                                             double scale, int Rr, int ob, int ls, int bx, int by, int fz) {
  typedef typename CT<T>::t V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // split: this CTA takes input field fz and the outputs formed from it alone
  const int nin = ops.split > 1 ? 1 : ops.nin;
  const int f0 = ops.split > 1 ? fz : 0;
  const int o_begin = ops.split > 1 ? fz * (ops.nout / ops.split) : 0;
  const int nout = ops.split > 1 ? o_begin + ops.nout / ops.split : ops.nout;
  V* X = reinterpret_cast<V*>(smem_raw);
  V* C = X + (size_t)nin * Rr * ls;
  V* scratch = C + (size_t)ob * Rr * ls;
  const int b = by + g.b0;
  if (inactive(g, b)) return;
  const int q0 = bx * Rr;
  const int nx = g.nx, mx = g.mx, nz = g.nz;
  const int nq = g.hy * nz;
  for (int f = 0; f < nin; ++f)
    for (int r = 0; r < Rr; ++r) {
      const int q = q0 + r;
      V* L = X + ((size_t)f * Rr + r) * ls;
      const V* S = sp_in + b * bstride_in + (f0 + f) * fstride_in + (size_t)(q / nz) * g.ncol + (q % nz);
      V x_[4];
      batched<4>(nx, [&](int u, int i) { x_[u] = q < nq ? ld_stream(S + (size_t)i * nz) : mk<V>((T)0.0, (T)0.0); },
                 [&](int u, int i) { L[in_slot<T>(P, i)] = x_[u]; });
    }
  __syncthreads();
  if (g.x_walls) {
    fc_append<T>(X, nin * Rr, ls, nx, g.n_cont, g.n_match, E, InSlot<T>{P}, P.wide);
    __syncthreads();
  }
  fft_ip<T, RM>(X, nin * Rr, ls, P, pool, scratch);
  const T ckx = (T)g.ckx_d, cky = (T)g.cky_d, ckz = (T)g.ckz_d;  // 2 pi / (mx dx), 2 pi / (my dy), 2 pi / (nz dz)
  const T tscale = (T)scale;
  for (int o0 = o_begin; o0 < nout; o0 += ob) {
    const int on = min(ob, nout - o0);
    for (int r = 0; r < Rr; ++r) {
      const int q = q0 + r < nq ? q0 + r : 0;
      const int ky = q / nz, kq = q - (q / nz) * nz;
      const int kzeta = (2 * kq <= nz) ? kq : kq - nz;
      const T kyw = mul_rn(cky, (T)ky), kz = mul_rn(ckz, (T)kzeta);
      const T kyy = mul_rn(kyw, kyw), kzz = mul_rn(kz, kz);
      const bool nyq_y = (g.my % 2 == 0) && (2 * ky == g.my);
      const bool nyq_z = (nz % 2 == 0) && (2 * kq == nz);
      // W_hat of row q from the context's table (Eq. 16, built once on the host)
      const T* Wq = Wt + (size_t)q * mx;
      T What_[2];
      int so_[2], si_[2];
      batched<2>(mx, [&](int u, int kxi) {
        What_[u] = Wq[kxi];
        so_[u] = out_slot<T>(P, kxi);
        si_[u] = in_slot<T>(P, kxi);
      }, [&](int u, int kxi) {
        const int kappa = (2 * kxi <= mx) ? kxi : kxi - mx;
        const T kx = mul_rn(ckx, (T)kappa);
        const bool nyq_x = (mx % 2 == 0) && (2 * kxi == mx);
        for (int oo = 0; oo < on; ++oo) {
          const int o = o0 + oo;
          V acc;
          for (int t = 0; t < ops.nterm[o]; ++t) {
            bool imag;
            const T sy = symbol<T>(ops.op[o][t], kx, kyw, kz, kyy, kzz, nz > 1, nyq_x, nyq_y, nyq_z, What_[u], imag);
            const V m = sym_mul(sy, imag, X[((size_t)(ops.field[o][t] - f0) * Rr + r) * ls + so_[u]]);
            acc = t == 0 ? m : cadd_rn(acc, m);
          }
          C[((size_t)oo * Rr + r) * ls + si_[u]] = cconj(cscale(acc, tscale));
        }
      });
    }
    __syncthreads();
    fft_ip<T, RM>(C, on * Rr, ls, P, pool, scratch);
    for (int oo = 0; oo < on; ++oo)
      for (int r = 0; r < Rr; ++r) {
        const int q = q0 + r;
        if (q >= nq) break;
        V* S = sp_out + b * bstride_out + (o0 + oo) * fstride_out + (size_t)(q / nz) * g.ncol + (q % nz);
        const V* Yl = C + ((size_t)oo * Rr + r) * ls;
        V y_[4];
        batched<4>(nx, [&](int u, int i) { y_[u] = Yl[out_slot<T>(P, i)]; },
                   [&](int u, int i) { S[(size_t)i * nz] = cconj(y_[u]); });
      }
    __syncthreads();
  }
}

template <typename T, int RM>
__global__ void __launch_bounds__(kMaxThreads, MinCtas<T, RM>::v) k_row_sym(const __grid_constant__ GridDev g, const typename CT<T>::t* __restrict__ sp_in,
                                                         typename CT<T>::t* __restrict__ sp_out, size_t fstride_in,
                                                         size_t bstride_in, size_t fstride_out, size_t bstride_out,
                                                         const __grid_constant__ RowOps ops,
                                                         const typename FcTab<T>::t* __restrict__ E,
                                                         const __grid_constant__ IpPlan P, const typename CT<T>::t* __restrict__ pool,
                                                         const T* __restrict__ Wt, double scale, int Rr, int ob, int ls) {
  row_sym_body<T, RM>(g, sp_in, sp_out, fstride_in, bstride_in, fstride_out, bstride_out, ops, E, P, pool, Wt, scale, Rr,
                  ob, ls, blockIdx.x, blockIdx.y, blockIdx.z);
}

// Per-lane constants of the register row pass for one row: lane k1 owns the
// frequencies kxi = k1 + M k2 (k2 < 32) of row q (Wq: its W_hat row).
struct WRowSym {
  float ckx, kyw, kz;
  bool nyq_y, nyq_z;
  int mx, k1;
  const float* Wq;
  float kx0, wrap;  // ckx k1 and ckx mx: kx = kx0 + ckx M k2 (- wrap past mx/2), no int-to-float per element
};

// v[k2] += symbol OP (kx of k1 + M k2) x spectrum value ([k2][lane] at xr, xi).
template <int OP, int M>
__device__ __forceinline__ void w_accumulate(float2* v, const float* xr, const float* xi, const WRowSym& r) {
#pragma unroll
  for (int k2 = 0; k2 < 32; ++k2) {
    const int kxi = r.k1 + M * k2;
    const float kxu = fmaf(r.ckx, (float)(M * k2), r.kx0);  // M k2 is a compile-time constant
    const float kx = (2 * kxi <= r.mx) ? kxu : kxu - r.wrap;
    const bool nyq_x = (r.mx % 2 == 0) && (2 * kxi == r.mx);
    const float What = (OP == SYM_ONE || OP == SYM_NPXX || OP == SYM_NPXY || OP == SYM_NPYY) ? 1.f : r.Wq[kxi];
    bool imag;
    const float sy = symbol<float>(OP, kx, r.kyw, r.kz, mul_rn(r.kyw, r.kyw), mul_rn(r.kz, r.kz), true, nyq_x, r.nyq_y,
                                   r.nyq_z, What, imag);
    const float2 x = make_float2(xr[k2 * 32], xi[k2 * 32]);
    if (OP == SYM_DX || OP == SYM_DY || OP == SYM_DZ) {  // purely imaginary symbol i sy
      v[k2].x = add_rn(v[k2].x, -mul_rn(sy, x.y));
      v[k2].y = add_rn(v[k2].y, mul_rn(sy, x.x));
    } else {  // real symbol
      v[k2].x = add_rn(v[k2].x, mul_rn(sy, x.x));
      v[k2].y = add_rn(v[k2].y, mul_rn(sy, x.y));
    }
  }
}

// Row pass of FP32 contexts with periodic x lines of mx = nx = 32 M points
// (M = 2 .. 32): the same operation as k_row_sym, with the register FFT of
// fcsph_warpfft.cuh.  One warp carries 32 / M rows through every transform;
// a CTA holds 4 warps.  The forward spectra of the nin inputs wait in shared
// memory ([field][k2][lane] of this warp, conflict-free) while the outputs are
// formed one at a time, each in the registers of the lane that owns its
// frequencies kx = k1 + M k2 (lane = l M + k1).
template <int M>
__global__ void __launch_bounds__(128, 3) k_row_sym_w(GridDev g, const float2* __restrict__ sp_in,
                                                      float2* __restrict__ sp_out, size_t fstride_in,
                                                      size_t bstride_in, size_t fstride_out, size_t bstride_out,
                                                      const __grid_constant__ RowOps ops,
                                                      const float2* __restrict__ tw,
                                                      const float* __restrict__ Wt, double scale) {
  constexpr int LPW = 32 / M;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nin = ops.nin, nout = ops.nout;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* xs = reinterpret_cast<float*>(smem_raw) + (size_t)warp * (kWarpXchgFloats + nin * 2 * 32 * 32);
  float* spre = xs + kWarpXchgFloats;
  float* spim = spre + nin * 32 * 32;
  const int b = blockIdx.y + g.b0;
  if (inactive(g, b)) return;
  const int mx = g.mx, nz = g.nz;
  const int nq = g.hy * nz;
  const int q0 = (blockIdx.x * 4 + warp) * LPW;
  if (q0 >= nq) return;  // whole warp beyond the last row (uniform)
  for (int f = 0; f < nin; ++f) {
    float2 v[32];
#pragma unroll
    for (int l = 0; l < LPW; ++l) {
      const int q = q0 + l;
      const float2* S = sp_in + b * bstride_in + f * fstride_in + (size_t)(q / nz) * g.ncol + (q % nz);
#pragma unroll
      for (int j = 0; j < M; ++j) v[l * M + j] = q < nq ? S[(size_t)(lane + 32 * j) * nz] : make_float2(0.f, 0.f);
    }
    warp_fft_fwd<M>(v, xs, tw, lane);
#pragma unroll
    for (int k2 = 0; k2 < 32; ++k2) {
      spre[(f * 32 + k2) * 32 + lane] = v[k2].x;
      spim[(f * 32 + k2) * 32 + lane] = v[k2].y;
    }
  }
  __syncwarp();
  const int l = lane / M, k1 = lane - (lane / M) * M;
  const int q = q0 + l < nq ? q0 + l : q0;
  const float ckx = g.ckx_f, cky = g.cky_f, ckz = g.ckz_f;
  const int ky = q / nz, kq = q - (q / nz) * nz;
  const int kzeta = (2 * kq <= nz) ? kq : kq - nz;
  const float kyw = cky * (float)ky, kz = ckz * (float)kzeta;
  const bool nyq_y = (g.my % 2 == 0) && (2 * ky == g.my);
  const bool nyq_z = (nz % 2 == 0) && (2 * kq == nz);
  const float* Wq = Wt + (size_t)q * mx;
  const float tscale = (float)scale;
  const WRowSym rs{ckx, kyw, kz, nyq_y, nyq_z, mx, k1, Wq, ckx * (float)k1, ckx * (float)mx};
  for (int o = 0; o < nout; ++o) {
    float2 v[32];
#pragma unroll
    for (int k2 = 0; k2 < 32; ++k2) v[k2] = make_float2(0.f, 0.f);
    for (int t = 0; t < ops.nterm[o]; ++t) {
      const float* xr = spre + ops.field[o][t] * 32 * 32 + lane;
      const float* xi = spim + ops.field[o][t] * 32 * 32 + lane;
      switch (ops.op[o][t]) {  // uniform over the warp: one unrolled loop per symbol
        case SYM_W: w_accumulate<SYM_W, M>(v, xr, xi, rs); break;
        case SYM_DX: w_accumulate<SYM_DX, M>(v, xr, xi, rs); break;
        case SYM_DY: w_accumulate<SYM_DY, M>(v, xr, xi, rs); break;
        case SYM_LAP: w_accumulate<SYM_LAP, M>(v, xr, xi, rs); break;
        case SYM_DZ: w_accumulate<SYM_DZ, M>(v, xr, xi, rs); break;
        case SYM_ONE: w_accumulate<SYM_ONE, M>(v, xr, xi, rs); break;
        case SYM_NPXX: w_accumulate<SYM_NPXX, M>(v, xr, xi, rs); break;
        case SYM_NPXY: w_accumulate<SYM_NPXY, M>(v, xr, xi, rs); break;
        default: w_accumulate<SYM_NPYY, M>(v, xr, xi, rs); break;
      }
    }
#pragma unroll
    for (int k2 = 0; k2 < 32; ++k2) v[k2] = cscale(v[k2], tscale);
    warp_fft_inv<M>(v, xs, tw, lane);
#pragma unroll
    for (int l2 = 0; l2 < LPW; ++l2) {
      const int qq = q0 + l2;
      if (qq < nq) {
        float2* S = sp_out + b * bstride_out + o * fstride_out + (size_t)(qq / nz) * g.ncol + (qq % nz);
#pragma unroll
        for (int j = 0; j < M; ++j) S[(size_t)(lane + 32 * j) * nz] = v[l2 * M + j];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Line operator: every column of [batch][nx][ny] is an independent
// wall-normal line.  Per column pair (packed as one complex line): FC-extend
// (table E), FFT (length my); then for each output the symbol at kx = 0 --
// W_hat(ky), i ky W_hat (zero on the Nyquist mode), -ky^2 W_hat, and 0 for
// d/dx -- times the spectrum, inverse FFT, truncation to ny, scale 1/my.  The
// symbols are Hermitian in ky, so the real and imaginary parts of the packed
// result are the two columns' outputs.  One kernel per call.
struct LineOuts {
  int nout;
  int op[4];
  void* out[4];
};

template <typename T, typename U, int RM>
__global__ void __launch_bounds__(kMaxThreads, LineMinCtas<T, RM>::v) k_line_op(const __grid_constant__ GridDev g, const U* __restrict__ f,
                                                                      long long ncols,
                                                                      const typename FcTab<T>::t* __restrict__ E,
                                                                      const __grid_constant__ IpPlan P,
                                                                      const typename CT<T>::t* __restrict__ pool,
                                                                      const __grid_constant__ LineOuts lo, int Pp,
                                                                      int ob, int ls) {
  typedef typename CT<T>::t V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* X = reinterpret_cast<V*>(smem_raw);
  V* C = X + (size_t)Pp * ls;
  V* scratch = C + (size_t)ob * Pp * ls;
  const long long c0 = (long long)blockIdx.x * 2 * Pp;
  const int ny = g.ny, my = g.my;
  for (int p = 0; p < Pp; ++p) {
    const long long cc = c0 + 2 * p;
    for (int j = threadIdx.x; j < ny; j += blockDim.x)
      X[(size_t)p * ls + in_slot<T>(P, j)] =
          mk<V>(cc < ncols ? to_t<T>(f[cc * ny + j]) : (T)0.0, cc + 1 < ncols ? to_t<T>(f[(cc + 1) * ny + j]) : (T)0.0);
  }
  __syncthreads();
  fc_append<T>(X, Pp, ls, ny, g.n_cont, g.n_match, E, InSlot<T>{P}, P.wide);
  __syncthreads();
  fft_ip<T, RM>(X, Pp, ls, P, pool, scratch);
  const T hh = (T)g.hh_d, cky = (T)g.cky_d;  // h^2 / 4, 2 pi / (my dy)
  const T tscale = (T)(1.0 / my);
  for (int o0 = 0; o0 < lo.nout; o0 += ob) {
    const int on = min(ob, lo.nout - o0);
    for (int p = 0; p < Pp; ++p)
    for (int k = threadIdx.x; k < my; k += blockDim.x) {
      const int kappa = (2 * k <= my) ? k : k - my;
      const T ky = cky * (T)kappa;
      const T What = cre(pool[g.ey_off + (kappa < 0 ? -kappa : kappa)]) * kernel_poly<T>(g.family, ky * ky * hh);
      const bool nyq = (my % 2 == 0) && (2 * k == my);
      const V x = X[(size_t)p * ls + out_slot<T>(P, k)];
      const int si = in_slot<T>(P, k);
      for (int oo = 0; oo < on; ++oo) {
        const int op = lo.op[o0 + oo];
        const T sy = op == SYM_W ? What : op == SYM_DY ? (nyq ? (T)0.0 : ky * What)
                                         : op == SYM_LAP ? -(ky * ky) * What : (T)0.0;
        C[((size_t)oo * Pp + p) * ls + si] = cconj(cscale(sym_mul(sy, op == SYM_DY, x), tscale));
      }
    }
    __syncthreads();
    fft_ip<T, RM>(C, on * Pp, ls, P, pool, scratch);
    for (int oo = 0; oo < on; ++oo) {
      U* out = reinterpret_cast<U*>(lo.out[o0 + oo]);
      for (int p = 0; p < Pp; ++p) {
        const long long cc = c0 + 2 * p;
        if (cc >= ncols) break;
        const V* Yl = C + ((size_t)oo * Pp + p) * ls;
        for (int j = threadIdx.x; j < ny; j += blockDim.x) {
          const V y = cconj(Yl[out_slot<T>(P, j)]);
          out[cc * ny + j] = (U)cre(y);
          if (cc + 1 < ncols) out[(cc + 1) * ny + j] = (U)cim(y);
        }
      }
    }
    __syncthreads();
  }
}

// Two adjacent FP32 columns (c0 = src[0..ny), c1 = src[ny..2 ny); c1 absent:
// zeros) packed into the complex line L[j] = (c0[j], c1[j]).  With ny a
// multiple of 4 and a 16-byte aligned start every thread issues its float4
// loads of both columns back to back; otherwise plain loads.
__device__ __forceinline__ void load_pair_f32(float2* L, const float* __restrict__ src, bool has1, int ny) {
  const int t = threadIdx.x, nt = blockDim.x;
  if ((ny & 3) == 0 && ((reinterpret_cast<uintptr_t>(src) & 15) == 0)) {
    const float4* c0 = reinterpret_cast<const float4*>(src);
    const float4* c1 = reinterpret_cast<const float4*>(src + ny);
    for (int m = t; m < ny / 4; m += nt) {
      const float4 a = c0[m];
      const float4 b = has1 ? c1[m] : make_float4(0.f, 0.f, 0.f, 0.f);
      float4* d = reinterpret_cast<float4*>(L + 4 * m);
      d[0] = make_float4(a.x, b.x, a.y, b.y);
      d[1] = make_float4(a.z, b.z, a.w, b.w);
    }
  } else {
    for (int j = t; j < ny; j += nt) L[j] = make_float2(src[j], has1 ? src[ny + j] : 0.f);
  }
}

// A thread's team of a packed CTA (line p < NP, place t < NV; idle threads: t >=
// NV, on line 0).
template <int NV, int NP> __device__ __forceinline__ void team_of(int& p, int& t) {
  if constexpr (NP == 1) {
    p = 0;
    t = threadIdx.x;
  } else {
    p = threadIdx.x / NV;
    t = threadIdx.x - p * NV;
    if (p >= NP) {
      p = 0;
      t = NV;
    }
  }
}

// Half spectra of the NP pairs' transformed lines (stride ls, length n) into
// spec[ky][i]; the pairs of one row ky are neighbouring lanes, whose 16-byte
// values are contiguous in memory.
template <int NP>
__device__ __forceinline__ void team_store_spectrum(const float2* L0, int ls, const GridDev& g, int i0, int n,
                                                    float2* __restrict__ spec) {
  for (int e = threadIdx.x; e < g.hy * NP; e += blockDim.x) {
    const int k = e / NP, p = e - k * NP, i = i0 + 2 * p;
    const float2* L = L0 + (size_t)p * ls;
    const float2 z = L[k], zm = L[k == 0 ? 0 : n - k];
    const float2 a = chalf(cadd(z, cconj(zm))), b = rot<float2, false>(chalf(csub(z, cconj(zm))));
    float2* S = spec + (size_t)k * g.ncol + i;
    if (i < g.ncol) S[0] = a;
    if (i + 1 < g.ncol) S[1] = b;
  }
}

// The Hermitian lines of NP pairs from one half spectrum, lanes as above.
template <int NP>
__device__ __forceinline__ void team_gather(float2* L0, int ls, const GridDev& g, int i0, int n,
                                            const float2* __restrict__ spec) {
  for (int e = threadIdx.x; e < g.hy * NP; e += blockDim.x) {
    const int k = e / NP, p = e - k * NP, i = i0 + 2 * p;
    const float2* S = spec + (size_t)k * g.ncol + i;
    float2* L = L0 + (size_t)p * ls;
    float2 A = make_float2(0.f, 0.f), B = A;
    if (i < g.ncol) A = ld_stream(S);
    if (i + 1 < g.ncol) B = ld_stream(S + 1);
    if (k == 0 || 2 * k == n) {
      L[k] = make_float2(A.x, B.x);
    } else {
      L[k] = cadd(A, rot<float2, true>(B));
      L[n - k] = cconj(cadd(A, rot<float2, false>(B)));
    }
  }
}

// The line operator of FP32 contexts with the register team FFT
// (fcsph_regfft.cuh) for extended lengths n = N1 N2: NP column pairs per CTA;
// the forward spectrum waits in shared memory, each value where the thread
// that owns its frequency (k = t + N1 k2) reads it back, while the outputs are
// formed one at a time.
template <int N1, int N2, int NP>
__global__ void __launch_bounds__(TeamFFT<N1, N2>::threads(NP), TeamFFT<N1, N2>::min_ctas(NP)) k_line_op_r(
    GridDev g, const float* __restrict__ f, long long ncols, const typename FcTab<float>::t* __restrict__ E,
    const float2* __restrict__ pool, const float2* __restrict__ tw, const __grid_constant__ LineOuts lo) {
  typedef TeamFFT<N1, N2> TF;
  constexpr int n = N1 * N2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int p, t;
  team_of<TF::NV, NP>(p, t);
  float2* L0 = reinterpret_cast<float2*>(smem_raw);
  float2* L = L0 + p * n;
  float2* xs = L0 + NP * n + p * TF::XCHG;
  const long long cb = (long long)blockIdx.x * 2 * NP, c0 = cb + 2 * p;
  const int ny = g.ny;
  for (int q = 0; q < NP; ++q)
    if (cb + 2 * q < ncols) load_pair_f32(L0 + q * n, f + (cb + 2 * q) * ny, cb + 2 * q + 1 < ncols, ny);
  __syncthreads();
  fc_append<float>(L0, NP, n, ny, g.n_cont, g.n_match, E, NatSlot());
  __syncthreads();
  float2 x[TF::NV];
  if (t < N2) {
#pragma unroll
    for (int j = 0; j < N1; ++j) x[j] = L[t + N2 * j];
  }
  TF::template fwd<false>(x, xs, tw, t);
  if (t < N1) {
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) L[t + N1 * k2] = x[k2];
  }
  const float hh = g.hh_f, cky = g.cky_f, tscale = g.inv_my_f;  // n = my
  const float ky0 = cky * (float)t;
  for (int o = 0; o < lo.nout; ++o) {
    const int op = lo.op[o];
    float2 y[TF::NV];
    if (t < N1) {
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) {
        const int k = t + N1 * k2;
        const int kappa = (2 * k <= n) ? k : k - n;
        const float kyu = fmaf(cky, (float)(N1 * k2), ky0);  // N1 k2 is a compile-time constant
        const float ky = (2 * k <= n) ? kyu : kyu - cky * (float)n;
        const float What = pool[g.ey_off + (kappa < 0 ? -kappa : kappa)].x * kernel_poly<float>(g.family, ky * ky * hh);
        const bool nyq = (n % 2 == 0) && (2 * k == n);
        float2 sy;
        if (op == SYM_W)
          sy = make_float2(What, 0.f);
        else if (op == SYM_DY)
          sy = make_float2(0.f, nyq ? 0.f : ky * What);
        else if (op == SYM_LAP)
          sy = make_float2(-(ky * ky) * What, 0.f);
        else
          sy = make_float2(0.f, 0.f);
        y[k2] = cscale(cmul(sy, L[k]), tscale);
      }
    }
    TF::template inv<false>(y, xs, tw, t);
    if (t < N2) {
      float* out = reinterpret_cast<float*>(lo.out[o]);
#pragma unroll
      for (int j = 0; j < N1; ++j) {
        const int row = t + N2 * j;
        if (row < ny) {
          if (c0 < ncols) out[c0 * ny + row] = y[j].x;
          if (c0 + 1 < ncols) out[(c0 + 1) * ny + row] = y[j].y;
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// z pass of the 3D channel: in the spectra [b][field][row][x][z] every run of
// nz values (fixed b, field, row, x) is one periodic z line; L lines per CTA
// are transformed in place, forward or (inv) unnormalised inverse.  Instances
// with active[b] == 0 (isph_step's mask, when given) are left alone.
template <typename T, int RM>
__global__ void __launch_bounds__(kMaxThreads, MinCtas<T, RM>::v) k_zlines(typename CT<T>::t* __restrict__ spec,
                                                                      int lines_per_field, size_t fstride,
                                                                      size_t bstride, const __grid_constant__ IpPlan P,
                                                                      const typename CT<T>::t* __restrict__ pool, int L,
                                                                      int ls, int inv, const unsigned char* active,
                                                                      int b0) {
  typedef typename CT<T>::t V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int b = blockIdx.z + b0;
  if (active && !active[b]) return;
  V* A = reinterpret_cast<V*>(smem_raw);
  const int n = P.n;
  V* base = spec + b * bstride + blockIdx.y * fstride;
  const int l0 = blockIdx.x * L;
  const int nl = min(L, lines_per_field - l0);
  for (int r = 0; r < nl; ++r) {
    const V* S = base + (size_t)(l0 + r) * n;
    V x_[4];
    batched<4>(n, [&](int u, int j) { x_[u] = ld_stream(S + j); },
               [&](int u, int j) { A[(size_t)r * ls + in_slot<T>(P, j)] = inv ? cconj(x_[u]) : x_[u]; });
  }
  __syncthreads();
  fft_ip<T, RM>(A, nl, ls, P, pool, A + (size_t)L * ls);
  for (int r = 0; r < nl; ++r) {
    V* S = base + (size_t)(l0 + r) * n;
    V y_[4];
    batched<4>(n, [&](int u, int j) { y_[u] = A[(size_t)r * ls + out_slot<T>(P, j)]; },
               [&](int u, int j) { S[j] = inv ? cconj(y_[u]) : y_[u]; });
  }
}

// ---------------------------------------------------------------------------
// PPE row pass (Eqs. 31-33): rows l < ny hold DCT-I-in-y coefficients.  x
// periodic: FFT (length nx); walled x: DCT-I via FFT of the even extension
// (length 2(nx-1)).  Multiply by -1/(lam_k^2 + lam_l^2) (apply = 0, (0,0) -> 0),
// or by -(lam_k^2 + lam_l^2) (apply = 1), times the inverse-transform scales,
// transform back, store.  3D: line q is the l = q / nz row at z index
// kq = q % nz of the DFT-z-transformed coefficients, elements at stride nz,
// and lam_z^2 joins the denominator.
template <typename T, int RM>
__device__ __forceinline__ void row_ppe_body(const GridDev& g, typename CT<T>::t* spec, size_t bstride, const IpPlan& P,
                                             const typename CT<T>::t* pool, int apply, int Rr, int ls, int bx, int by) {
  typedef typename CT<T>::t V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* X = reinterpret_cast<V*>(smem_raw);
  V* O = X + (size_t)Rr * ls;
  V* scratch = O + (size_t)Rr * ls;
  const int b = by + g.b0;
  if (inactive(g, b)) return;
  const int q0 = bx * Rr;
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int nq = ny * nz;
  const int n = P.n;  // nx or 2(nx-1)
  for (int r = 0; r < Rr; ++r) {
    const int q = q0 + r;
    V* L = X + (size_t)r * ls;
    const V* S = spec + b * bstride + (size_t)(q / nz) * g.ncol + (q % nz);
    V x_[4];
    batched<4>(nx, [&](int u, int i) { x_[u] = q < nq ? ld_stream(S + (size_t)i * nz) : mk<V>((T)0.0, (T)0.0); }, [&](int u, int i) {
      L[in_slot<T>(P, i)] = x_[u];
      if (g.x_walls && i >= 1 && i <= nx - 2) L[in_slot<T>(P, n - i)] = x_[u];
    });
  }
  __syncthreads();
  fft_ip<T, RM>(X, Rr, ls, P, pool, scratch);
  const T norm = (T)(1.0 / ((double)n * 2.0 * (ny - 1) * nz));
  const int nk = g.x_walls ? nx : n;
  for (int r = 0; r < Rr; ++r) {
    const int q = q0 + r < nq ? q0 + r : 0;
    const int l = q / nz, kq = q - (q / nz) * nz;
    // lam_l^2 (+ lam_z^2) from the per-axis tables (Eq. 33 eigenvalues)
    const T dyz = cre(pool[g.ly2_off + l]) + cre(pool[g.lz2_off + kq]);
    const bool zero_yz = l == 0 && kq == 0;
    T lx_[2];
    V x_[2];
    batched<2>(nk, [&](int u, int k) {
      lx_[u] = cre(pool[g.lx2_off + k]);
      x_[u] = X[(size_t)r * ls + out_slot<T>(P, k)];
    }, [&](int u, int k) {
      const T den = lx_[u] + dyz;
      T f;
      if (apply == 1)
        f = -(den * norm);
      else
        f = (k == 0 && zero_yz) ? (T)0.0 : -(norm / den);
      const V y = cscale(x_[u], f);
      if (g.x_walls) {  // DCT-I is its own inverse up to the folded scale
        O[(size_t)r * ls + in_slot<T>(P, k)] = y;
        if (k >= 1 && k <= nx - 2) O[(size_t)r * ls + in_slot<T>(P, n - k)] = y;
      } else {
        O[(size_t)r * ls + in_slot<T>(P, k)] = cconj(y);
      }
    });
  }
  __syncthreads();
  fft_ip<T, RM>(O, Rr, ls, P, pool, scratch);
  for (int r = 0; r < Rr; ++r) {
    const int q = q0 + r;
    if (q >= nq) break;
    V* S = spec + b * bstride + (size_t)(q / nz) * g.ncol + (q % nz);
    const V* Yl = O + (size_t)r * ls;
    V y_[4];
    batched<4>(nx, [&](int u, int i) { y_[u] = Yl[out_slot<T>(P, i)]; },
               [&](int u, int i) { S[(size_t)i * nz] = g.x_walls ? y_[u] : cconj(y_[u]); });
  }
}

template <typename T, int RM>
__global__ void __launch_bounds__(kMaxThreads, MinCtas<T, RM>::v) k_row_ppe(const __grid_constant__ GridDev g, typename CT<T>::t* __restrict__ spec,
                                                      size_t bstride, const __grid_constant__ IpPlan P,
                                                      const typename CT<T>::t* __restrict__ pool, int apply, int Rr,
                                                      int ls) {
  row_ppe_body<T, RM>(g, spec, bstride, P, pool, apply, Rr, ls, blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Column inverse with epilogues.
enum { EPI_OUT = 0, EPI_MOM = 1, EPI_DIV = 2, EPI_CORR = 3, EPI_PPE_SOLVE = 4, EPI_PPE_RESID = 5, EPI_PPE_ADD = 6 };

struct EpiArgs {
  // EPI_OUT
  void* outs[6];
  int out_double;
  // step state (double), per velocity component (2D: u, v; 3D: u, v, w)
  const double* vel[3];   // MOM: velocity at the start of the substep
  double* Fp[3];          // MOM: F^{k-1} in, F^k out
  double* vs[3];          // MOM: u* out; CORR: u* in
  double* vo[3];          // CORR: corrected velocity out
  int mom_terms;          // MOM: outputs per component (d/dx, d/dy, [d/dz], lap)
  double* bvec;       // DIV: out b; PPE_RESID: in b
  double* phi;        // PPE_*: out phi / residual / accumulate
  void* phi_any;      // PPE_SOLVE in the context's I/O type when not double
  int phi_double;
  StepDev s;
  // fused forward: nf fields, table, plan, output spectra, dct
  int fwd_nf;
  int fwd_dct;
  const void* fwdE;   // FC table in the transform's FcTab type
  IpPlan fwdP;
  void* fwd_spec;
  size_t fwd_fstride, fwd_bstride;
  int* status;
};

// L2 prefetch hints for the column pass.  Only addresses the kernel reads
// later are named, so every one lies inside its buffer.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Rows k < hy of one field's half-spectrum at the CTA's column pairs.
template <typename V>
__device__ void prefetch_spec_pairs(const GridDev& g, int i0, int Pp, const V* spec) {
  for (int t = threadIdx.x; t < g.hy * Pp; t += blockDim.x) {
    const int k = t / Pp, p = t - k * Pp;
    if (i0 + 2 * p < g.ncol) prefetch_l2(spec + (size_t)k * g.ncol + i0 + 2 * p);
  }
}

// The CTA's columns of one FP64 field of instance b, 128-byte lines.
__device__ void prefetch_field_cols(const GridDev& g, int b, int i0, int Pp, const double* f) {
  const int per = (g.ny + 15) / 16 + 1;  // lines of one column, one more for an unaligned start
  const int nc = min(2 * Pp, g.ncol - i0);
  for (int t = threadIdx.x; t < nc * per; t += blockDim.x) {
    const int c = t / per, l = t - c * per;
    prefetch_l2(f + fidx(g, b, i0 + c, min(16 * l, g.ny - 1)));
  }
}

// The FP64 field the fused forward of a column pass transforms: its f-th new
// field, which the epilogue has written to global memory.
__device__ __forceinline__ const double* fwd_field(const EpiArgs& ea, int EPI, int f) {
  if (EPI == EPI_MOM) return ea.vs[f];
  if (EPI == EPI_CORR) return ea.vo[f];
  if (EPI == EPI_DIV) return ea.bvec;
  return ea.phi;  // PPE_SOLVE, PPE_ADD
}

// The epilogue kind is a runtime argument (uniform across the grid): one
// instantiation per precision keeps the build small.
//
// Column pairs i0 + 2p, i0 + 2p + 1 (p < Pp) of one instance.  The nout
// inverse transforms run og at a time: gather the half spectra of the group's
// outputs into packed lines, invert them together, then the epilogue consumes
// them in order.  Per-point FP64 values that a later group or the fused
// forward needs stay in global memory, in the arrays the epilogue writes
// anyway (and in L2 between the passes over one CTA's columns): the momentum
// terms accumulate u.grad + nu lap of each component in registers within a
// group and in its u* array between groups (overwritten by u* at the last
// term), and the fused forward transforms fwd_field(f) (f < fwd_nf), the new
// fields of this pass, og at a time in the same lines.  Shared memory holds
// only the lines: og Pp of them (and a scratch line for a large prime radix).
template <typename T, int RM>
__device__ __forceinline__ void col_inv_body(const GridDev& g, const typename CT<T>::t* spec, size_t fstride,
                                             size_t bstride, int nout, const IpPlan& P,
                                             const typename CT<T>::t* pool, const EpiArgs& ea, int Pp, int og, int ls,
                                             const int EPI, int bx, int by, int part, int nparts) {
  typedef typename CT<T>::t V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // nparts > 1 (momentum and correction): this CTA takes the outputs and the
  // fused forward transform of velocity component `part`
  const int per = (nout + nparts - 1) / nparts;
  const int o_begin = part * per, o_end = min(o_begin + per, nout);
  const int f_begin = nparts > 1 ? part : 0, f_end = nparts > 1 ? min(part + 1, ea.fwd_nf) : ea.fwd_nf;
  V* Z = reinterpret_cast<V*>(smem_raw);
  V* scratch = Z + (size_t)og * Pp * ls;
  const int b = by + g.b0;
  if (inactive(g, b)) return;
  const int i0 = bx * 2 * Pp;
  const int ny = g.ny;
  const bool ppe = (EPI == EPI_PPE_SOLVE || EPI == EPI_PPE_RESID || EPI == EPI_PPE_ADD);
  // the instance's step parameters and the epilogue factors, once per CTA:
  // inside the point loops the compiler would reload them after every store
  // and repeat the FP64 divisions per point
  const double nu_b = ea.s.nu_inst ? ea.s.nu_inst[b] : ea.s.nu;
  const double fx_b = ea.s.fx_inst ? ea.s.fx_inst[b] : ea.s.fx;
  const double dt_b = ea.s.dt_inst ? ea.s.dt_inst[b] : ea.s.dt;
  const double div_c = EPI == EPI_DIV ? ea.s.rho / (ea.s.a * dt_b) : 0.0;   // rho / (a dt)
  const double corr_c = EPI == EPI_CORR ? ea.s.a * dt_b / ea.s.rho : 0.0;  // a dt / rho
  const int nt = EPI == EPI_MOM ? ea.mom_terms : 1;
  for (int o0 = o_begin; o0 < o_end; o0 += og) {
    const int on = min(og, o_end - o0);
    if (ppe) {
      col_gather_dct<T>(Z, Pp, ls, g, i0, spec + b * bstride, P);
    } else {
      for (int oo = 0; oo < on; ++oo)
        col_gather_hermitian<T>(Z + (size_t)oo * Pp * ls, Pp, ls, g, i0, spec + b * bstride + (o0 + oo) * fstride, P.n,
                                [&](V* L, int k, V z) { L[in_slot<T>(P, k)] = cconj(z); });
      // while this group is transformed, bring the next one's spectra and this
      // group's FP64 epilogue operands (state columns) into L2
      for (int o = o0 + on; o < min(o0 + 2 * on, o_end); ++o)
        prefetch_spec_pairs(g, i0, Pp, spec + b * bstride + o * fstride);
      for (int o = o0; o < o0 + on; ++o) {
        if (EPI == EPI_MOM) {
          const int comp = o / nt, term = o - comp * nt;
          prefetch_field_cols(g, b, i0, Pp, ea.vel[term < nt - 1 ? term : comp]);
          if (term == nt - 1) prefetch_field_cols(g, b, i0, Pp, ea.Fp[comp]);
        } else if (EPI == EPI_CORR) {
          prefetch_field_cols(g, b, i0, Pp, ea.vs[o]);
        }
      }
    }
    __syncthreads();
    fft_ip<T, RM>(Z, on * Pp, ls, P, pool, scratch);
    for (int p = 0; p < Pp; ++p)
    for (int j = threadIdx.x; j < ny; j += blockDim.x) {
      const int so = out_slot<T>(P, j);
      double acc[2] = {0.0, 0.0};  // MOM: the component's running sum, both columns
      for (int oo = 0; oo < on; ++oo) {
        const int o = o0 + oo;
        V z = Z[((size_t)oo * Pp + p) * ls + so];
        if (!ppe) z = cconj(z);
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          const int i = i0 + 2 * p + w;
          if (i >= g.ncol) continue;
          const size_t id = fidx(g, b, i, j);
          const T zv = w ? cim(z) : cre(z);
          if (EPI == EPI_OUT) {
            // straight from the compute type to the output type
            if (ea.out_double)
              reinterpret_cast<double*>(ea.outs[o])[id] = (double)zv;
            else
              reinterpret_cast<float*>(ea.outs[o])[id] = (float)zv;
            continue;
          }
          const double val = (double)zv;
          if (EPI == EPI_MOM) {
            // output comp * nt + term: d/dx, d/dy, (d/dz,) lap of component comp;
            // F_comp = u . grad(comp) - nu lap(comp)
            const int comp = o / nt, term = o - comp * nt;
            double* a = ea.vs[comp] + id;
            if (term == 0)
              acc[w] = __dmul_rn(ld_stream(ea.vel[0] + id), val);
            else {
              if (oo == 0) acc[w] = *a;
              if (term < nt - 1) acc[w] = __fma_rn(ld_stream(ea.vel[term] + id), val, acc[w]);
            }
            if (term < nt - 1) {
              if (oo == on - 1) *a = acc[w];
            } else {
              const double nu = nu_b;
              const double F = __fma_rn(-nu, val, acc[w]);
              const double f = comp == 0 ? fx_b : (comp == 1 ? ea.s.fy : ea.s.fz);
              const double dt = dt_b;
              double cs = ld_stream(ea.vel[comp] + id) + dt * (-ea.s.g * F - ea.s.z * ld_stream(ea.Fp[comp] + id) + ea.s.a * f);
              // y walls: the tangential x velocity takes the wall speeds, the others 0
              if (j == 0) cs = comp == 0 ? ea.s.u_bottom : 0.0;
              if (j == ny - 1) cs = comp == 0 ? ea.s.u_top : 0.0;
              if (g.x_walls && (i == 0 || i == g.nx - 1)) cs = 0.0;
              ea.Fp[comp][id] = F;
              *a = cs;
              if (!isfinite(cs)) atomicOr(ea.status, 1);
            }
          } else if (EPI == EPI_DIV) {
            ea.bvec[id] = div_c * val;
          } else if (EPI == EPI_CORR) {
            // output o: d phi / d(axis o) -> component o
            const double c = corr_c;
            double cn = ld_stream(ea.vs[o] + id) - c * val;
            if (j == 0) cn = o == 0 ? ea.s.u_bottom : 0.0;
            if (j == ny - 1) cn = o == 0 ? ea.s.u_top : 0.0;
            if (g.x_walls && (i == 0 || i == g.nx - 1)) cn = 0.0;
            ea.vo[o][id] = cn;
            if (!isfinite(cn)) atomicOr(ea.status, 1);
          } else if (EPI == EPI_PPE_SOLVE) {
            if (ea.phi_double)
              reinterpret_cast<double*>(ea.phi_any)[id] = val;
            else
              reinterpret_cast<float*>(ea.phi_any)[id] = (float)val;
            if (ea.phi) ea.phi[id] = val;
          } else if (EPI == EPI_PPE_RESID) {
            ea.phi[id] = ld_stream(ea.bvec + id) - val;  // r = b - L phi
          } else if (EPI == EPI_PPE_ADD) {
            ea.phi[id] = ea.phi[id] + val;
          }
        }
      }
    }
    __syncthreads();
  }
  const IpPlan& FP = ea.fwdP;
  for (int f0 = f_begin; f0 < f_end; f0 += og) {
    const int fn = min(og, f_end - f0);
    // the new fields as this CTA's threads stored them above (a thread reads
    // back its own points; columns beyond nx, a ragged last pair, are zero)
    for (int ff_ = 0; ff_ < fn; ++ff_) {
      const double* a = fwd_field(ea, EPI, f0 + ff_);
      for (int p = 0; p < Pp; ++p) {
        const int i = i0 + 2 * p;
        V* L = Z + ((size_t)ff_ * Pp + p) * ls;
        constexpr int U = std::is_same<T, double>::value ? 1 : 2;  // FP64 spills (fc_append_f64)
        double x_[U], y_[U];
        batched<U>(ny, [&](int u, int j) {
          x_[u] = i < g.ncol ? ld_stream(a + fidx(g, b, i, j)) : 0.0;
          y_[u] = i + 1 < g.ncol ? ld_stream(a + fidx(g, b, i + 1, j)) : 0.0;
        }, [&](int u, int j) { L[in_slot<T>(FP, j)] = mk<V>(to_t<T>(x_[u]), to_t<T>(y_[u])); });
      }
    }
    __syncthreads();
    col_forward_store<T, RM>(Z, scratch, fn, Pp, ls, g, i0, reinterpret_cast<const typename FcTab<T>::t*>(ea.fwdE), FP, pool,
                         ea.fwd_dct, reinterpret_cast<V*>(ea.fwd_spec) + b * ea.fwd_bstride + f0 * ea.fwd_fstride,
                         ea.fwd_fstride);
    __syncthreads();
  }
}

template <typename T, int RM>
__global__ void __launch_bounds__(kMaxThreads, MinCtas<T, RM>::v) k_col_inv(const __grid_constant__ GridDev g, const typename CT<T>::t* __restrict__ spec,
                                                         size_t fstride, size_t bstride, int nout,
                                                         const __grid_constant__ IpPlan P,
                                                         const typename CT<T>::t* __restrict__ pool,
                                                         const __grid_constant__ EpiArgs ea, int Pp, int og, int ls,
                                                         const int EPI) {
  col_inv_body<T, RM>(g, spec, fstride, bstride, nout, P, pool, ea, Pp, og, ls, EPI, blockIdx.x, blockIdx.y, blockIdx.z,
                  gridDim.z);
}

// ---------------------------------------------------------------------------
// Persistent step of several size classes in one launch.  Every pass of one
// RK3 step of every class is recorded as a descriptor (the arguments its
// launch would get); a work item is one CTA's share of one pass for one
// instance: (descriptor, tile x, tile y, instance).  Items are listed pass by
// pass (pass index p of every class, then p + 1, ...), and the CTAs of one
// launch take them in that order from an atomic counter.  Item (c, b, p)
// waits until every tile of pass p - 1 of the same instance has finished
// (a per-(class, instance, pass) counter), so the classes' passes and their
// instances interleave freely.  No deadlock is possible: an item only waits
// for items taken before it, and the oldest unfinished item waits for nothing.
// Waits are bounded (time and spin count); one that runs out sets bit 1 of
// the plan's status word, and from then on every item is skipped (and
// counted) so the launch drains at once.
enum { PK_COL_FWD = 1, PK_ROW_SYM = 2, PK_COL_INV = 3, PK_ROW_PPE = 4 };

struct PassDesc {
  int kind;
  int gx, gy, gz;  // the grid the pass's own launch would have
  size_t smem;
  int Pp, Rr, ob, og, ls;
  GridDev g;
  IpPlan P;
  const void* pool;
  const void* E;
  // column forward / column inverse
  const void* f[3];
  int dct;
  void* spec;
  size_t fstride, bstride;
  // row passes
  const void* sp_in;
  void* sp_out;
  size_t fs_in, bs_in, fs_out, bs_out;
  RowOps ops;
  const void* W;
  double scale;
  int apply;
  // column inverse
  int nout, epi;
  EpiArgs ea;
};

struct WorkItem {
  int desc, bx, by, b;
  int dep;   // counter the item waits on (-1: none)
  int need;  // value that counter must reach
  int self;  // counter the item increments when done
};

constexpr int kPersistTimeout = 2;          // status bit: a dependency wait ran out
constexpr long long kPersistMaxSpins = 1ll << 26;

__device__ __forceinline__ long long global_ns() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// One function per pass kind, each compiled (and register-allocated) on its
// own rather than all four inlined into the persistent loop.  The descriptor
// is read-only for the whole launch and aliases nothing the pass writes
// (__restrict__): its fields are loaded once, not again after every store.
template <typename T, int RM> __device__ __noinline__ void item_col_fwd(const PassDesc& __restrict__ d, int bx, int by, int b) {
  typedef typename CT<T>::t V;
  col_fwd_body<T, double, RM>(d.g, (const double*)d.f[0], (const double*)d.f[1], (const double*)d.f[2],
                          (const typename FcTab<T>::t*)d.E, d.P, (const V*)d.pool, d.dct, (V*)d.spec, d.fstride,
                          d.bstride, d.Pp, d.ls, bx, by, b);
}
template <typename T, int RM> __device__ __noinline__ void item_row_sym(const PassDesc& __restrict__ d, int bx, int fz, int b) {
  typedef typename CT<T>::t V;
  row_sym_body<T, RM>(d.g, (const V*)d.sp_in, (V*)d.sp_out, d.fs_in, d.bs_in, d.fs_out, d.bs_out, d.ops,
                  (const typename FcTab<T>::t*)d.E, d.P, (const V*)d.pool, (const T*)d.W, d.scale, d.Rr, d.ob, d.ls, bx, b, fz);
}
template <typename T, int RM> __device__ __noinline__ void item_col_inv(const PassDesc& __restrict__ d, int bx, int b) {
  typedef typename CT<T>::t V;
  col_inv_body<T, RM>(d.g, (const V*)d.spec, d.fstride, d.bstride, d.nout, d.P, (const V*)d.pool, d.ea, d.Pp, d.og, d.ls,
                  d.epi, bx, b, 0, 1);
}
template <typename T, int RM> __device__ __noinline__ void item_row_ppe(const PassDesc& __restrict__ d, int bx, int b) {
  typedef typename CT<T>::t V;
  row_ppe_body<T, RM>(d.g, (V*)d.spec, d.bstride, d.P, (const V*)d.pool, d.apply, d.Rr, d.ls, bx, b);
}

__device__ __forceinline__ void red_release_gpu_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <typename T, int RM>
__device__ __forceinline__ void run_item(const PassDesc& d, int bx, int by, int b) {
  switch (d.kind) {
    case PK_COL_FWD: item_col_fwd<T, RM>(d, bx, by, b); break;
    case PK_ROW_SYM: item_row_sym<T, RM>(d, bx, by, b); break;
    case PK_COL_INV: item_col_inv<T, RM>(d, bx, b); break;
    case PK_ROW_PPE: item_row_ppe<T, RM>(d, bx, b); break;
    default: break;
  }
}

// stall >= 0: item `stall` waits for a count that never comes (a test of the
// bounded wait).
// Register budget of the persistent kernel: its pass bodies read the grid,
// plan and epilogue fields from the descriptor in global memory, where the
// per-pass kernels take them as constant-bank operands, so the same code needs
// more registers; the FP32-pair kernel of large radices gets up to 255 (8
// warps per SM) rather than spilling at 168.
template <typename T, int RM> struct PersistMinCtas { static constexpr int v = 3; };
template <> struct PersistMinCtas<ff, 31> { static constexpr int v = 2; };

// Built for RM = 9 and 31 only.
template <typename F> cudaError_t with_persist_rm(int rmax, F&& f) {
  if (rmax <= 9) return f(std::integral_constant<int, 9>{});
  return f(std::integral_constant<int, 31>{});
}

template <typename T, int RM>
__global__ void __launch_bounds__(kMaxThreads, PersistMinCtas<T, RM>::v) k_persist(const PassDesc* descs, const WorkItem* items,
                                                                  int n_items, unsigned* counters, unsigned* next,
                                                                  int* status, long long wait_ns, int stall) {
  __shared__ int s_idx, s_run;
  for (;;) {
    if (threadIdx.x == 0) {
      const int idx = (int)atomicAdd(next, 1u);
      int run = 1;
      if (idx < n_items) {
        const WorkItem it = items[idx];
        if (it.dep >= 0) {
          const unsigned need = idx == stall ? 0xffffffffu : (unsigned)it.need;
          const unsigned* cnt = counters + it.dep;
          const long long t0 = global_ns();
          for (long long spin = 0;; ++spin) {
            if (ld_acquire_gpu(cnt) >= need) break;
            if ((*(volatile int*)status & kPersistTimeout) || spin > kPersistMaxSpins || global_ns() - t0 > wait_ns) {
              atomicOr(status, kPersistTimeout);
              run = 0;
              break;
            }
            __nanosleep(100);
          }
        }
        if (*(volatile int*)status & kPersistTimeout) run = 0;
      }
      s_idx = idx;
      s_run = run;
    }
    // thread 0's acquire of the dependency count, then the CTA barrier, orders
    // the dependency's writes before every load of this item
    __syncthreads();
    const int idx = s_idx, run = s_run;
    if (idx >= n_items) return;
    const WorkItem& it = items[idx];
    if (run) run_item<T, RM>(descs[it.desc], it.bx, it.by, it.b);
    // the barrier, then thread 0's release increment, orders every write of
    // this item before its count
    __syncthreads();
    if (threadIdx.x == 0 && it.self >= 0) red_release_gpu_add(counters + it.self, 1u);
  }
}

// ---------------------------------------------------------------------------
// Wall-normal passes of FP32 contexts with the register team FFT of
// fcsph_regfft.cuh, NP column pairs per CTA: BS = false for extended lengths n =
// N1 N2 with a direct plan; BS = true for lengths with a large prime factor (n
// = 537 and 1049 with n_cont = 25 at 512 and 1024 nodes), Bluestein's
// convolution on a team FFT of length m = N1 N2 = 1080 or 2100 (chirp, filter
// and m roots from the context's plan in the FP32 pool).  k_col_fwd_r does
// what k_col_fwd does for FP32 fields (load, FC, forward transform, half
// spectrum); k_col_out_r what k_col_inv does with EPI_OUT into FP32 outputs
// (Hermitian gather, inverse transform, store), for every output.  Line and
// exchange block share a buffer.
//
// What bounds them: the forward pass waited on the twiddle gathers
// (long_scoreboard 3.7 cycles per instruction) and both kept the shared-memory
// and L1 data pipe 59 % busy, half of that scattered twiddles; they are now read
// from a table in the threads' order.  Pairs per CTA as measured (64 planes of
// 1024^2, n = 1050: forward 229 us at 3 against 246, 237 and 240 at 2, 4 and 7;
// output 457 at 3, 485, 478 and 580; 512^2, n = 540: forward 62 at 4 against 82
// at 1, output 110 at 1 against 124 at 4).  One pair per CTA and gathered roots
// -> now: forward 308 -> 221 us (37 % of the copy rate on its bytes), output
// 513 -> 400 us (61 %); at n = 1049 834 -> 714 and 2181 -> 1662 us; the line
// operator on 4096 lines of 512 at n = 537 88 -> 63 us.
template <int N1, int N2, int NP, bool BS>
__global__ void __launch_bounds__(TeamFFT<N1, N2>::threads(NP), TeamFFT<N1, N2>::min_ctas(NP)) k_col_fwd_r(
    GridDev g, const float* __restrict__ f0, const float* __restrict__ f1, const float* __restrict__ f2,
    const typename FcTab<float>::t* __restrict__ E, const float2* __restrict__ chirp,
    const float2* __restrict__ bhat, const float2* __restrict__ tw, float2* __restrict__ spec, size_t fstride,
    size_t bstride) {
  typedef TeamFFT<N1, N2> TF;
  const int n = BS ? g.my : N1 * N2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int p, t;
  team_of<TF::NV, NP>(p, t);
  float2* L0 = reinterpret_cast<float2*>(smem_raw);
  float2* L = L0 + p * TF::LINE;
  const int b = blockIdx.z + g.b0, f = blockIdx.y;
  if (inactive(g, b)) return;
  const int i0 = blockIdx.x * 2 * NP;
  const float* src = (f == 0 ? f0 : (f == 1 ? f1 : f2)) + (size_t)b * g.ncol * g.ny;
  const int ny = g.ny;
  for (int q = 0; q < NP; ++q) {
    const int i = i0 + 2 * q;
    if (i < g.ncol) load_pair_f32(L0 + q * TF::LINE, src + (size_t)i * ny, i + 1 < g.ncol, ny);
  }
  __syncthreads();
  fc_append<float>(L0, NP, TF::LINE, ny, g.n_cont, g.n_match, E, NatSlot());
  __syncthreads();
  if constexpr (BS) {
    bluestein_team<N1, N2, false, true, NP == 1>(L, L, n, chirp, bhat, tw, t);
  } else {
    float2 v[TF::NV];
    if (t < N2) {
#pragma unroll
      for (int j = 0; j < N1; ++j) v[j] = L[t + N2 * j];
    }
    TF::template fwd<true>(v, L, tw, t);
    if (t < N1) {
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) L[t + N1 * k2] = v[k2];
    }
    __syncthreads();
  }
  team_store_spectrum<NP>(L0, TF::LINE, g, i0, n, spec + b * bstride + f * fstride);
}

// The inverse transform of one team's line and the store of its pair's output.
template <int N1, int N2, int NP, bool BS>
__device__ __forceinline__ void team_inv_store(const GridDev& g, float2* L, int n, const float2* __restrict__ chirp,
                                               const float2* __restrict__ bhat, const float2* __restrict__ tw, int t,
                                               float* out, int b, int i) {
  typedef TeamFFT<N1, N2> TF;
  const int ny = g.ny;
  if constexpr (BS) {
    bluestein_team<N1, N2, true, true, NP == 1>(L, L, n, chirp, bhat, tw, t);
    if (i < g.ncol)
      team_each<N1, N2, NP == 1>(t, ny, [&](int j) {
        out[fidx(g, b, i, j)] = L[j].x;
        if (i + 1 < g.ncol) out[fidx(g, b, i + 1, j)] = L[j].y;
      });
    __syncthreads();  // L is rewritten by the next output
  } else {
    float2 v[TF::NV];
    if (t < N1) {
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) v[k2] = L[t + N1 * k2];
    }
    TF::template inv<true>(v, L, tw, t);
    if (t < N2 && i < g.ncol) {
#pragma unroll
      for (int j = 0; j < N1; ++j) {
        const int row = t + N2 * j;
        if (row < ny) {
          out[fidx(g, b, i, row)] = v[j].x;
          if (i + 1 < g.ncol) out[fidx(g, b, i + 1, row)] = v[j].y;
        }
      }
    }
  }
}

template <int N1, int N2, int NP, bool BS>
__global__ void __launch_bounds__(TeamFFT<N1, N2>::threads(NP), TeamFFT<N1, N2>::min_ctas(NP)) k_col_out_r(
    GridDev g, const float2* __restrict__ spec, size_t fstride, size_t bstride, int nout, const EpiArgs ea,
    const float2* __restrict__ chirp, const float2* __restrict__ bhat, const float2* __restrict__ tw) {
  typedef TeamFFT<N1, N2> TF;
  const int n = BS ? g.my : N1 * N2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int p, t;
  team_of<TF::NV, NP>(p, t);
  float2* L0 = reinterpret_cast<float2*>(smem_raw);
  const int b = blockIdx.y + g.b0;
  if (inactive(g, b)) return;
  const int i0 = blockIdx.x * 2 * NP;
  for (int o = 0; o < nout; ++o) {
    team_gather<NP>(L0, TF::LINE, g, i0, n, spec + b * bstride + o * fstride);
    // the next output's half spectrum into L2 while this one is transformed
    if (o + 1 < nout) prefetch_spec_pairs(g, i0, NP, spec + b * bstride + (o + 1) * fstride);
    __syncthreads();
    team_inv_store<N1, N2, NP, BS>(g, L0 + p * TF::LINE, n, chirp, bhat, tw, t, reinterpret_cast<float*>(ea.outs[o]), b,
                               i0 + 2 * p);
  }
}

// line_op on the Bluestein team transform: the forward spectrum stays in L,
// each output is formed in W (symbol times spectrum over n) and inverted there.
template <int N1, int N2, int NP>
__global__ void __launch_bounds__(TeamFFT<N1, N2>::threads(NP), TeamFFT<N1, N2>::min_ctas(NP)) k_line_op_rb(
    GridDev g, const float* __restrict__ f, long long ncols, const typename FcTab<float>::t* __restrict__ E,
    const float2* __restrict__ pool, const float2* __restrict__ chirp, const float2* __restrict__ bhat,
    const float2* __restrict__ tw, const __grid_constant__ LineOuts lo) {
  typedef TeamFFT<N1, N2> TF;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int p, t;
  team_of<TF::NV, NP>(p, t);
  float2* L0 = reinterpret_cast<float2*>(smem_raw);
  float2* L = L0 + p * TF::LINE;
  float2* W = L + NP * TF::LINE;
  const long long cb = (long long)blockIdx.x * 2 * NP, c0 = cb + 2 * p;
  const int ny = g.ny, n = g.my;
  for (int q = 0; q < NP; ++q)
    if (cb + 2 * q < ncols) load_pair_f32(L0 + q * TF::LINE, f + (cb + 2 * q) * ny, cb + 2 * q + 1 < ncols, ny);
  __syncthreads();
  fc_append<float>(L0, NP, TF::LINE, ny, g.n_cont, g.n_match, E, NatSlot());
  __syncthreads();
  bluestein_team<N1, N2, false, true, NP == 1>(L, L, n, chirp, bhat, tw, t);
  const float hh = g.hh_f, cky = g.cky_f, tscale = g.inv_my_f;  // n = my
  for (int o = 0; o < lo.nout; ++o) {
    const int op = lo.op[o];
    team_each<N1, N2, NP == 1>(t, n, [&](int k) {
      const int kappa = (2 * k <= n) ? k : k - n;
      const float ky = cky * (float)kappa;
      const float What = pool[g.ey_off + (kappa < 0 ? -kappa : kappa)].x * kernel_poly<float>(g.family, ky * ky * hh);
      const bool nyq = (n % 2 == 0) && (2 * k == n);
      float2 sy;
      if (op == SYM_W)
        sy = make_float2(What, 0.f);
      else if (op == SYM_DY)
        sy = make_float2(0.f, nyq ? 0.f : ky * What);
      else if (op == SYM_LAP)
        sy = make_float2(-(ky * ky) * What, 0.f);
      else
        sy = make_float2(0.f, 0.f);
      W[k] = cscale(cmul(sy, L[k]), tscale);
    });
    __syncthreads();
    bluestein_team<N1, N2, true, true, NP == 1>(W, W, n, chirp, bhat, tw, t);
    float* out = reinterpret_cast<float*>(lo.out[o]);
    team_each<N1, N2, NP == 1>(t, ny, [&](int j) {
      if (c0 < ncols) out[c0 * ny + j] = W[j].x;
      if (c0 + 1 < ncols) out[(c0 + 1) * ny + j] = W[j].y;
    });
    __syncthreads();
  }
}

// k_col_out_r with TMA staging, persistent over (NP column pairs, output)
// units: while one unit's inverse transforms run, the next unit's half-spectrum
// rows (the pairs' complex values of rows ky < hy, 16 NP bytes a row) arrive in
// a staging buffer by 2D tiled bulk copies (nbox boxes of rows_box rows) on
// one mbarrier, so the column pass no longer waits on its strided gather.
// The wait for a copy is bounded: on a timeout the CTA sets bit 1 of the
// status word, waits once more (bounded) for its copy in flight and returns.
template <int N1, int N2, int NP, bool BS>
__global__ void __launch_bounds__(TeamFFT<N1, N2>::threads(NP), TeamFFT<N1, N2>::min_ctas(NP)) k_col_out_rt(
    GridDev g, const __grid_constant__ CUtensorMap tmap, int rows_box, int nbox, int nfo, int nout,
    const EpiArgs ea, const float2* __restrict__ tw, int ngroups, const float2* __restrict__ chirp,
    const float2* __restrict__ bhat) {
  typedef TeamFFT<N1, N2> TF;
  const int n = BS ? g.my : N1 * N2;  // the line's length (BS: transformed by Bluestein on length N1 N2)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // bulk tensor copies land on 128-byte boundaries (the launch adds 128 bytes)
  float4* stage = reinterpret_cast<float4*>(smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u));
  float2* L0 = reinterpret_cast<float2*>(stage + (size_t)nbox * rows_box * NP);
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_ok;
  int p, t;
  team_of<TF::NV, NP>(p, t);
  const int hy = g.hy;
  const long long W = (long long)g.nb * ngroups;
  const uint32_t bytes = (uint32_t)(nbox * rows_box * 16 * NP);
  auto group_of = [&](long long k) { return (long long)blockIdx.x + (k / nout) * gridDim.x; };
  auto issue = [&](long long k) {  // thread 0: copies of unit k into the stage
    const long long w = group_of(k);
    const int o = (int)(k % nout);
    const int b = g.b0 + (int)(w / ngroups), i0 = (int)(w % ngroups) * 2 * NP;
    const int row0 = (b * nfo + o) * g.rows;
    fence_proxy_async();
    mbar_arrive_expect_tx(&bar, bytes);
    for (int q = 0; q < nbox; ++q)
      tma_load_2d(stage + (size_t)q * rows_box * NP, &tmap, 2 * i0, row0 + q * rows_box, &bar);
  };
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (group_of(0) >= W) return;
  if (threadIdx.x == 0) issue(0);
  for (long long k = 0; group_of(k) < W; ++k) {
    const long long w = group_of(k);
    const int o = (int)(k % nout);
    const int b = g.b0 + (int)(w / ngroups), i0 = (int)(w % ngroups) * 2 * NP;
    const uint32_t par = (uint32_t)(k & 1);
    if (threadIdx.x == 0) s_ok = mbar_wait_bounded(&bar, par) ? 1 : 0;
    __syncthreads();
    if (!s_ok) {
      if (threadIdx.x == 0) {
        atomicOr(ea.status, 2);
        mbar_wait_bounded(&bar, par);
      }
      return;
    }
    mbar_try_wait(&bar, par);  // every thread observes the completed phase
    // Hermitian unpack: Z_k = A_k + i B_k, Z_{n-k} = conj(A_k) + i conj(B_k)
    for (int e = threadIdx.x; e < hy * NP; e += blockDim.x) {
      const int kk = e / NP, q = e - kk * NP;
      const float4 r = stage[e];
      float2* L = L0 + (size_t)q * TF::LINE;
      if (kk == 0 || 2 * kk == n) {
        L[kk] = make_float2(r.x, r.z);
      } else {
        L[kk] = make_float2(r.x - r.w, r.y + r.z);
        L[n - kk] = make_float2(r.x + r.w, r.z - r.y);
      }
    }
    __syncthreads();
    if (threadIdx.x == 0 && group_of(k + 1) < W) issue(k + 1);  // the stage is free again
    team_inv_store<N1, N2, NP, BS>(g, L0 + p * TF::LINE, n, chirp, bhat, tw, t, reinterpret_cast<float*>(ea.outs[o]), b,
                               i0 + 2 * p);
  }
}

// ---------------------------------------------------------------------------
// fc_extend (Eq. 30) as a standalone kernel: y continuation of every column,
// then x continuation of every extended row (walled x).
template <typename U>
__global__ void k_fc_extend_y(GridDev g, const U* __restrict__ f, U* __restrict__ fe, const double* __restrict__ E) {
  const size_t total = (size_t)g.batch * g.ncol * g.my;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(t % g.my);
    const size_t bi = t / g.my;
    const int i = (int)(bi % g.ncol);
    const int b = (int)(bi / g.ncol);
    const U* col = f + ((size_t)b * g.ncol + i) * g.ny;
    double v;
    if (j < g.ny) {
      v = (double)col[j];
    } else {
      const int c = j - g.ny, d = g.n_match;
      Dot2 acc;
      for (int m = 0; m < d; ++m) {
        acc.add(E[c * 2 * d + m], (double)col[g.ny - d + m]);
        acc.add(E[c * 2 * d + d + m], (double)col[m]);
      }
      v = acc.value();
    }
    fe[((size_t)b * (g.x_walls ? g.mx : g.ncol) + i) * g.my + j] = (U)v;
  }
}

template <typename U>
__global__ void k_fc_extend_x(GridDev g, U* __restrict__ fe, const double* __restrict__ E) {
  const int C = g.n_cont, d = g.n_match;
  const size_t total = (size_t)g.batch * C * g.my;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(t % g.my);
    const size_t bc = t / g.my;
    const int c = (int)(bc % C);
    const int b = (int)(bc / C);
    U* base = fe + (size_t)b * g.mx * g.my;
    Dot2 acc;
    for (int m = 0; m < d; ++m) {
      acc.add(E[c * 2 * d + m], (double)base[(size_t)(g.nx - d + m) * g.my + j]);
      acc.add(E[c * 2 * d + d + m], (double)base[(size_t)m * g.my + j]);
    }
    base[(size_t)(g.nx + c) * g.my + j] = (U)acc.value();
  }
}

// Batched DFT of contiguous lines with the ping-pong engine (no index tables).
template <typename T, bool INV>
__global__ void __launch_bounds__(kThreads) k_dft_lines(int n, int nlines, const typename CT<T>::t* __restrict__ in,
                                                        typename CT<T>::t* __restrict__ out,
                                                        const __grid_constant__ FftPlan P,
                                                        const typename CT<T>::t* __restrict__ pool, int L, int ls) {
  typedef typename CT<T>::t V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* A = reinterpret_cast<V*>(smem_raw);
  V* B = A + (size_t)L * ls;
  const int l0 = blockIdx.x * L;
  for (int e = threadIdx.x; e < L * n; e += blockDim.x) {
    const int r = e / n, j = e - (e / n) * n;
    A[(size_t)r * ls + j] = l0 + r < nlines ? in[(size_t)(l0 + r) * n + j] : mk<V>((T)0, (T)0);
  }
  __syncthreads();
  V* Y = fft_any<T, INV>(A, B, L, ls, P, pool);
  for (int e = threadIdx.x; e < L * n; e += blockDim.x) {
    const int r = e / n, j = e - (e / n) * n;
    if (l0 + r < nlines) out[(size_t)(l0 + r) * n + j] = Y[(size_t)r * ls + j];
  }
}

// The same with the in-place engine of the passes (fcsph_dft); IO is the
// element type in memory (double2 for FP32 pairs, else the engine's own).
template <typename T, typename IO>
__global__ void __launch_bounds__(kMaxThreads, MinCtas<T, 31>::v) k_dft_ip(int n, int nlines, const IO* __restrict__ in,
                                                                    IO* __restrict__ out,
                                                                    const __grid_constant__ IpPlan P,
                                                                    const typename CT<T>::t* __restrict__ pool, int L,
                                                                    int ls, int inv) {
  typedef typename CT<T>::t V;
  typedef decltype(IO().x) E;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* A = reinterpret_cast<V*>(smem_raw);
  const int l0 = blockIdx.x * L;
  const int nl = min(L, nlines - l0);
  for (int r = 0; r < nl; ++r)
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      const IO x = in[(size_t)(l0 + r) * n + j];
      const V v = mk<V>((T)x.x, (T)x.y);
      A[(size_t)r * ls + in_slot<T>(P, j)] = inv ? cconj(v) : v;
    }
  __syncthreads();
  fft_ip<T, 31>(A, nl, ls, P, pool, A + (size_t)L * ls);
  for (int r = 0; r < nl; ++r)
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      V y = A[(size_t)r * ls + out_slot<T>(P, j)];
      if (inv) y = cconj(y);
      out[(size_t)(l0 + r) * n + j] = mk<IO>(static_cast<E>(cre(y)), static_cast<E>(cim(y)));
    }
}

// Residual diagnostics, one block per instance: out[0] += sum_b (r - mean_b(r))^2,
// out[1] += sum_b b^2 (two passes over the instance: mean, then deviations).
__global__ void k_resid_inst(const double* __restrict__ r, const double* __restrict__ b, size_t n_inst, double* out) {
  __shared__ double sh[2][kThreads];
  const double* ri = r + blockIdx.x * n_inst;
  const double* bi = b + blockIdx.x * n_inst;
  double s0 = 0.0;
  for (size_t t = threadIdx.x; t < n_inst; t += blockDim.x) s0 += ri[t];
  sh[0][threadIdx.x] = s0;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
    __syncthreads();
  }
  const double mean = sh[0][0] / (double)n_inst;
  __syncthreads();
  double d2 = 0.0, b2 = 0.0;
  for (size_t t = threadIdx.x; t < n_inst; t += blockDim.x) {
    const double d = ri[t] - mean;
    d2 += d * d;
    b2 += bi[t] * bi[t];
  }
  sh[0][threadIdx.x] = d2;
  sh[1][threadIdx.x] = b2;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    atomicAdd(out + 0, sh[0][0]);
    atomicAdd(out + 1, sh[1][0]);
  }
}

// The constant (0,0) mode of the PPE transforms (DCT-I in y and, walled x, in x:
// end nodes count half; DFT along periodic axes) removed from every instance:
// out = b - sum(w b) / sum(w).  First kernel: partial sums of kMeanParts runs
// of columns per instance (grid kMeanParts x batch, fixed order: the result
// does not depend on scheduling); second: every CTA adds the partial sums of
// its instance and subtracts.  One read and one write of the field in place of
// the forward and inverse FP64 transforms that used to clear the mode (2016 ->
// 1170 us for a refined solve of 4 channels of 512^2, with the solve's copies).
constexpr int kMeanParts = 64;

__global__ void __launch_bounds__(kThreads) k_mean_part(GridDev g, const double* __restrict__ b,
                                                        double* __restrict__ part) {
  __shared__ double sh[kThreads];
  const int ny = g.ny;
  const int c0 = (int)((long long)g.ncol * blockIdx.x / kMeanParts), c1 = (int)((long long)g.ncol * (blockIdx.x + 1) / kMeanParts);
  double s = 0.0;
  for (int c = c0; c < c1; ++c) {
    const double* col = b + ((size_t)blockIdx.y * g.ncol + c) * ny;
    const double wx = g.x_walls && (c == 0 || c == g.nx - 1) ? 0.5 : 1.0;
    for (int j = threadIdx.x; j < ny; j += kThreads) s += (j == 0 || j == ny - 1 ? 0.5 : 1.0) * wx * col[j];
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.y * kMeanParts + blockIdx.x] = sh[0];
}

__global__ void __launch_bounds__(kThreads) k_sub_mean(GridDev g, const double* __restrict__ b,
                                                       const double* __restrict__ part, double inv_w,
                                                       double* __restrict__ out) {
  __shared__ double sh[kMeanParts];
  if (threadIdx.x < kMeanParts) sh[threadIdx.x] = part[blockIdx.y * kMeanParts + threadIdx.x];
  __syncthreads();
  for (int w = kMeanParts / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  const double mean = sh[0] * inv_w;
  const size_t n = (size_t)g.ncol * g.ny, base = blockIdx.y * n;
  for (size_t t = blockIdx.x * (size_t)kThreads + threadIdx.x; t < n; t += (size_t)gridDim.x * kThreads)
    out[base + t] = b[base + t] - mean;
}

__global__ void k_widen(double* __restrict__ y, const float* __restrict__ x, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    y[t] = (double)x[t];
}

__global__ void k_narrow(float* __restrict__ y, const double* __restrict__ x, size_t n) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
    y[t] = (float)x[t];
}

// ---------------------------------------------------------------------------
// Host-side launch helpers.

// Largest count (>= 1, <= cap) of units fitting in `budget` bytes.
int fit_units(size_t per_unit, size_t budget, int cap) {
  int u = (int)(budget / per_unit);
  if (u < 1) u = 1;
  if (u > cap) u = cap;
  return u;
}

constexpr size_t kSmemBudget = 96 * 1024;  // per CTA of the multi-line engine test kernel
constexpr size_t kSmemMax = 227 * 1024;

// Every kernel's dynamic shared-memory limit is raised once, at the first
// context creation (init_kernel_attributes), so that no attribute call ever
// happens while a stream is being captured; launches only check the size.
cudaError_t check_smem(size_t bytes) {
  return bytes > kSmemMax ? cudaErrorInvalidValue : cudaSuccess;
}

template <typename K> cudaError_t raise_smem(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
}

// FC table (bc) in the FcTab type of precision prec.
const void* fc_table(const fcsph_ctx* c, int prec, int bc) {
  const size_t off = (bc == FCSPH_NEUMANN ? 1 : 0) * (size_t)c->gd.n_cont * 2 * c->gd.n_match;
  if (prec == FCSPH_F32X2 || prec == FCSPH_F32) return static_cast<const ff*>(c->dEff) + off;
  return c->dE + off;
}

// Fields per instance of the spectrum buffers: spec_in holds the forward
// transforms of the velocity components (2D: 2, 3D: 3), spec_out the row
// pass outputs (2D: 6, 3D: 12).
size_t spec_in_fields(const fcsph_ctx* c) { return c->gd.nz > 1 ? 3 : 2; }
size_t spec_out_fields(const fcsph_ctx* c) { return c->gd.nz > 1 ? 12 : 6; }

int col_ls(const fcsph_ctx* c) {
  int ls = c->plan_y.line_len();
  if (c->plan_py.line_len() > ls) ls = c->plan_py.line_len();
  return ls;
}

// Warps an SM holds of CTAs of nt threads and `lines` lines of shared memory.
int warps_fitting(size_t lines, size_t line_bytes, int nt) {
  const size_t per_sm = 228 * 1024, reserved = 1024, cta = lines * line_bytes;
  return cta > kSmemMax ? 0 : (int)(per_sm / (cta + reserved)) * (nt / 32);
}
constexpr int kWantWarps = 12;

// Outputs a CTA transforms together (`per` lines each, beside `base` lines): the
// most up to `want` that leave 12 resident warps; at least one.  More lines in
// one transform fill more lanes of every stage (a 280-point line alone: 35, 56
// and 40 butterflies on 32 lanes), fewer warps hide less latency: row pass of
// 32 cavities of 256^2 in FP32 pairs 420 us at three outputs and 12 warps, 555
// at one and 20.
int fit_group(int want, int base, int per, size_t line_bytes, int nt) {
  for (int u = want; u > 1; --u)
    if (warps_fitting(base + u * per, line_bytes, nt) >= kWantWarps) return u;
  return 1;
}

// Plan P as a launch of `ctas` CTAs runs it: FP64 stages wide where the CTAs do
// not outnumber the SMs (ip_stage_wide); outside the time step large prime
// radices by symmetry (ip_stage_sym).
template <typename T> IpPlan launch_plan(const fcsph_ctx* c, const IpPlan& P, long long ctas) {
  IpPlan Q = P;
  Q.wide = std::is_same<T, double>::value && !c->rec && ctas <= 152;
  Q.sym = !c->in_step;
  return Q;
}

// Launch shape of one pass: `units` (rows or column pairs of all instances)
// dealt `u` to a CTA of `nt` threads.
struct Shape {
  int u, nt;
};
// `row`: the row passes' setting, else the column passes'.  A context whose
// caller has set no tiling or width picks per pass: passes with few units keep
// one per CTA at the width the context started with (several warps per line);
// otherwise one-warp CTAs for lines up to 128 points and two warps beyond, with
// units enough that each stage has two butterflies per thread, while at least
// 8 CTAs per SM remain.  Steps and operators of batches of 40^2 to 512^2 in FP64 and
// pairs, geometric mean of 52 against these lines: 1.6 % longer with 4 CTAs per SM
// (80^2, 64 fields, pairs, 80 -> 105 us), 1.7 % with 16; 4.9 % with one warp up to 64
// points only, 1.0 % less up to 256 points but 16 % more at worst.  `together`: lines
// of one unit in one transform, `held`: lines a unit keeps in shared memory.  In both cases a pass whose
// lines leave room for fewer than 12 warps runs wider (2048-point convolutions
// of a 512^2 box: row pass of the pressure 1224 us at one warp per CTA, 670 at
// two, 481 at four).
Shape pass_shape(const fcsph_ctx* c, bool row, long long units, int n, int together, int held, size_t line_bytes) {
  Shape s{row ? c->row_lines : c->col_pairs, row ? c->row_threads : c->col_threads};
  if (c->auto_shape && c->prec.fft_prec != FCSPH_F32) {
    s.u = 1;
    const long long full = 152LL * kWantWarps;
    s.nt = 4 * units <= full ? 128 : 2 * units <= full ? 64 : 32;
    if (s.nt == 32) {
      if (n > 128) s.nt = 64;
      while (s.u < 4 && s.u * together * (n / 8) < 2 * s.nt && units / (2 * s.u) >= 152 * 8 &&
             warps_fitting((size_t)2 * s.u * held, line_bytes, s.nt) >= kWantWarps)
        s.u *= 2;
    }
  }
  while (s.nt < kMaxThreads && warps_fitting((size_t)s.u * held, line_bytes, s.nt) < kWantWarps) s.nt *= 2;
  return s;
}

}  // namespace

// ===========================================================================
// Launchers

// Recording (fcsph_ctx::rec set): a pass of isph_step is appended to the
// recording as a descriptor instead of being launched.  FP64 and FP32x2 only
// (the persistent kernel's types).
struct PersistRec {
  std::vector<PassDesc> descs;
};

template <typename T> cudaError_t rec_push(fcsph_ctx* c, PassDesc& d) {
  if (!std::is_same<T, double>::value && !std::is_same<T, ff>::value) return cudaErrorNotSupported;
  d.pool = PoolOf<T>::get(c);
  c->rec->descs.push_back(d);
  return cudaSuccess;
}

static PassDesc new_desc(const fcsph_ctx* c, int kind, dim3 grid, size_t smem) {
  PassDesc d;
  memset(&d, 0, sizeof(d));
  d.kind = kind;
  d.gx = (int)grid.x;
  d.gy = (int)grid.y;
  d.gz = (int)grid.z;
  d.smem = smem;
  d.g = c->gd;
  return d;
}

cudaError_t init_kernel_attributes() {
  cudaError_t e = cudaSuccess;
#define FCSPH_RAISE(K)                           \
  if ((e = raise_smem(K)) != cudaSuccess) return e;
  FCSPH_RAISE((k_dft_lines<double, false>))
  FCSPH_RAISE((k_dft_lines<double, true>))
  FCSPH_RAISE((k_dft_lines<float, false>))
  FCSPH_RAISE((k_dft_lines<float, true>))
  FCSPH_RAISE((k_dft_ip<double, double2>))
  FCSPH_RAISE((k_dft_ip<float, float2>))
  FCSPH_RAISE((k_dft_ip<ff, double2>))
  FCSPH_RAISE((k_line_op_r<20, 27, kTeamsLine>))
  FCSPH_RAISE((k_line_op_r<30, 35, kTeamsLine>))
  FCSPH_RAISE((k_line_op_rb<30, 36, 7>))
  FCSPH_RAISE((k_line_op_rb<42, 50, 5>))
  FCSPH_RAISE((k_line_op_rb<30, 36, 1>))
  FCSPH_RAISE((k_line_op_rb<42, 50, 1>))
  FCSPH_RAISE((k_col_fwd_r<20, 27, 1, false>))
  FCSPH_RAISE((k_col_fwd_r<30, 35, 1, false>))
  FCSPH_RAISE((k_col_fwd_r<30, 36, 1, true>))
  FCSPH_RAISE((k_col_fwd_r<42, 50, 1, true>))
  FCSPH_RAISE((k_col_out_r<30, 35, 1, false>))
  FCSPH_RAISE((k_col_out_r<30, 36, 1, true>))
  FCSPH_RAISE((k_col_out_r<42, 50, 1, true>))
  FCSPH_RAISE((k_col_fwd_r<20, 27, 4, false>))
  FCSPH_RAISE((k_col_fwd_r<30, 35, 3, false>))
  FCSPH_RAISE((k_col_fwd_r<30, 36, 7, true>))
  FCSPH_RAISE((k_col_fwd_r<42, 50, 5, true>))
  FCSPH_RAISE((k_col_out_r<20, 27, 4, false>))
  FCSPH_RAISE((k_col_out_r<30, 35, 3, false>))
  FCSPH_RAISE((k_col_out_r<30, 36, 7, true>))
  FCSPH_RAISE((k_col_out_r<42, 50, 5, true>))
#define FCSPH_RAISE_RT(K)                                                                                     \
  if ((e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax - 64)) != \
      cudaSuccess)                                                                                            \
    return e;
  FCSPH_RAISE_RT((k_col_out_rt<20, 27, 1, false>))
  FCSPH_RAISE_RT((k_col_out_rt<30, 35, 3, false>))
  FCSPH_RAISE_RT((k_col_out_rt<30, 36, 7, true>))
  FCSPH_RAISE_RT((k_col_out_rt<42, 50, 5, true>))
  FCSPH_RAISE_RT((k_col_out_rt<30, 35, 1, false>))
  FCSPH_RAISE_RT((k_col_out_rt<30, 36, 1, true>))
  FCSPH_RAISE_RT((k_col_out_rt<42, 50, 1, true>))
#undef FCSPH_RAISE_RT
  FCSPH_RAISE((k_row_sym_w<2>))
  FCSPH_RAISE((k_row_sym_w<4>))
  FCSPH_RAISE((k_row_sym_w<8>))
  FCSPH_RAISE((k_row_sym_w<16>))
  FCSPH_RAISE((k_row_sym_w<32>))
  // the persistent kernel holds two static shared words besides its dynamic
  // shared memory
  for (int rm : {9, 31}) {
    e = with_persist_rm(rm, [](auto w) {
      constexpr int RM = decltype(w)::value;
      const int lim = (int)kSmemMax - 64;
      cudaError_t r = cudaFuncSetAttribute(k_persist<double, RM>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
      if (r != cudaSuccess) return r;
      return cudaFuncSetAttribute(k_persist<ff, RM>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    });
    if (e != cudaSuccess) return e;
  }
  for (int rm : {9, 17, 31}) {
    e = with_rm(rm, [](auto w) {
      constexpr int RM = decltype(w)::value;
      cudaError_t r;
      if ((r = raise_smem(k_col_fwd<double, double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_col_fwd<ff, double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_col_fwd<float, double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_col_fwd<float, float, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_line_op<double, double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_line_op<ff, double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_line_op<float, float, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_row_sym<double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_row_sym<ff, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_row_sym<float, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_row_ppe<double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_row_ppe<ff, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_row_ppe<float, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_col_inv<double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_col_inv<ff, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_col_inv<float, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_zlines<double, RM>)) != cudaSuccess) return r;
      if ((r = raise_smem(k_zlines<ff, RM>)) != cudaSuccess) return r;
      return raise_smem(k_zlines<float, RM>);
    });
    if (e != cudaSuccess) return e;
  }
#undef FCSPH_RAISE
  return cudaSuccess;
}

// Largest dynamic shared memory any FFT kernel of context c needs with
// row_lines rows per row-pass CTA and col_pairs column pairs per column CTA.
size_t tiling_smem(const fcsph_ctx* c, int row_lines, int col_pairs) {
  const size_t cb = c->prec.fft_prec == FCSPH_F32 ? sizeof(float2) : sizeof(double2);
  const size_t row = (c->gd.nz > 1 ? 6 : 4) * (size_t)row_lines * c->plan_x.line_len() * cb;
  const size_t ppe = 2 * (size_t)row_lines * c->plan_px.line_len() * cb;
  const size_t col = (size_t)col_pairs * 2 * (size_t)col_ls(c) * cb;
  size_t m = row > ppe ? row : ppe;
  return m > col ? m : col;
}

size_t tiling_smem_limit() { return kSmemMax; }

cudaError_t launch_fc_extend(fcsph_ctx* c, const void* f, void* fext, int bc) {
  ProfScope ps(c, FCSPH_PROF_OTHER);
  const double* E = c->dE + (bc == FCSPH_NEUMANN ? 1 : 0) * c->gd.n_cont * 2 * c->gd.n_match;
  const int blocks = 152 * 8;
  if (c->prec.fft_prec != FCSPH_F32) {  // double fields (F64, F32X2)
    k_fc_extend_y<double><<<blocks, kThreads, 0, c->stream>>>(c->gd, (const double*)f, (double*)fext, E);
    c->launches++;
    if (c->gd.x_walls) {
      k_fc_extend_x<double><<<blocks, kThreads, 0, c->stream>>>(c->gd, (double*)fext, E);
      c->launches++;
    }
  } else {
    k_fc_extend_y<float><<<blocks, kThreads, 0, c->stream>>>(c->gd, (const float*)f, (float*)fext, E);
    c->launches++;
    if (c->gd.x_walls) {
      k_fc_extend_x<float><<<blocks, kThreads, 0, c->stream>>>(c->gd, (float*)fext, E);
      c->launches++;
    }
  }
  return cudaGetLastError();
}


// Register column FFT for FP32 contexts: the split n = N1 N2 of the extended
// wall-normal length when the plan is direct and the length is one of the
// supported ones, else 0.
int col_r_split(const fcsph_ctx* c) {
  const FftPlan& P = c->plan_y;
  if (c->prec.fft_prec != FCSPH_F32 || P.bs || P.rd) return 0;
  switch (P.base.n) {
    case 540: return 20;
    case 1050: return 30;
    default: return 0;
  }
}

// Register Bluestein column FFT for FP32 contexts: the split N1 of the
// Bluestein length m (1080 = 30 x 36, 2100 = 42 x 50) of the extended
// wall-normal length, else 0.
int col_rb_split(const fcsph_ctx* c) {
  const FftPlan& P = c->plan_y;
  if (c->prec.fft_prec != FCSPH_F32 || !P.bs) return 0;
  switch (P.sub.n) {
    case 1080: return 30;
    case 2100: return 42;
    default: return 0;
  }
}

// Whether a register pass over ncol columns of each of `sets` fields and instances
// takes one team per CTA rather than NP: while an SM gets at most four such CTAs
// (n = 540 forward, 128 pairs, 10.1 -> 8.6 us, 512 pairs 10.2 packed and 10.5; n = 1050
// output, 512 pairs, 16.4 -> 14.7, 640 pairs 16.4 either way).  Chirp-z lengths hold
// four CTAs of one team per SM (64 threads of up to 255 registers) or one of NP (256
// of them), and a wave of either takes about as long: whichever needs fewer waves,
// one on a tie (line operator at n = 537: up to 512 pairs 34.8 -> 28.7 us, 640 pairs
// 35.0 packed and 47.2; n = 1049: 512 pairs 63.8 -> 53.3, 640 pairs 64.7 and 104.6,
// 1536 pairs 186 -> 154).
static bool one_team(long long ncol, long long sets, int NP, bool chirp) {
  const long long one = (ncol + 1) / 2 * sets, packed = (ncol + 2 * NP - 1) / (2 * NP) * sets;
  return one <= 4 * 152 || (chirp && (one + 4 * 152 - 1) / (4 * 152) <= (packed + 151) / 152);
}

template <int N1, int N2, int NP, bool BS>
static cudaError_t col_fwd_r(fcsph_ctx* c, int nf, const void* const* fields, int bc, void* spec) {
  if constexpr (NP > 1)
    if (one_team(c->gd.ncol, (long long)nf * c->gd.nb, NP, BS)) return col_fwd_r<N1, N2, 1, BS>(c, nf, fields, bc, spec);
  typedef TeamFFT<N1, N2> TF;
  const GridDev& g = c->gd;
  const FftPlan& P = c->plan_y;
  const size_t smem = (size_t)NP * TF::LINE * sizeof(float2);
  const auto* E = static_cast<const typename FcTab<float>::t*>(fc_table(c, FCSPH_F32, bc));
  dim3 grid((g.ncol + 2 * NP - 1) / (2 * NP), nf, g.nb);
  const size_t fstride = (size_t)g.rows * g.ncol;
  const size_t bstride = spec_in_fields(c) * fstride;
  ProfScope ps(c, FCSPH_PROF_COL_FWD);
  const float* f0 = (const float*)fields[0];
  k_col_fwd_r<N1, N2, NP, BS><<<grid, TF::threads(NP), smem, c->stream>>>(
      g, f0, (const float*)(nf > 1 ? fields[1] : fields[0]), (const float*)(nf > 2 ? fields[2] : fields[0]), E,
      c->pool32 + P.chirp, c->pool32 + P.bhat, c->pool32 + c->tw_team, (float2*)spec, fstride, bstride);
  c->launches++;
  return cudaGetLastError();
}

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// The TMA column-output pass: needs an even number of columns (16-byte rows
// of the tensor map and 16-byte aligned pair coordinates), a 16-byte aligned
// spectrum buffer and no instance mask; returns cudaErrorNotSupported
// otherwise (the caller then runs k_col_out_r).
template <int N1, int N2, int NP, bool BS>
static cudaError_t col_out_rt(fcsph_ctx* c, const void* spec, int nout, EpiArgs& ea) {
  if constexpr (NP > 1)
    if (one_team(c->gd.ncol, c->gd.nb, NP, BS)) return col_out_rt<N1, N2, 1, BS>(c, spec, nout, ea);
  typedef TeamFFT<N1, N2> TF;
  const GridDev& g = c->gd;
  EncodeTiledFn enc = encode_tiled();
  if (!enc || g.ncol % 2 || ((uintptr_t)spec & 15) || g.active) return cudaErrorNotSupported;
  const int nfo = spec_out_fields(c);
  const int nbox = (g.hy + 255) / 256;
  const int rows_box = ((g.hy + nbox - 1) / nbox + 7) / 8 * 8;
  CUtensorMap map;
  const cuuint64_t dims[2] = {(cuuint64_t)2 * g.ncol, (cuuint64_t)g.batch * nfo * g.rows};
  const cuuint64_t strides[1] = {(cuuint64_t)2 * g.ncol * sizeof(float)};
  const cuuint32_t box[2] = {4 * NP, (cuuint32_t)rows_box};
  const cuuint32_t es[2] = {1, 1};
  if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(spec), dims, strides, box, es,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorNotSupported;
  const size_t smem = 128 + (size_t)nbox * rows_box * 16 * NP + (size_t)NP * TF::LINE * sizeof(float2);
  cudaError_t e = check_smem(smem + 64);
  if (e != cudaSuccess) return cudaErrorNotSupported;
  int dev = 0, sms = 0, occ = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_col_out_rt<N1, N2, NP, BS>, TF::threads(NP), smem)) !=
          cudaSuccess)
    return e;
  const int ngroups = (g.ncol + 2 * NP - 1) / (2 * NP);
  const long long W = (long long)g.nb * ngroups;
  const long long grid = std::min<long long>(W, (long long)sms * (occ > 0 ? occ : 1));
  ea.status = c->dstatus;
  ProfScope ps(c, FCSPH_PROF_COL_OUT);
  const FftPlan& P = c->plan_y;
  k_col_out_rt<N1, N2, NP, BS><<<(unsigned)grid, TF::threads(NP), smem, c->stream>>>(
      g, map, rows_box, nbox, nfo, nout, ea, c->pool32 + c->tw_team, ngroups, BS ? c->pool32 + P.chirp : nullptr,
      BS ? c->pool32 + P.bhat : nullptr);
  c->launches++;
  return cudaGetLastError();
}

template <int N1, int N2, int NP, bool BS>
static cudaError_t col_out_r(fcsph_ctx* c, const void* spec, int nout, EpiArgs& ea) {
  // at n = 540 the gather of four pairs is the better one at any count (128 pairs 14.4 us, one by one 15.3)
  if constexpr (NP > 1 && N1 != 20)
    if (one_team(c->gd.ncol, c->gd.nb, NP, BS)) return col_out_r<N1, N2, 1, BS>(c, spec, nout, ea);
  typedef TeamFFT<N1, N2> TF;
  const GridDev& g = c->gd;
  const FftPlan& P = c->plan_y;
  const size_t smem = (size_t)NP * TF::LINE * sizeof(float2);
  const size_t fs = (size_t)g.rows * g.ncol;
  dim3 grid((g.ncol + 2 * NP - 1) / (2 * NP), g.nb);
  ProfScope ps(c, FCSPH_PROF_COL_OUT);
  k_col_out_r<N1, N2, NP, BS><<<grid, TF::threads(NP), smem, c->stream>>>(
      g, (const float2*)spec, fs, spec_out_fields(c) * fs, nout, ea, c->pool32 + P.chirp, c->pool32 + P.bhat,
      c->pool32 + c->tw_team);
  c->launches++;
  return cudaGetLastError();
}

template <typename T, typename U>
static cudaError_t col_fwd_t(fcsph_ctx* c, int prec, int nf, const void* const* fields, int bc, void* spec, int dct) {
  const GridDev& g = c->gd;
  if constexpr (sizeof(T) == sizeof(float) && sizeof(U) == sizeof(float)) {
    if (!dct) {
      switch (col_r_split(c)) {
        case 20: return col_fwd_r<20, 27, 4, false>(c, nf, fields, bc, spec);
        case 30: return col_fwd_r<30, 35, 3, false>(c, nf, fields, bc, spec);
        default: break;
      }
      switch (col_rb_split(c)) {
        case 30: return col_fwd_r<30, 36, 7, true>(c, nf, fields, bc, spec);
        case 42: return col_fwd_r<42, 50, 5, true>(c, nf, fields, bc, spec);
        default: break;
      }
    }
  }
  IpPlan P = dct ? c->ip_py : c->ip_y;
  const int ls = ip_ls<T>(P);
  const Shape sh = pass_shape(c, false, (long long)((g.ncol + 1) / 2) * nf * g.nb, P.m, 1, 1, ls * sizeof(typename CT<T>::t));
  const int Pp = sh.u;
  // what a pass accepts is the size rule of fcsph_set_tiling (two lines per pair)
  cudaError_t e = check_smem(2 * (size_t)(dct ? c->plan_py : c->plan_y).line_len() * sizeof(typename CT<T>::t) * Pp);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)(Pp + P.big) * ls * sizeof(typename CT<T>::t);
  const auto* E = static_cast<const typename FcTab<T>::t*>(fc_table(c, prec, bc));
  dim3 grid((g.ncol + 2 * Pp - 1) / (2 * Pp), nf, g.nb);
  P = launch_plan<T>(c, P, (long long)grid.x * grid.y * grid.z);
  const size_t fstride = (size_t)g.rows * g.ncol;
  const size_t bstride = (dct ? 1 : spec_in_fields(c)) * fstride;
  if (c->rec) {
    if (!std::is_same<U, double>::value) return cudaErrorNotSupported;
    PassDesc d = new_desc(c, PK_COL_FWD, grid, smem);
    d.Pp = Pp;
    d.ls = ls;
    d.P = P;
    d.E = E;
    for (int k = 0; k < 3; ++k) d.f[k] = fields[k < nf ? k : 0];
    d.dct = dct;
    d.spec = spec;
    d.fstride = fstride;
    d.bstride = bstride;
    return rec_push<T>(c, d);
  }
  ProfScope ps(c, FCSPH_PROF_COL_FWD);
  return with_rm(P.rmax, [&](auto w) {
    constexpr int RM = decltype(w)::value;
    k_col_fwd<T, U, RM><<<grid, sh.nt, smem, c->stream>>>(g, (const U*)fields[0],
                                                       (const U*)(nf > 1 ? fields[1] : fields[0]),
                                                       (const U*)(nf > 2 ? fields[2] : fields[0]), E, P,
                                                       PoolOf<T>::get(c), dct, (typename CT<T>::t*)spec, fstride,
                                                       bstride, Pp, ls);
    c->launches++;
    return cudaGetLastError();
  });
}

cudaError_t launch_col_fwd(fcsph_ctx* c, int prec, int nf, const void* const* fields, int fields_double, int bc,
                           void* spec, int dct) {
  if (prec == FCSPH_F64) {
    if (!fields_double) return cudaErrorInvalidValue;
    return col_fwd_t<double, double>(c, prec, nf, fields, bc, spec, dct);
  }
  if (prec == FCSPH_F32X2) {
    if (!fields_double) return cudaErrorInvalidValue;
    return col_fwd_t<ff, double>(c, prec, nf, fields, bc, spec, dct);
  }
  if (fields_double) return col_fwd_t<float, double>(c, prec, nf, fields, bc, spec, dct);
  return col_fwd_t<float, float>(c, prec, nf, fields, bc, spec, dct);
}

// Shared memory of k_row_sym_w: per warp the exchange block and nin spectra.
size_t row_w_smem(int nin) { return 4 * ((size_t)kWarpXchgFloats + (size_t)nin * 2 * 32 * 32) * sizeof(float); }

// M = mx / 32 when the FP32 row pass can take the register FFT (periodic x,
// direct plan, mx = 32 M with M a power of two in 2 .. 32), else 0.
int row_w_m(const fcsph_ctx* c) {
  const GridDev& g = c->gd;
  if (c->prec.fft_prec != FCSPH_F32 || g.x_walls || g.mx != g.nx || c->plan_x.bs || c->plan_x.rd) return 0;
  for (int m = 2; m <= 32; m *= 2)
    if (g.mx == 32 * m) return m;
  return 0;
}

template <int M>
static cudaError_t row_sym_w(fcsph_ctx* c, const void* sp_in, void* sp_out, const RowOps& ops, double scale, int kind) {
  const GridDev& g = c->gd;
  const size_t smem = row_w_smem(ops.nin);
  cudaError_t e = check_smem(smem);
  if (e != cudaSuccess) return e;
  constexpr int rows_per_cta = 4 * (32 / M);
  dim3 grid((g.hy * g.nz + rows_per_cta - 1) / rows_per_cta, g.nb);
  const size_t fs = (size_t)g.rows * g.ncol;
  ProfScope ps(c, kind);
  k_row_sym_w<M><<<grid, 128, smem, c->stream>>>(g, (const float2*)sp_in, (float2*)sp_out, fs, spec_in_fields(c) * fs,
                                                 fs, spec_out_fields(c) * fs, ops, c->pool32 + c->tw_row,
                                                 static_cast<const float*>(c->dW), scale);
  c->launches++;
  return cudaGetLastError();
}

template <typename T>
static cudaError_t row_sym_t(fcsph_ctx* c, int prec, const void* sp_in, void* sp_out, const RowOps& ops, double scale,
                             int bc, int kind) {
  const GridDev& g = c->gd;
  if (prec == FCSPH_F32) {
    switch (row_w_m(c)) {
      case 2: return row_sym_w<2>(c, sp_in, sp_out, ops, scale, kind);
      case 4: return row_sym_w<4>(c, sp_in, sp_out, ops, scale, kind);
      case 8: return row_sym_w<8>(c, sp_in, sp_out, ops, scale, kind);
      case 16: return row_sym_w<16>(c, sp_in, sp_out, ops, scale, kind);
      case 32: return row_sym_w<32>(c, sp_in, sp_out, ops, scale, kind);
      default: break;
    }
  }
  IpPlan P = c->ip_x;
  const size_t cb = sizeof(typename CT<T>::t);
  const int ls = ip_ls<T>(P);
  const int nin = ops.split > 1 ? 1 : ops.nin, nout = ops.nout / (ops.split > 1 ? ops.split : 1);
  const Shape sh = pass_shape(c, true, (long long)g.hy * g.nz * g.nb * (ops.split > 1 ? ops.split : 1), P.m,
                              std::min(nout, 3), nin + 1, ls * cb);
  const int Rr = sh.u;
  cudaError_t e = check_smem((size_t)(2 * ops.nin + (ops.nin == 1 ? 1 : 0)) * Rr * c->plan_x.line_len() * cb);
  if (e != cudaSuccess) return e;
  const int ob = fit_group(std::min(nout, 3), nin * Rr + P.big, Rr, ls * cb, sh.nt);
  const size_t smem = (size_t)((nin + ob) * Rr + P.big) * ls * cb;
  const auto* E = static_cast<const typename FcTab<T>::t*>(fc_table(c, prec, bc));
  const size_t fs = (size_t)g.rows * g.ncol;
  dim3 grid((g.hy * g.nz + Rr - 1) / Rr, g.nb, ops.split > 1 ? ops.split : 1);
  P = launch_plan<T>(c, P, (long long)grid.x * grid.y * grid.z);
  if (c->rec) {
    PassDesc d = new_desc(c, PK_ROW_SYM, grid, smem);
    d.Rr = Rr;
    d.ob = ob;
    d.ls = ls;
    d.P = P;
    d.E = E;
    d.sp_in = sp_in;
    d.sp_out = sp_out;
    d.fs_in = fs;
    d.bs_in = spec_in_fields(c) * fs;
    d.fs_out = fs;
    d.bs_out = spec_out_fields(c) * fs;
    d.ops = ops;
    d.W = c->dW;
    d.scale = scale;
    return rec_push<T>(c, d);
  }
  ProfScope ps(c, kind);
  return with_rm(P.rmax, [&](auto w) {
    constexpr int RM = decltype(w)::value;
    k_row_sym<T, RM><<<grid, sh.nt, smem, c->stream>>>(g, (const typename CT<T>::t*)sp_in, (typename CT<T>::t*)sp_out,
                                                    fs, spec_in_fields(c) * fs, fs, spec_out_fields(c) * fs, ops, E, P,
                                                    PoolOf<T>::get(c), static_cast<const T*>(c->dW), scale, Rr, ob, ls);
    c->launches++;
    return cudaGetLastError();
  });
}

// One launch for any number of outputs: they are formed and inverted up to three
// at a time (fit_group), so shared memory does not grow with them.
cudaError_t launch_row_sym(fcsph_ctx* c, int prec, const void* sp_in, void* sp_out, const RowOps& ops, double scale,
                           int bc, int kind) {
  if (prec == FCSPH_F64) return row_sym_t<double>(c, prec, sp_in, sp_out, ops, scale, bc, kind);
  if (prec == FCSPH_F32X2) return row_sym_t<ff>(c, prec, sp_in, sp_out, ops, scale, bc, kind);
  return row_sym_t<float>(c, prec, sp_in, sp_out, ops, scale, bc, kind);
}

template <int N1, int N2, int NP>
static cudaError_t line_op_r(fcsph_ctx* c, const void* f, const LineOuts& lo, int bc) {
  typedef TeamFFT<N1, N2> TF;
  const GridDev& g = c->gd;
  const size_t smem = (size_t)NP * (N1 * N2 + TF::XCHG) * sizeof(float2);
  const long long ncols = (long long)g.batch * g.ncol;
  const auto* E = static_cast<const typename FcTab<float>::t*>(fc_table(c, FCSPH_F32, bc));
  ProfScope ps(c, FCSPH_PROF_COL_OUT);
  k_line_op_r<N1, N2, NP><<<(unsigned)((ncols + 2 * NP - 1) / (2 * NP)), TF::threads(NP), smem, c->stream>>>(
      g, (const float*)f, ncols, E, c->pool32, c->pool32 + c->tw_team, lo);
  c->launches++;
  return cudaGetLastError();
}

template <int N1, int N2, int NP>
static cudaError_t line_op_rb(fcsph_ctx* c, const void* f, const LineOuts& lo, int bc) {
  if constexpr (NP > 1)
    if (one_team((long long)c->gd.batch * c->gd.ncol, 1, NP, true)) return line_op_rb<N1, N2, 1>(c, f, lo, bc);
  typedef TeamFFT<N1, N2> TF;
  const GridDev& g = c->gd;
  const FftPlan& P = c->plan_y;
  const size_t smem = 2 * (size_t)NP * TF::LINE * sizeof(float2);
  const long long ncols = (long long)g.batch * g.ncol;
  const auto* E = static_cast<const typename FcTab<float>::t*>(fc_table(c, FCSPH_F32, bc));
  ProfScope ps(c, FCSPH_PROF_COL_OUT);
  k_line_op_rb<N1, N2, NP><<<(unsigned)((ncols + 2 * NP - 1) / (2 * NP)), TF::threads(NP), smem, c->stream>>>(
      g, (const float*)f, ncols, E, c->pool32, c->pool32 + P.chirp, c->pool32 + P.bhat, c->pool32 + c->tw_team, lo);
  c->launches++;
  return cudaGetLastError();
}

template <typename T, typename U>
static cudaError_t line_op_t(fcsph_ctx* c, int prec, const void* f, const int* ops, int nout, int bc, void* const* outs) {
  const GridDev& g = c->gd;
  if constexpr (sizeof(T) == sizeof(float) && sizeof(U) == sizeof(float)) {
    const int split = col_r_split(c);
    if (split) {
      LineOuts lo;
      memset(&lo, 0, sizeof(lo));
      lo.nout = nout;
      for (int o = 0; o < nout; ++o) {
        lo.op[o] = ops[o];
        lo.out[o] = outs[o];
      }
      if (split == 20) return line_op_r<20, 27, kTeamsLine>(c, f, lo, bc);
      if (split == 30) return line_op_r<30, 35, kTeamsLine>(c, f, lo, bc);
    }
    const int bsplit = col_rb_split(c);
    if (bsplit) {
      LineOuts lo;
      memset(&lo, 0, sizeof(lo));
      lo.nout = nout;
      for (int o = 0; o < nout; ++o) {
        lo.op[o] = ops[o];
        lo.out[o] = outs[o];
      }
      if (bsplit == 30) return line_op_rb<30, 36, 7>(c, f, lo, bc);
      if (bsplit == 42) return line_op_rb<42, 50, 5>(c, f, lo, bc);
    }
  }
  IpPlan P = c->ip_y;
  const size_t cb = sizeof(typename CT<T>::t);
  const int ls = ip_ls<T>(P);
  const Shape sh = pass_shape(c, false, (long long)((g.ncol + 1) / 2) * g.batch, P.m, nout, 2, ls * cb);
  const int Pp = sh.u;
  cudaError_t e = check_smem(3 * (size_t)Pp * c->plan_y.line_len() * cb);
  if (e != cudaSuccess) return e;
  const long long ncols = (long long)g.batch * g.ncol;
  const long long blocks = (ncols + 2 * Pp - 1) / (2 * Pp);
  P = launch_plan<T>(c, P, blocks);
  const int ob = fit_group(nout, Pp + P.big, Pp, ls * cb, sh.nt);
  const size_t smem = (size_t)((1 + ob) * Pp + P.big) * ls * cb;
  LineOuts lo;
  memset(&lo, 0, sizeof(lo));
  lo.nout = nout;
  for (int o = 0; o < nout; ++o) {
    lo.op[o] = ops[o];
    lo.out[o] = outs[o];
  }
  const auto* E = static_cast<const typename FcTab<T>::t*>(fc_table(c, prec, bc));
  ProfScope ps(c, FCSPH_PROF_COL_OUT);
  return with_rm(P.rmax, [&](auto w) {
    constexpr int RM = decltype(w)::value;
    k_line_op<T, U, RM><<<(unsigned)blocks, sh.nt, smem, c->stream>>>(g, (const U*)f, ncols, E, P, PoolOf<T>::get(c),
                                                                   lo, Pp, ob, ls);
    c->launches++;
    return cudaGetLastError();
  });
}

cudaError_t launch_line_op(fcsph_ctx* c, const void* f, const int* ops, int nout, int bc, void* const* outs) {
  const int prec = c->prec.fft_prec;
  if (prec == FCSPH_F64) return line_op_t<double, double>(c, prec, f, ops, nout, bc, outs);
  if (prec == FCSPH_F32X2) return line_op_t<ff, double>(c, prec, f, ops, nout, bc, outs);
  return line_op_t<float, float>(c, prec, f, ops, nout, bc, outs);
}

template <typename T>
static cudaError_t zpass_t(fcsph_ctx* c, void* spec, int nf, size_t bstride, int rows_used, int inv) {
  const GridDev& g = c->gd;
  IpPlan P = c->ip_z;
  const int ls = ip_ls<T>(P);
  int L = 256 / g.nz;
  if (L < 1) L = 1;
  if (L > 8) L = 8;
  cudaError_t e = check_smem(2 * (size_t)L * c->plan_z.line_len() * sizeof(typename CT<T>::t));
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)(L + P.big) * ls * sizeof(typename CT<T>::t);
  const int lines = rows_used * g.nx;
  dim3 grid((lines + L - 1) / L, nf, g.nb);
  P = launch_plan<T>(c, P, (long long)grid.x * grid.y * grid.z);
  ProfScope ps(c, FCSPH_PROF_OTHER);
  return with_rm(P.rmax, [&](auto w) {
    constexpr int RM = decltype(w)::value;
    k_zlines<T, RM><<<grid, c->row_threads, smem, c->stream>>>((typename CT<T>::t*)spec, lines, (size_t)g.rows * g.ncol, bstride,
                                                   P, PoolOf<T>::get(c), L, ls, inv, g.active, g.b0);
    c->launches++;
    return cudaGetLastError();
  });
}

// 3D: z transforms of nf fields of every instance (fields 0..nf-1 of the
// buffer, instance stride bstride, rows_used spectrum rows each); no-op in 2D.
cudaError_t launch_zpass(fcsph_ctx* c, int prec, void* spec, int nf, size_t bstride, int rows_used, int inv) {
  if (c->gd.nz <= 1 || nf <= 0) return cudaSuccess;
  if (prec == FCSPH_F64) return zpass_t<double>(c, spec, nf, bstride, rows_used, inv);
  if (prec == FCSPH_F32X2) return zpass_t<ff>(c, spec, nf, bstride, rows_used, inv);
  return zpass_t<float>(c, spec, nf, bstride, rows_used, inv);
}

template <typename T>
static cudaError_t col_inv_common(fcsph_ctx* c, int epi, const void* spec, int nout, EpiArgs& ea) {
  if (epi < EPI_OUT || epi > EPI_PPE_ADD) return cudaErrorInvalidValue;
  // the components of a momentum pass, or of a correction that transforms them at all, are all transformed
  if (nout < 1 || ea.fwd_nf > 3 || (epi == EPI_MOM && nout != ea.fwd_nf * ea.mom_terms) ||
      (epi == EPI_CORR && ea.fwd_nf > 0 && nout != ea.fwd_nf))
    return cudaErrorInvalidValue;
  // the fused forward of a PPE pass reads the FP64 potential
  if (ea.fwd_nf > 0 && (epi == EPI_PPE_SOLVE || epi == EPI_PPE_ADD) && ea.phi == nullptr) return cudaErrorInvalidValue;
  if (ea.fwd_nf > 0 && (epi == EPI_OUT || epi == EPI_PPE_RESID)) return cudaErrorInvalidValue;
  const GridDev& g = c->gd;
  IpPlan P = epi >= EPI_PPE_SOLVE ? c->ip_py : c->ip_y;
  // lines sized for the inverse plan and the fused forward's plan
  const size_t cb = sizeof(typename CT<T>::t);
  int ls = ip_ls<T>(P), old_ls = (epi >= EPI_PPE_SOLVE ? c->plan_py : c->plan_y).line_len();
  int big = P.big, rmax = P.rmax;
  if (ea.fwd_nf > 0) {
    const FftPlan& F = ea.fwd_dct ? c->plan_py : c->plan_y;
    ls = std::max(ls, ip_ls<T>(ea.fwdP));
    old_ls = std::max(old_ls, F.line_len());
    big |= ea.fwdP.big;
    rmax = std::max(rmax, ea.fwdP.rmax);
  }
  const Shape sh = pass_shape(c, false, (long long)((g.ncol + 1) / 2) * g.nb, std::max(P.m, ea.fwd_nf > 0 ? ea.fwdP.m : 0),
                              std::min(nout, 3), 1, ls * cb);
  const int Pp = sh.u;
  // Up to two CTAs per SM each velocity component of the momentum and
  // correction passes is a CTA of its own (the components share nothing but the
  // loads of the velocity; a single 64^2 solve has 32 column pairs for 152 SMs:
  // momentum pass in FP64 86 -> 60 us)
  const long long ctas = (long long)((g.ncol + 2 * Pp - 1) / (2 * Pp)) * g.nb;
  const int comps = epi == EPI_MOM ? ea.fwd_nf : epi == EPI_CORR ? nout : 1;
  const int nparts = !c->rec && ctas <= 152 ? comps : 1;
  const int want = epi == EPI_MOM ? ea.mom_terms
                                  : std::min(3, std::max((nout + nparts - 1) / nparts, nparts > 1 ? 1 : ea.fwd_nf));
  const int og = fit_group(want, big, Pp, ls * cb, sh.nt);
  // the lines only: FP64 values kept across outputs stay in global memory
  const size_t smem = (size_t)(og * Pp + big) * ls * cb;
  const size_t fs = (size_t)g.rows * g.ncol;
  const size_t bs = (epi >= EPI_PPE_SOLVE ? 1 : spec_out_fields(c)) * fs;  // spec_ppe or spec_out
  dim3 grid((g.ncol + 2 * Pp - 1) / (2 * Pp), g.nb, nparts);
  P = launch_plan<T>(c, P, ctas * nparts);
  ea.fwdP = launch_plan<T>(c, ea.fwdP, ctas * nparts);
  const typename CT<T>::t* pool = PoolOf<T>::get(c);
  ea.status = c->dstatus;
  cudaError_t e = check_smem((size_t)2 * old_ls * cb * Pp);
  if (e != cudaSuccess) return e;
  if (c->rec) {
    PassDesc d = new_desc(c, PK_COL_INV, grid, smem);
    d.Pp = Pp;
    d.og = og;
    d.ls = ls;
    d.P = P;
    d.spec = const_cast<void*>(spec);
    d.fstride = fs;
    d.bstride = bs;
    d.nout = nout;
    d.epi = epi;
    d.ea = ea;
    return rec_push<T>(c, d);
  }
  static const int kinds[7] = {FCSPH_PROF_COL_OUT, FCSPH_PROF_COL_MOM, FCSPH_PROF_COL_DIV, FCSPH_PROF_COL_CORR,
                               FCSPH_PROF_COL_PPE, FCSPH_PROF_COL_PPE, FCSPH_PROF_COL_PPE};
  ProfScope ps(c, kinds[epi]);
  return with_rm(rmax, [&](auto w) {
    constexpr int RM = decltype(w)::value;
    k_col_inv<T, RM><<<grid, sh.nt, smem, c->stream>>>(g, (const typename CT<T>::t*)spec, fs, bs, nout, P, pool,
                                                    ea, Pp, og, ls, epi);
    c->launches++;
    return cudaGetLastError();
  });
}

static cudaError_t col_inv(fcsph_ctx* c, int prec, int epi, const void* spec, int nout, EpiArgs& ea) {
  if (prec == FCSPH_F64) return col_inv_common<double>(c, epi, spec, nout, ea);
  if (prec == FCSPH_F32X2) return col_inv_common<ff>(c, epi, spec, nout, ea);
  return col_inv_common<float>(c, epi, spec, nout, ea);
}

static EpiArgs epi_defaults() {
  EpiArgs ea;
  memset(&ea, 0, sizeof(ea));
  return ea;
}

cudaError_t launch_col_out(fcsph_ctx* c, const void* spec, int nout, void* const* outs) {
  EpiArgs ea = epi_defaults();
  for (int o = 0; o < nout; ++o) ea.outs[o] = outs[o];
  ea.out_double = c->prec.fft_prec != FCSPH_F32;
  if (!ea.out_double) {
    cudaError_t e = cudaErrorNotSupported;
    switch (col_r_split(c)) {
      case 20:
        if (c->tma) e = col_out_rt<20, 27, 1, false>(c, spec, nout, ea);
        return e == cudaErrorNotSupported ? col_out_r<20, 27, 4, false>(c, spec, nout, ea) : e;
      case 30:
        if (c->tma) e = col_out_rt<30, 35, 3, false>(c, spec, nout, ea);
        return e == cudaErrorNotSupported ? col_out_r<30, 35, 3, false>(c, spec, nout, ea) : e;
      default: break;
    }
    switch (col_rb_split(c)) {
      case 30:
        if (c->tma) e = col_out_rt<30, 36, 7, true>(c, spec, nout, ea);
        return e == cudaErrorNotSupported ? col_out_r<30, 36, 7, true>(c, spec, nout, ea) : e;
      case 42:
        if (c->tma) e = col_out_rt<42, 50, 5, true>(c, spec, nout, ea);
        return e == cudaErrorNotSupported ? col_out_r<42, 50, 5, true>(c, spec, nout, ea) : e;
      default: break;
    }
  }
  return col_inv(c, c->prec.fft_prec, EPI_OUT, spec, nout, ea);
}

template <typename T>
static cudaError_t row_ppe_t(fcsph_ctx* c, void* spec, int apply) {
  const GridDev& g = c->gd;
  IpPlan P = c->ip_px;
  const size_t cb = sizeof(typename CT<T>::t);
  const int ls = ip_ls<T>(P);
  const Shape sh = pass_shape(c, true, (long long)g.ny * g.nz * g.nb, P.m, 1, 2, ls * cb);
  int Rr = sh.u;
  cudaError_t e = check_smem(2 * (size_t)c->plan_px.line_len() * cb * Rr);
  if (e != cudaSuccess) return e;
  // whole 128-byte blocks and the scratch line can pass the limit the plain
  // lines just kept: fewer rows per CTA then (the result does not depend on it)
  while (Rr > 1 && (size_t)(2 * Rr + P.big) * ls * cb > kSmemMax) --Rr;
  const size_t smem = (size_t)(2 * Rr + P.big) * ls * cb;
  if ((e = check_smem(smem)) != cudaSuccess) return e;
  dim3 grid((g.ny * g.nz + Rr - 1) / Rr, g.nb);
  P = launch_plan<T>(c, P, (long long)grid.x * grid.y);
  if (c->rec) {
    PassDesc d = new_desc(c, PK_ROW_PPE, grid, smem);
    d.Rr = Rr;
    d.ls = ls;
    d.P = P;
    d.spec = spec;
    d.bstride = (size_t)g.rows * g.ncol;
    d.apply = apply;
    return rec_push<T>(c, d);
  }
  ProfScope ps(c, FCSPH_PROF_ROW_PPE);
  return with_rm(P.rmax, [&](auto w) {
    constexpr int RM = decltype(w)::value;
    k_row_ppe<T, RM><<<grid, sh.nt, smem, c->stream>>>(g, (typename CT<T>::t*)spec, (size_t)g.rows * g.ncol, P,
                                                    PoolOf<T>::get(c), apply, Rr, ls);
    c->launches++;
    return cudaGetLastError();
  });
}

cudaError_t launch_row_ppe(fcsph_ctx* c, int prec, void* spec, int apply) {
  if (prec == FCSPH_F64) return row_ppe_t<double>(c, spec, apply);
  if (prec == FCSPH_F32X2) return row_ppe_t<ff>(c, spec, apply);
  return row_ppe_t<float>(c, spec, apply);
}

// mode: 0 solve (phi out, optional Neumann-FC forward), 1 residual r = rhs - L phi into `phi`
// (double), 2 accumulate phi += value (double).
cudaError_t launch_col_ppe_inv(fcsph_ctx* c, int prec, const void* spec, void* phi, int phi_double, double* phi64,
                               int mode, const double* rhs, int neumann_fwd, void* spec_fwd) {
  EpiArgs ea = epi_defaults();
  int epi = EPI_PPE_SOLVE;
  if (mode == 0) {
    ea.phi_any = phi;
    ea.phi_double = phi_double;
    ea.phi = phi64;
  } else if (mode == 1) {
    epi = EPI_PPE_RESID;
    ea.phi = (double*)phi;
    ea.bvec = (double*)rhs;
  } else {
    epi = EPI_PPE_ADD;
    ea.phi = (double*)phi;
  }
  if (neumann_fwd) {
    ea.fwd_nf = 1;
    ea.fwd_dct = 0;
    ea.fwdE = fc_table(c, prec, FCSPH_NEUMANN);
    ea.fwdP = c->ip_y;
    ea.fwd_spec = spec_fwd;
    ea.fwd_fstride = (size_t)c->gd.rows * c->gd.ncol;
    ea.fwd_bstride = spec_in_fields(c) * ea.fwd_fstride;
  }
  return col_inv(c, prec, epi, spec, 1, ea);
}

cudaError_t launch_step_mom(fcsph_ctx* c, const StepDev& s, const void* spec_mom, const double* const* vel,
                            double* const* Fp, double* const* vs, void* spec_next) {
  const int nc = c->gd.nz > 1 ? 3 : 2;
  EpiArgs ea = epi_defaults();
  for (int q = 0; q < nc; ++q) {
    ea.vel[q] = vel[q];
    ea.Fp[q] = Fp[q];
    ea.vs[q] = vs[q];
  }
  ea.mom_terms = nc + 1;
  ea.s = s;
  ea.fwd_nf = nc;
  ea.fwd_dct = 0;
  ea.fwdE = fc_table(c, c->prec.fft_prec, FCSPH_DIRICHLET);
  ea.fwdP = c->ip_y;
  ea.fwd_spec = spec_next;
  ea.fwd_fstride = (size_t)c->gd.rows * c->gd.ncol;
  ea.fwd_bstride = nc * ea.fwd_fstride;
  return col_inv(c, c->prec.fft_prec, EPI_MOM, spec_mom, nc * (nc + 1), ea);
}

cudaError_t launch_step_div(fcsph_ctx* c, const StepDev& s, const void* spec1, double* b, void* spec_dct) {
  EpiArgs ea = epi_defaults();
  ea.bvec = b;
  ea.s = s;
  ea.fwd_nf = 1;
  ea.fwd_dct = 1;
  ea.fwdE = fc_table(c, c->prec.fft_prec, FCSPH_DIRICHLET);
  ea.fwdP = c->ip_py;
  ea.fwd_spec = spec_dct;
  ea.fwd_fstride = (size_t)c->gd.rows * c->gd.ncol;
  ea.fwd_bstride = ea.fwd_fstride;
  return col_inv(c, c->prec.fft_prec, EPI_DIV, spec1, 1, ea);
}

cudaError_t launch_step_corr(fcsph_ctx* c, const StepDev& s, const void* spec_grad, double* const* vs,
                             double* const* vo, void* spec_next) {
  const int nc = c->gd.nz > 1 ? 3 : 2;
  EpiArgs ea = epi_defaults();
  for (int q = 0; q < nc; ++q) {
    ea.vs[q] = vs[q];
    ea.vo[q] = vo[q];
  }
  ea.s = s;
  if (spec_next) {
    ea.fwd_nf = nc;
    ea.fwd_dct = 0;
    ea.fwdE = fc_table(c, c->prec.fft_prec, FCSPH_DIRICHLET);
    ea.fwdP = c->ip_y;
    ea.fwd_spec = spec_next;
    ea.fwd_fstride = (size_t)c->gd.rows * c->gd.ncol;
    ea.fwd_bstride = nc * ea.fwd_fstride;
  }
  return col_inv(c, c->prec.fft_prec, EPI_CORR, spec_grad, nc, ea);
}

template <typename T>
cudaError_t dft_lines_t(int n, int nlines, int dir, const void* in, void* out, cudaStream_t st, const FftPlan& plan,
                        const void* pool) {
  typedef typename CT<T>::t V;
  const int ls = plan.line_len();
  const size_t per = 2 * (size_t)ls * sizeof(V);
  const int L = fit_units(per, kSmemBudget, 16);
  const size_t smem = per * L;
  const int blocks = (nlines + L - 1) / L;
  cudaError_t e = check_smem(smem);
  if (e != cudaSuccess) return e;
  if (dir < 0)
    k_dft_lines<T, false><<<blocks, kThreads, smem, st>>>(n, nlines, (const V*)in, (V*)out, plan, (const V*)pool, L, ls);
  else
    k_dft_lines<T, true><<<blocks, kThreads, smem, st>>>(n, nlines, (const V*)in, (V*)out, plan, (const V*)pool, L, ls);
  return cudaGetLastError();
}

template <typename T, typename IO>
cudaError_t dft_ip_t(int n, int nlines, int dir, const void* in, void* out, cudaStream_t st, const FftPlan& plan,
                     IpPlan ip, const void* pool) {
  typedef typename CT<T>::t V;
  ip.sym = 1;
  const size_t per = 2 * (size_t)plan.line_len() * sizeof(V);
  const int L = fit_units(per, kSmemBudget, 16);
  cudaError_t e = check_smem(per * L);
  if (e != cudaSuccess) return e;
  const int ls = ip_ls<T>(ip);
  const size_t smem = (size_t)(L + ip.big) * ls * sizeof(V);
  k_dft_ip<T, IO><<<(nlines + L - 1) / L, 128, smem, st>>>(n, nlines, (const IO*)in, (IO*)out, ip, (const V*)pool, L, ls,
                                                           dir > 0);
  return cudaGetLastError();
}

size_t dft_lines_smem(int prec, const FftPlan& plan) {
  const size_t cb = prec == FCSPH_F32 ? sizeof(CT<float>::t) : prec == FCSPH_F32X2 ? sizeof(CT<ff>::t)
                                                                                 : sizeof(CT<double>::t);
  const size_t per = 2 * (size_t)plan.line_len() * cb;
  return per * fit_units(per, kSmemBudget, 16);
}

size_t dft_smem_max() { return kSmemMax; }

cudaError_t launch_dft_lines(int n, int nlines, int dir, int prec, const void* in, void* out, cudaStream_t st,
                             const FftPlan& plan, const void* pool) {
  if (prec == FCSPH_F64) return dft_lines_t<double>(n, nlines, dir, in, out, st, plan, pool);
  return dft_lines_t<float>(n, nlines, dir, in, out, st, plan, pool);
}

cudaError_t launch_dft_ip(int n, int nlines, int dir, int prec, const void* in, void* out, cudaStream_t st,
                          const FftPlan& plan, const IpPlan& ip, const void* pool) {
  if (prec == FCSPH_F64) return dft_ip_t<double, double2>(n, nlines, dir, in, out, st, plan, ip, pool);
  if (prec == FCSPH_F32X2) return dft_ip_t<ff, double2>(n, nlines, dir, in, out, st, plan, ip, pool);
  return dft_ip_t<float, float2>(n, nlines, dir, in, out, st, plan, ip, pool);
}

cudaError_t launch_resid_norm(fcsph_ctx* c, const double* r, const double* b, double* out2) {
  cudaMemsetAsync(out2, 0, 2 * sizeof(double), c->stream);
  ProfScope ps(c, FCSPH_PROF_OTHER);
  k_resid_inst<<<c->gd.batch, kThreads, 0, c->stream>>>(r, b, (size_t)c->gd.ncol * c->gd.ny, out2);
  c->launches++;
  return cudaGetLastError();
}

cudaError_t launch_remove_mean(fcsph_ctx* c, const double* b, double* out) {
  const GridDev& g = c->gd;
  const double wx = g.x_walls ? g.nx - 1 : g.nx, wy = g.ny - 1;  // sums of the weights
  ProfScope ps(c, FCSPH_PROF_OTHER);
  k_mean_part<<<dim3(kMeanParts, g.batch), kThreads, 0, c->stream>>>(g, b, c->dred + 8);
  k_sub_mean<<<dim3((unsigned)std::min<size_t>(152, ((size_t)g.ncol * g.ny + kThreads - 1) / kThreads), g.batch), kThreads, 0,
               c->stream>>>(g, b, c->dred + 8, 1.0 / (wx * g.nz * wy), out);
  c->launches += 2;
  return cudaGetLastError();
}
size_t mean_scratch(const fcsph_ctx* c) { return (size_t)c->gd.batch * kMeanParts; }

cudaError_t launch_widen(fcsph_ctx* c, double* y, const float* x, size_t n) {
  ProfScope ps(c, FCSPH_PROF_OTHER);
  k_widen<<<152 * 4, kThreads, 0, c->stream>>>(y, x, n);
  c->launches++;
  return cudaGetLastError();
}

cudaError_t launch_narrow(fcsph_ctx* c, float* y, const double* x, int n) {
  ProfScope ps(c, FCSPH_PROF_OTHER);
  k_narrow<<<152 * 4, kThreads, 0, c->stream>>>(y, x, (size_t)n);
  c->launches++;
  return cudaGetLastError();
}

// ===========================================================================
// Persistent multi-class step (see k_persist)

struct PersistPlan {
  int prec = FCSPH_F32X2;
  std::vector<PersistRec*> recs;     // one recording per class
  std::vector<int> inst;             // instances per class
  PassDesc* d_descs = nullptr;
  WorkItem* d_items = nullptr;
  unsigned* d_counters = nullptr;    // counters, then the item dispenser
  int* d_status = nullptr;
  int n_items = 0, n_counters = 0, grid = 0, threads = 32, rmax = 0;
  size_t smem = 0;
  cudaGraphExec_t gexec = nullptr;
  long long graph_wait_ns = -1;
};

PersistPlan* persist_create(int prec) {
  PersistPlan* p = new PersistPlan();
  p->prec = prec;
  return p;
}

void persist_destroy(PersistPlan* p) {
  if (!p) return;
  for (PersistRec* r : p->recs) delete r;
  if (p->gexec) cudaGraphExecDestroy(p->gexec);
  cudaFree(p->d_descs);
  cudaFree(p->d_items);
  cudaFree(p->d_counters);
  cudaFree(p->d_status);
  delete p;
}

PersistRec* persist_add_class(PersistPlan* p, int instances) {
  PersistRec* r = new PersistRec();
  p->recs.push_back(r);
  p->inst.push_back(instances);
  return r;
}

// Tiles of descriptor d per instance, and the instance count of its grid.
static int desc_fields(const PassDesc& d) { return d.kind == PK_COL_FWD ? d.gy : (d.kind == PK_ROW_SYM ? d.gz : 1); }
static int desc_tiles(const PassDesc& d) { return d.gx * desc_fields(d); }
static int desc_insts(const PassDesc& d) { return d.kind == PK_COL_FWD ? d.gz : d.gy; }

cudaError_t persist_finalize(PersistPlan* p, cudaStream_t st, std::string* err) {
  std::vector<PassDesc> descs;
  std::vector<int> first(p->recs.size()), npass(p->recs.size()), cbase(p->recs.size());
  int maxp = 0, nc = 0;
  for (size_t c = 0; c < p->recs.size(); ++c) {
    first[c] = (int)descs.size();
    npass[c] = (int)p->recs[c]->descs.size();
    cbase[c] = nc;
    for (const PassDesc& d : p->recs[c]->descs) {
      if (desc_insts(d) != p->inst[c]) {
        *err = "persistent plan: a pass does not cover the class's instances";
        return cudaErrorInvalidValue;
      }
      descs.push_back(d);
      if (d.smem > p->smem) p->smem = d.smem;
      p->rmax = std::max(p->rmax, std::max(d.P.rmax, d.ea.fwd_nf > 0 ? d.ea.fwdP.rmax : 0));
    }
    nc += p->inst[c] * npass[c];
    if (npass[c] > maxp) maxp = npass[c];
  }
  // within a pass, the classes with the longest lines (most work per item)
  // come first, so that the short items of small classes fill the end of it
  std::vector<size_t> order(p->recs.size());
  for (size_t c = 0; c < order.size(); ++c) order[c] = c;
  auto weight = [&](size_t c) { return npass[c] ? descs[first[c]].g.my + descs[first[c]].g.mx : 0; };
  std::stable_sort(order.begin(), order.end(), [&](size_t a, size_t b2) { return weight(a) > weight(b2); });
  std::vector<WorkItem> items;
  size_t most = 0;  // items of the longest pass
  for (int ps = 0; ps < maxp; ++ps) {
    const size_t before = items.size();
    for (size_t c : order) {
      if (ps >= npass[c]) continue;
      const int di = first[c] + ps;
      const PassDesc& d = descs[di];
      const int prev_tiles = ps > 0 ? desc_tiles(descs[di - 1]) : 0;
      for (int b = 0; b < p->inst[c]; ++b) {
        const int self = cbase[c] + b * npass[c] + ps;
        const int ny = desc_fields(d);
        for (int by = 0; by < ny; ++by)
          for (int bx = 0; bx < d.gx; ++bx) {
            WorkItem it;
            it.desc = di;
            it.bx = bx;
            it.by = by;
            it.b = b;
            it.dep = ps > 0 ? self - 1 : -1;
            it.need = prev_tiles;
            it.self = self;
            items.push_back(it);
          }
      }
    }
    most = std::max(most, items.size() - before);
  }
  if (items.empty() || p->smem + 64 > kSmemMax) {  // 64: the kernel's own static shared words
    *err = items.empty() ? "persistent plan: nothing to run" : "persistent plan: a pass exceeds shared memory";
    return cudaErrorInvalidValue;
  }
  p->n_items = (int)items.size();
  p->n_counters = nc;
  cudaError_t e;
  if ((e = cudaMalloc(&p->d_descs, descs.size() * sizeof(PassDesc))) != cudaSuccess ||
      (e = cudaMalloc(&p->d_items, items.size() * sizeof(WorkItem))) != cudaSuccess ||
      (e = cudaMalloc(&p->d_counters, (size_t)(nc + 1) * sizeof(unsigned))) != cudaSuccess ||
      (e = cudaMalloc(&p->d_status, sizeof(int))) != cudaSuccess) {
    *err = "persistent plan: device memory";
    return e;
  }
  // on the launching stream, and landed before the host lists go
  e = cudaMemcpyAsync(p->d_descs, descs.data(), descs.size() * sizeof(PassDesc), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(p->d_items, items.data(), items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(p->d_status, 0, sizeof(int), st);
  const cudaError_t es = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = es;
  if (e != cudaSuccess) {
    *err = "persistent plan: upload";
    return e;
  }
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  // CTA width: the one with the most resident warps per SM (the narrowest on
  // a tie): one warp per CTA unless shared memory (the largest pass of any
  // class) caps the CTAs an SM holds; wider while the CTAs outnumber the items of
  // the longest pass, whose warps would otherwise idle (8 channels of 150^2, at
  // most 1408 items for 1824 one-warp CTAs: FP64 step 3355 -> 2181 us, pairs 1779 -> 1139)
  int best_warps = 0;
  for (int nt : {32, 64, 128}) {
    int occ = 0;
    e = with_persist_rm(p->rmax, [&](auto w) {
      constexpr int RM = decltype(w)::value;
      return p->prec == FCSPH_F64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_persist<double, RM>, nt, p->smem)
                                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_persist<ff, RM>, nt, p->smem);
    });
    if (e != cudaSuccess) return e;
    if (occ * nt / 32 > best_warps || (occ > 0 && (size_t)p->grid > most)) {
      best_warps = occ * nt / 32;
      p->threads = nt;
      p->grid = sms * occ;
    }
  }
  if (best_warps == 0) {
    *err = "persistent plan: no CTA fits an SM";
    return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

static cudaError_t persist_enqueue(PersistPlan* p, cudaStream_t st, long long wait_ns, int stall) {
  cudaError_t e = cudaMemsetAsync(p->d_counters, 0, (size_t)(p->n_counters + 1) * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  unsigned* next = p->d_counters + p->n_counters;
  return with_persist_rm(p->rmax, [&](auto w) {
    constexpr int RM = decltype(w)::value;
    if (p->prec == FCSPH_F64)
      k_persist<double, RM><<<p->grid, p->threads, p->smem, st>>>(p->d_descs, p->d_items, p->n_items, p->d_counters, next,
                                                          p->d_status, wait_ns, stall);
    else
      k_persist<ff, RM><<<p->grid, p->threads, p->smem, st>>>(p->d_descs, p->d_items, p->n_items, p->d_counters, next,
                                                      p->d_status, wait_ns, stall);
    return cudaGetLastError();
  });
}

// One persistent launch (counter reset + kernel).  Without a stall it replays
// a CUDA graph of the two, captured on first use.
cudaError_t persist_launch(PersistPlan* p, cudaStream_t st, cudaStream_t cap, long long wait_ns, int stall) {
  if (stall >= 0) return persist_enqueue(p, st, wait_ns, stall);
  if (!p->gexec || p->graph_wait_ns != wait_ns) {
    if (p->gexec) {
      cudaGraphExecDestroy(p->gexec);
      p->gexec = nullptr;
    }
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeRelaxed);
    if (e != cudaSuccess) return e;
    cudaError_t le = persist_enqueue(p, cap, wait_ns, -1);
    cudaGraph_t g = nullptr;
    e = cudaStreamEndCapture(cap, &g);
    if (le != cudaSuccess || e != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      return le != cudaSuccess ? le : e;
    }
    e = cudaGraphInstantiate(&p->gexec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return e;
    p->graph_wait_ns = wait_ns;
  }
  return cudaGraphLaunch(p->gexec, st);
}

// Reads and clears the plan's status word (synchronises st).
cudaError_t persist_status(PersistPlan* p, cudaStream_t st, int* status) {
  *status = 0;
  cudaError_t e = cudaMemcpyAsync(status, p->d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess && *status) e = cudaMemsetAsync(p->d_status, 0, sizeof(int), st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

long long persist_items(const PersistPlan* p) { return p ? p->n_items : 0; }
