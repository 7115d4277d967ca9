// In-place shared-memory FFT of the method's passes (one CTA, several lines,
// one buffer per line).
//
// A stage with radix R combines the R values of a butterfly and writes its R
// outputs back to the places they came from, so a line needs no second buffer
// (half the shared memory of a ping-pong transform: twice the lines per warp
// at the same residency, whose butterflies then fill the lanes: a 280-point
// line has 35, 56 and 40 butterflies a stage for 32 lanes).  The arithmetic is
// the Stockham recurrence of fcsph_fft.cuh, butterfly by butterfly; only the
// places differ.  With n = R_1 ... R_S, N_s = R_1 ... R_{s-1}, M_s = n /
// (R_1 ... R_s) and the digits i = sum_s d_s M_s of an input, k = sum_s q_s
// N_s of an output, stage s turns digit d_s into q_s in place.  Two layouts:
//   D: input i at address i, output k at address sum q_s M_s (digit-reversed);
//      stage s: R values M_s apart;
//   T: input i at address sum d_s N_s, output k at address k; stage s: R
//      values N_s apart.
// A direct plan runs D.  Rader (prime n, n - 1 factors directly) and Bluestein
// run T, multiply by the transformed kernel as the last T stage stores its
// outputs (which are then in natural order), and D.  Index tables (in_tab,
// out_tab) say where the producers of a line put element k and where its
// consumers find output k, so that no pass moves data only to reorder it.
// Every transform is a forward one: for the inverse, IDFT(x) = conj(DFT(conj
// x)), the producers store conjugates and the consumers conjugate what they
// load.
//
// Addresses are swizzled within blocks of 128 bytes (XOR of the element's
// place in its block with the block's number): the butterflies of neighbouring
// lanes, whose addresses lie R or M_s R apart, then fall on different banks
// for every radix, power-of-two strides included.
//
// What it gave, together with the packed FP32-pair arithmetic of fcsph_ff.cuh
// and several outputs per transform (fit_group in fcsph_kernels.cu), results
// bitwise unchanged: RK3 step of 32 cavities of 256^2 in FP32 pairs (Rader
// lines of 281) 9.21 -> 6.69 ms, 8 slots of 512^2 (lines of 540) 8.61 -> 6.52
// ms, two 64^3 channels 4.88 -> 2.87 ms, the pressure solve of 32 boxes of
// 256^2 579 -> 473 us, ten steps of one 64^2 channel in FP64 5.47 -> 2.84 ms.
// On its own, with the lines staying in shared memory, a 281-point transform
// of FP32 pairs takes 2150 SM cycles at 8 lines per 128 threads (1450 of them
// FP32 pipe: 63 % busy), one of 280 points 935.
#pragma once

#include <cuda_runtime.h>

#include "fcsph_fft.cuh"

namespace fcsph {

// log2 of the elements in 128 bytes
template <typename T> struct SwBits { static constexpr int v = sizeof(typename CT<T>::t) == 16 ? 3 : 4; };
template <typename T> __host__ __device__ __forceinline__ int swz(int a) {
  return a ^ ((a >> SwBits<T>::v) & ((1 << SwBits<T>::v) - 1));
}
// Elements a line occupies: whole 128-byte blocks.
template <typename T> inline int ip_ls(const IpPlan& P) {
  const int b = 1 << SwBits<T>::v;
  return (P.slots + b - 1) / b * b;
}

// Slots of a line's input element k and output element k.
template <typename T> __device__ __forceinline__ int in_slot(const IpPlan& P, int k) {
  return swz<T>(P.in_tab < 0 ? k : __ldg(P.itab + P.in_tab + k));
}
template <typename T> __device__ __forceinline__ int out_slot(const IpPlan& P, int k) {
  return swz<T>(P.out_tab < 0 ? k : __ldg(P.itab + P.out_tab + k));
}

// What the last stage of a pass does with its outputs y_k: IP_MUL stores
// conj(y_k bhat_k) and keeps y_0 (Rader: the sum of the inputs) in slot m + 1;
// IP_X0 (Rader's second pass) stores x_0 + conj(y), x_0 from slot m, and
// X_0 = x_0 + y_0 in slot m + 1.
enum { IP_PLAIN = 0, IP_MUL = 1, IP_X0 = 2 };

template <typename T, int R>
__device__ __forceinline__ void ip_stage(typename CT<T>::t* lines, int nl, int ls, const IpStage S, int type_t,
                                         bool first, const typename CT<T>::t* __restrict__ tw,
                                         const int* __restrict__ itab, int mode, int keep, int m,
                                         const typename CT<T>::t* __restrict__ bh) {
  typedef typename CT<T>::t V;
  for (int t = threadIdx.x; t < nl * S.nb; t += blockDim.x) {
    const int line = fdiv(t, S.dnb);
    const int b = t - line * S.nb;
    const int q = fdiv(b, S.dstep);
    const int rem = b - q * S.step;
    const int base = q * S.step * R + rem;
    const int ks = first ? 0 : (type_t ? rem * S.ks : __ldg(itab + S.ks + q));
    V* L = lines + (size_t)line * ls;
    V v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = L[swz<T>(base + r * S.step)];
    if (ks > 0) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul_nr(v[r], tw[r * ks]);
    }
    dft_reg<T, R, false>(v);
    if (mode == IP_PLAIN) {
#pragma unroll
      for (int r = 0; r < R; ++r) L[swz<T>(base + r * S.step)] = cnorm(v[r]);
    } else if (mode == IP_MUL) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = cnorm(v[r]);
      if (keep && base == 0) L[swz<T>(m + 1)] = v[0];
#pragma unroll
      for (int r = 0; r < R; ++r) L[swz<T>(base + r * S.step)] = cconj(cmul(v[r], bh[base + r * S.step]));
    } else {
      const V x0 = L[swz<T>(m)];
      if (base == 0) L[swz<T>(m + 1)] = cadd(x0, L[swz<T>(m + 1)]);
#pragma unroll
      for (int r = 0; r < R; ++r) L[swz<T>(base + r * S.step)] = cadd(x0, cconj(cnorm(v[r])));
    }
  }
  __syncthreads();
}

// Wide stages (FP64, launches that leave SMs idle).  GB300 has half an FP64
// lane per scheduler: every FP64 warp instruction takes 64 cycles of its
// scheduler, however few lanes are active, so a stage costs as many of them as
// its longest thread executes (an 11-point butterfly 150, its twiddles 40 more:
// 6 us).  Here a thread computes one pair of outputs, q and R - q (odd R) or q
// and q + R/2 (R = 2, 4, 8), from all R inputs, with the operations the whole
// butterfly does for them (results unchanged): 44 for R = 11, 24 for R = 8.  The
// twiddles go first, one value per thread.  The extra work would only cost on
// an SM whose other CTAs need the FP64 units.  Ten steps of one 64^2 channel 2.49
// -> 2.03 ms, the line operator on its 32 column pairs 47 -> 39 us.
// Rounds of blockDim / tasks butterflies a wide stage may take.  Against 3, steps
// and operators of one to four fields of 24^2 to 200^2 take 0.7 % longer on average
// at 1 (line operator of 128^2 31.3 -> 35.6 us, of 100^2 23.2 -> 20.4) and 1.1 % at 8
// (step of 200^2 916 -> 1024).
constexpr int kWideRounds = 3;
template <int R> struct WideTasks { static constexpr int v = R % 2 ? (R + 1) / 2 : R / 2; };

// cosk<R>(j), sink<R>(j), j < R, for an exponent known only at run time.
template <int R> struct OddRoots {
  double c[R], s[R];
};
template <int R> constexpr OddRoots<R> make_odd_roots() {
  OddRoots<R> t{};
  for (int j = 0; j < R; ++j) {
    t.c[j] = cosk<R>(j);
    t.s[j] = sink<R>(j);
  }
  return t;
}
static __constant__ OddRoots<3> kOdd3 = make_odd_roots<3>();
static __constant__ OddRoots<5> kOdd5 = make_odd_roots<5>();
static __constant__ OddRoots<7> kOdd7 = make_odd_roots<7>();
static __constant__ OddRoots<11> kOdd11 = make_odd_roots<11>();
static __constant__ OddRoots<13> kOdd13 = make_odd_roots<13>();
static __constant__ OddRoots<17> kOdd17 = make_odd_roots<17>();
template <int R> __device__ __forceinline__ const OddRoots<R>& odd_roots() {
  if constexpr (R == 3) return kOdd3;
  else if constexpr (R == 5) return kOdd5;
  else if constexpr (R == 7) return kOdd7;
  else if constexpr (R == 11) return kOdd11;
  else if constexpr (R == 13) return kOdd13;
  else return kOdd17;
}

// Outputs q and its partner of the R-point DFT of v (q < WideTasks<R>::v); odd
// R, q = 0: only o0.
template <int R> __device__ __forceinline__ void wide_outputs(const double2* v, int q, double2& o0, double2& o1) {
  if constexpr (R % 2) {
    constexpr int h = (R - 1) / 2;
    double2 A[h], B[h];
#pragma unroll
    for (int r = 1; r <= h; ++r) {
      A[r - 1] = cadd_nr(v[r], v[R - r]);
      B[r - 1] = csub_nr(v[r], v[R - r]);
    }
    if (q == 0) {
      o0 = v[0];
#pragma unroll
      for (int r = 0; r < h; ++r) o0 = cadd_nr(o0, A[r]);
      o1 = o0;
    } else {
      const OddRoots<R>& w = odd_roots<R>();
      double2 re = cmadd_nr(v[0], A[0], w.c[q]);
      double2 im = cmul0_nr(B[0], w.s[q]);
      int e = q;
#pragma unroll
      for (int r = 2; r <= h; ++r) {
        e += q;
        if (e >= R) e -= R;
        re = cmadd_nr(re, A[r - 1], w.c[e]);
        im = cmadd_nr(im, B[r - 1], w.s[e]);
      }
      const double2 ri = rot<double2, false>(im);
      o0 = cadd_nr(re, ri);
      o1 = csub_nr(re, ri);
    }
  } else {
    auto flip = [](double2 a, bool neg) {  // -a or a, exactly
      const long long m = neg ? (long long)0x8000000000000000ull : 0;
      return make_double2(__longlong_as_double(__double_as_longlong(a.x) ^ m),
                          __longlong_as_double(__double_as_longlong(a.y) ^ m));
    };
    if constexpr (R == 2) {
      o0 = cadd_nr(v[0], v[1]);
      o1 = csub_nr(v[0], v[1]);
    } else {
      const bool odd = q & 1;
      // t0/t1 and t2/t3 of dft4 for the even (and, R = 8, the odd) inputs
      auto half = [&](double2 a0, double2 a1, double2 a2, double2 a3, double2& s, double2& d) {
        s = cadd_nr(a0, flip(a2, odd));
        d = cadd_nr(a1, flip(a3, odd));
        const double2 rd = rot<double2, false>(d);
        d = make_double2(odd ? rd.x : d.x, odd ? rd.y : d.y);
      };
      double2 s, d;
      if constexpr (R == 4) {
        half(v[0], v[1], v[2], v[3], s, d);
        o0 = cadd_nr(s, d);
        o1 = csub_nr(s, d);
      } else {
        half(v[0], v[2], v[4], v[6], s, d);
        const double2 e = cadd_nr(s, flip(d, q >= 2));
        half(v[1], v[3], v[5], v[7], s, d);
        double2 o = cadd_nr(s, flip(d, q >= 2));
        // q = 1, 3: e +/- h x with the products fused with the sums, as in dft_reg
        const double hh = 0.70710678118654752440;
        if (odd) {
          const double2 x = q == 1 ? make_double2(o.x + o.y, o.y - o.x) : make_double2(o.y - o.x, -(o.x + o.y));
          o0 = cmadd_nr(e, x, hh);
          o1 = cmadd_nr(e, x, -hh);
        } else {
          if (q == 2) o = rot<double2, false>(o);
          o0 = cadd_nr(e, o);
          o1 = csub_nr(e, o);
        }
      }
    }
  }
}

template <int R>
__device__ __forceinline__ void ip_stage_wide(double2* lines, int nl, int ls, const IpStage S, int type_t, bool first,
                                              const double2* __restrict__ tw, const int* __restrict__ itab, int mode,
                                              int keep, int m, const double2* __restrict__ bh, FastDiv dm) {
  constexpr int H = WideTasks<R>::v;
  if (!first) {
    for (int t = threadIdx.x; t < nl * m; t += blockDim.x) {
      const int line = fdiv(t, dm), a = t - line * m;
      const int x = fdiv(a, S.dstep), rem = a - x * S.step;  // a = (q R + r) step + rem
      const int q = x / R, r = x - q * R;
      const int e = r * (type_t ? rem * S.ks : __ldg(itab + S.ks + q));
      if (e > 0) {
        double2* p = lines + (size_t)line * ls + swz<double>(a);
        *p = cmul_nr(*p, tw[e]);
      }
    }
    __syncthreads();
  }
  // whole butterflies per round, so that one barrier between a round's loads
  // and stores is enough (a loop, not unrolled: these launches run every
  // instruction a few times, and fetching them is a large part of their time)
  const int nb = nl * S.nb, per = blockDim.x / H;
#pragma unroll 1
  for (int b0 = 0; b0 < nb; b0 += per) {
    const int cnt = min(per, nb - b0);
    const int q = threadIdx.x / cnt, bb = b0 + threadIdx.x - q * cnt;
    const int line = fdiv(bb, S.dnb), b = bb - line * S.nb;
    const int x = fdiv(b, S.dstep);
    const int base = x * S.step * R + (b - x * S.step);
    double2* L = lines + (size_t)line * ls;
    double2 o0, o1;
    if (q < H) {
      double2 v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = L[swz<double>(base + r * S.step)];
      wide_outputs<R>(v, q, o0, o1);
    }
    __syncthreads();
    if (q < H) {
      const double2 x0 = mode == IP_X0 ? L[swz<double>(m)] : o0;  // slot m exists in Rader lines only
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        if (w == 1 && R % 2 && q == 0) continue;
        const int a = base + (w == 0 ? q : (R % 2 ? R - q : q + H)) * S.step;
        double2 y = w ? o1 : o0;
        if (mode == IP_MUL) {
          if (keep && a == 0) L[swz<double>(m + 1)] = y;
          y = cconj(cmul(y, bh[a]));
        } else if (mode == IP_X0) {
          if (a == 0) L[swz<double>(m + 1)] = cadd(x0, L[swz<double>(m + 1)]);
          y = cadd(x0, cconj(y));
        }
        L[swz<double>(a)] = y;
      }
    }
  }
  __syncthreads();
}

// Large prime radix (19, 23, 29, 31): one thread per output, line by line
// through the scratch line (its R inputs must outlive every output).
template <typename T>
__device__ __forceinline__ void ip_stage_big(typename CT<T>::t* lines, int nl, int ls, const IpStage S, int type_t,
                                             bool first, const typename CT<T>::t* __restrict__ tw,
                                             const int* __restrict__ itab, int mode, int keep, int m,
                                             const typename CT<T>::t* __restrict__ bh, typename CT<T>::t* scratch) {
  typedef typename CT<T>::t V;
  const int R = S.R, n = S.nb * R;
  for (int line = 0; line < nl; ++line) {
    V* L = lines + (size_t)line * ls;
    for (int o = threadIdx.x; o < n; o += blockDim.x) {
      const int rr = o / S.nb, b = o - rr * S.nb;
      const int q = fdiv(b, S.dstep);
      const int rem = b - q * S.step;
      const int base = q * S.step * R + rem;
      const int ks = first ? 0 : (type_t ? rem * S.ks : __ldg(itab + S.ks + q));
      const int estep = (rr * S.nb + ks) % n;  // exponent increment per input
      V acc = L[swz<T>(base)];
      int e = 0;
      for (int r = 1; r < R; ++r) {
        e += estep;
        if (e >= n) e -= n;
        acc = cadd(acc, cmul(L[swz<T>(base + r * S.step)], tw[e]));
      }
      const int a = base + rr * S.step;
      if (mode == IP_MUL) {
        if (keep && a == 0) L[swz<T>(m + 1)] = acc;
        acc = cconj(cmul(acc, bh[a]));
      } else if (mode == IP_X0) {
        const V x0 = L[swz<T>(m)];
        if (a == 0) L[swz<T>(m + 1)] = cadd(x0, L[swz<T>(m + 1)]);
        acc = cadd(x0, cconj(acc));
      }
      scratch[swz<T>(a)] = acc;
    }
    __syncthreads();
    for (int a = threadIdx.x; a < n; a += blockDim.x) L[swz<T>(a)] = scratch[swz<T>(a)];
    __syncthreads();
  }
}

// The same radices in FP64 and FP32 pairs with the conjugate symmetry of the
// roots, as in dft_odd: the sums and differences of the inputs r and R - r in
// place, then a thread computes outputs q and R - q, 4 operations per pair of
// inputs where the in-order sum takes 24 for the two outputs.  W, DX, DY and LAP
// of 8 boxes of 161^2 in FP64 (extended length 186 = 31 3 2): 578 us with
// ip_stage_big, 244 so; projection of 12 channels of 200 x 127 in FP32 pairs (152
// = 19 8): 118 and 104.5; errors 1 to 3% smaller.  (Pairs renormalise every sum;
// without, their errors grew by 10%.)  The sums run in another order than
// ip_stage_big's, which the time step keeps: walled steps amplify a rounding
// difference by up to 1e7, and trajectories are to stay reproducible bit for
// bit.  FP32 keeps it as well: its Laplacians are rounding of the extended line.
template <typename T>
__device__ __forceinline__ void ip_stage_sym(typename CT<T>::t* lines, int nl, int ls, const IpStage S, int type_t,
                                             bool first, const typename CT<T>::t* __restrict__ tw,
                                             const int* __restrict__ itab, int mode, int keep, int m,
                                             const typename CT<T>::t* __restrict__ bh) {
  typedef typename CT<T>::t V;
  const int R = S.R, h = (R - 1) / 2, H = h + 1;
  const int nb = nl * S.nb, per = blockDim.x / H;  // whole butterflies per round: one barrier between loads and stores
  for (int t = threadIdx.x; t < nb * h; t += blockDim.x) {
    const int r1 = t / nb, bb = t - r1 * nb, r = r1 + 1;
    const int line = fdiv(bb, S.dnb), b = bb - line * S.nb;
    const int x = fdiv(b, S.dstep), rem = b - x * S.step;
    V* L = lines + (size_t)line * ls;
    const int base = x * S.step * R + rem, au = swz<T>(base + r * S.step), av = swz<T>(base + (R - r) * S.step);
    const int ks = first ? 0 : (type_t ? rem * S.ks : __ldg(itab + S.ks + x));
    V u = L[au], v = L[av];
    if (ks > 0) {
      u = cmul_nr(u, tw[r * ks]);
      v = cmul_nr(v, tw[(R - r) * ks]);
    }
    L[au] = cadd(u, v);
    L[av] = csub(u, v);
  }
  __syncthreads();
#pragma unroll 1
  for (int b0 = 0; b0 < nb; b0 += per) {
    const int cnt = min(per, nb - b0);
    const int q = threadIdx.x / cnt, bb = b0 + threadIdx.x - q * cnt;
    const int line = fdiv(bb, S.dnb), b = bb - line * S.nb;
    const int x = fdiv(b, S.dstep), rem = b - x * S.step;
    const int base = x * S.step * R + rem;
    V* L = lines + (size_t)line * ls;
    V re, im;
    if (q < H) {
      re = L[swz<T>(base)];
      im = mk<V>((T)0.0, (T)0.0);
      int e = 0;
      for (int r = 1; r <= h; ++r) {
        const V A = L[swz<T>(base + r * S.step)];
        if (q == 0) {
          re = cadd(re, A);
        } else {
          e += q;
          if (e >= R) e -= R;
          const V w = tw[e * S.nb];  // exp(-2 pi i e / R)
          re = cnorm(cmadd_nr(re, A, cre(w)));
          im = cnorm(cmadd_nr(im, L[swz<T>(base + (R - r) * S.step)], -cim(w)));
        }
      }
    }
    __syncthreads();
    if (q < H) {
      const V ri = rot<V, false>(im);
      const V x0 = mode == IP_X0 ? L[swz<T>(m)] : re;  // slot m exists in Rader lines only
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        if (w == 1 && q == 0) continue;
        const int a = base + (w ? R - q : q) * S.step;
        V y = q == 0 ? re : (w ? csub(re, ri) : cadd(re, ri));
        if (mode == IP_MUL) {
          if (keep && a == 0) L[swz<T>(m + 1)] = y;
          y = cconj(cmul(y, bh[a]));
        } else if (mode == IP_X0) {
          if (a == 0) L[swz<T>(m + 1)] = cadd(x0, L[swz<T>(m + 1)]);
          y = cadd(x0, cconj(y));
        }
        L[swz<T>(a)] = y;
      }
    }
  }
  __syncthreads();
}

template <typename T, int R>
__device__ __forceinline__ void ip_any(typename CT<T>::t* lines, int nl, int ls, const IpStage& S, int type_t, bool first,
                                       const typename CT<T>::t* __restrict__ tw, const int* __restrict__ itab, int mode,
                                       int keep, int m, const typename CT<T>::t* __restrict__ bh, int wide, FastDiv dm) {
  if constexpr (std::is_same<T, double>::value) {
    if (wide && nl * S.nb <= kWideRounds * ((int)blockDim.x / WideTasks<R>::v)) {
      ip_stage_wide<R>(lines, nl, ls, S, type_t, first, tw, itab, mode, keep, m, bh, dm);
      return;
    }
  }
  ip_stage<T, R>(lines, nl, ls, S, type_t, first, tw, itab, mode, keep, m, bh);
}

// Length-n DFT of nl lines in place (line stride ls >= ip_ls; element k of the
// input in slot in_slot(k), output k in slot out_slot(k)).  scratch: one more
// line, used by plans with a large prime radix only.  All threads of the CTA
// call it, after a barrier behind the producers; it ends with one.
template <typename T, int RM>
__device__ __noinline__ void fft_ip(typename CT<T>::t* lines, int nl, int ls, const IpPlan& P,
                                    const typename CT<T>::t* __restrict__ pool, typename CT<T>::t* scratch) {
  typedef typename CT<T>::t V;
  const int kind = P.kind, m = P.m, n = P.n;
  const int* itab = P.itab;
  const V* bh = pool + P.bhat;
  const int wide = P.wide;
  const FastDiv dm = P.dm;
  if (kind == IP_BLUESTEIN) {
    const V* ch = pool + P.chirp;
    for (int t = threadIdx.x; t < nl * m; t += blockDim.x) {
      const int line = fdiv(t, dm);
      const int j = t - line * m;
      V* x = lines + (size_t)line * ls + in_slot<T>(P, j);
      *x = j < n ? cmulc(*x, ch[j]) : mk<V>(0.0, 0.0);
    }
    __syncthreads();
  }
  const int passes = kind == IP_DIRECT ? 1 : 2;
#pragma unroll 1
  for (int pass = 0; pass < passes; ++pass) {
    const IpSub& U = pass == passes - 1 ? P.d : P.t;
    const int type_t = pass != passes - 1;
    const V* tw = pool + U.tw;
    const int nst = U.nst;
#pragma unroll 1
    for (int s = 0; s < nst; ++s) {
      const IpStage S = U.st[s];
      int mode = IP_PLAIN;
      if (s == nst - 1 && passes == 2) mode = type_t ? IP_MUL : (kind == IP_RADER ? IP_X0 : IP_PLAIN);
      const int keep = kind == IP_RADER;
      switch (S.R) {
        case 2: ip_any<T, 2>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm); break;
        case 3: ip_any<T, 3>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm); break;
        case 4: ip_any<T, 4>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm); break;
        case 5: ip_any<T, 5>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm); break;
        case 7: ip_any<T, 7>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm); break;
        case 8: ip_any<T, 8>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm); break;
        case 9: ip_stage<T, 9>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 11:
          if constexpr (RM >= 11) ip_any<T, 11>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm);
          break;
        case 13:
          if constexpr (RM >= 13) ip_any<T, 13>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm);
          break;
        case 17:
          if constexpr (RM >= 17) ip_any<T, 17>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, wide, dm);
          break;
        default:
          if constexpr (RM > 17) {
            if constexpr (!std::is_same<T, float>::value) {
              if (P.sym) {
                ip_stage_sym<T>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh);
                break;
              }
            }
            ip_stage_big<T>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, scratch);
          }
          break;
      }
    }
  }
  if (kind == IP_BLUESTEIN) {
    const V* ch = pool + P.chirp;
    const FastDiv dn = P.dn;
    for (int t = threadIdx.x; t < nl * n; t += blockDim.x) {
      const int line = fdiv(t, dn);
      const int j = t - line * n;
      V* x = lines + (size_t)line * ls + out_slot<T>(P, j);
      *x = cmulc(cconj(*x), ch[j]);
    }
    __syncthreads();
  }
}

}  // namespace fcsph
