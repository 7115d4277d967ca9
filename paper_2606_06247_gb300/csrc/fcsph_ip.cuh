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
  if (kind == IP_BLUESTEIN) {
    const V* ch = pool + P.chirp;
    const FastDiv dm = P.dm;
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
        case 2: ip_stage<T, 2>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 3: ip_stage<T, 3>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 4: ip_stage<T, 4>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 5: ip_stage<T, 5>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 7: ip_stage<T, 7>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 8: ip_stage<T, 8>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 9: ip_stage<T, 9>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh); break;
        case 11:
          if constexpr (RM >= 11) ip_stage<T, 11>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh);
          break;
        case 13:
          if constexpr (RM >= 13) ip_stage<T, 13>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh);
          break;
        case 17:
          if constexpr (RM >= 17) ip_stage<T, 17>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh);
          break;
        default:
          if constexpr (RM > 9) ip_stage_big<T>(lines, nl, ls, S, type_t, s == 0, tw, itab, mode, keep, m, bh, scratch);
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
