// fft_line.cuh -- line-private transforms of the FP32 passes: T = L/EPT threads
// transform one line (V = float) or two lines at once (V = F2: packed FP32
// arithmetic, one twiddle load, one exchange and one barrier for both) through
// ONE exchange buffer of L elements.  The arithmetic of a line is that of
// block_fft_fwd / block_fft_inv (fft_core.cuh) term by term.
//
// Why pairs: the passes are bound by the L1 / shared-memory data pipe (2048^2 TE:
// 68 % of its cycles in the x forward pass, 65 % in the fused pass, DRAM at 20 %),
// and 43 % of its traffic was 16-byte twiddles.  Two lines per thread halve that
// and the instructions (packed adds and FMAs).
//
// Synchronisation spans the line's own threads only: a warp barrier where they
// lie in one warp (T <= 32, a power of two), else the named barrier `bar`.
#pragma once

#include <type_traits>

#include "fft_core.cuh"

namespace psatd {

// SUB: several lines of a warp may run apart (FP64, whose groups need not be whole
// warps): only the line's own lanes meet.  The block's x dimension is T, so that a line's
// lanes are an aligned run of T.
template <int T, bool SUB = false>
__device__ __forceinline__ void line_sync(int bar) {
  static_assert((T & (T - 1)) == 0, "a line's threads must not straddle warps");
  if constexpr (T > 32) {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(T) : "memory");
  } else if constexpr (SUB && T < 32) {
    unsigned lane;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    __syncwarp(((1u << T) - 1u) << (lane & ~(unsigned)(T - 1)));
  } else {
    __syncwarp();
  }
}

// Position of element i in the exchange buffer that stage S writes.  8-byte
// elements: sw<> (fft_core.cuh).  16-byte elements (pairs; a warp's access runs
// in phases of 8 lanes over 8 bank groups): i ^ (i >> 3) in the low three bits,
// >> 4 for the radix-16 stages of span < 8, none for a radix-3 or -6 first stage; gx, a
// multiple of the line's number where 8 lanes hold several lines (T < 8).  Of the
// shifts 3..7 and multipliers 0..7 these measured the fewest wavefronts (one per
// phase for all power-of-two lengths of 8 or more threads).
template <class P, int S, int ES>
struct ExPos {
  static constexpr bool kOdd = P::kMixed && S == 0 && (P::kR0 == 3 || P::kR0 == 6);
  static constexpr int kShift = (P::kEPT == 16 && P::radix(S) == 16 && P::span(S) < 8) ? 4 : 3;
  static __device__ __forceinline__ int at(int i, int gx) {
    if constexpr (ES == 8) return sw<P::swz(S)>(i);
    else if constexpr (kOdd) return i ^ gx;
    else return i ^ ((i >> kShift) & 7) ^ gx;
  }
  // at(i | off) from p = at(i): the swizzle is linear over XOR, so for disjoint bits
  // only the constant at(off) enters; a plain offset where it leaves the low bits alone
  static __device__ __forceinline__ int add(int p, int i, int off, int gx) {
    if constexpr (P::kMixed) return at(i + off, gx);
    const int c = at(off, 0);
    return (off & 255) == 0 ? p + off : p ^ c;
  }
};
// gx of line g of a block (see ExPos)
template <class P>
__device__ __forceinline__ int line_gx(int g) {
  return P::kT == 2 ? (2 * g) & 7 : P::kT == 4 ? ((P::kMixed ? 4 : 2) * g) & 7 : 0;
}

// Opaque copy of the twiddle pointer: keeps a stage's twiddle loads in that stage
// (the compiler would otherwise hoist every stage's into registers).
template <class W>
__device__ __forceinline__ const W* stage_ptr(const W* p) {
  asm volatile("" : "+l"(p));
  return p;
}

template <int L, int EPT, int S, class W>
__device__ __forceinline__ void line_load_tw(W (&w)[PFCount<L, EPT>::value], const W* __restrict__ tw, int t) {
  typedef FFTPlan<L, EPT> P;
  if constexpr (S >= 1 && S < P::kStages) {
    constexpr int RS = P::radix(S), NS = P::span(S), Q = EPT / RS, T = P::kT;
    const W* base = stage_ptr(tw) + P::tw_off(S);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = t + q * T;
      const int k = is_pow2(NS) ? (j & (NS - 1)) : (int)((unsigned)j % (unsigned)NS);
#pragma unroll
      for (int r = 1; r < RS; ++r) w[q * (RS - 1) + r - 1] = __ldg(&base[(r - 1) * NS + k]);
    }
  }
}

// Forward stage S.  PF: the next stage's twiddles are loaded before this stage's
// exchange barrier (in registers to spare); else each stage loads its own.
template <class V, int L, int EPT, bool PF, int S>
__device__ __forceinline__ void line_fwd_stage(typename Types<V>::C (&v)[EPT], typename Types<V>::C* buf,
                                               const typename Types<V>::W* __restrict__ tw, int t, int gx, int bar,
                                               typename Types<V>::W (&w)[PFCount<L, EPT>::value]) {
  typedef typename Types<V>::C C;
  typedef FFTPlan<L, EPT> P;
  typedef ExPos<P, S, (int)sizeof(C)> X;
  constexpr int RS = P::radix(S), NS = P::span(S), Q = EPT / RS, T = P::kT;
  constexpr bool LAST = (S == P::kStages - 1);
  if constexpr (!LAST) line_sync<T, std::is_same<V, double>::value>(bar);  // the buffer's earlier reads are done
  if constexpr (!PF) line_load_tw<L, EPT, S>(w, tw, t);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = t + q * T;
    const int k = is_pow2(NS) ? (j & (NS - 1)) : (int)((unsigned)j % (unsigned)NS);
    C a[RS];
#pragma unroll
    for (int r = 0; r < RS; ++r) a[r] = v[q + r * Q];
    if constexpr (NS > 1) {
#pragma unroll
      for (int r = 1; r < RS; ++r) a[r] = twmul(a[r], w[q * (RS - 1) + r - 1]);
    }
    butterfly<RS, false>(a);
    if constexpr (LAST) {
#pragma unroll
      for (int r = 0; r < RS; ++r) v[q + r * Q] = a[r];
    } else {
      const int base = (j - k) * RS + k;
      const int pb = X::at(base, gx);
#pragma unroll
      for (int r = 0; r < RS; ++r) buf[X::add(pb, base, r * NS, gx)] = a[r];
    }
  }
  if constexpr (!LAST) {
    if constexpr (PF) line_load_tw<L, EPT, S + 1>(w, tw, t);
    line_sync<T, std::is_same<V, double>::value>(bar);
    const int pt = X::at(t, gx);
#pragma unroll
    for (int m = 0; m < EPT; ++m) v[m] = buf[X::add(pt, t, T * m, gx)];
  }
}

// Adjoint of line_fwd_stage (the stage's twiddles are applied after its butterfly).
// OWN: the buffer's elements at the thread's own positions are the only ones any
// thread touched since (the first exchange of an inverse).
template <class V, int L, int EPT, bool PF, int S>
__device__ __forceinline__ void line_inv_stage(typename Types<V>::C (&v)[EPT], typename Types<V>::C* buf,
                                               const typename Types<V>::W* __restrict__ tw, int t, int gx, int bar,
                                               typename Types<V>::W (&w)[PFCount<L, EPT>::value]) {
  typedef typename Types<V>::C C;
  typedef FFTPlan<L, EPT> P;
  typedef ExPos<P, S, (int)sizeof(C)> X;
  constexpr int RS = P::radix(S), NS = P::span(S), Q = EPT / RS, T = P::kT;
  constexpr bool FIRST = (S == P::kStages - 1);
  if constexpr (!FIRST) {
    if constexpr (S < P::kStages - 2) line_sync<T, std::is_same<V, double>::value>(bar);  // the previous exchange's reads are done
    const int pt = X::at(t, gx);
#pragma unroll
    for (int m = 0; m < EPT; ++m) buf[X::add(pt, t, T * m, gx)] = v[m];
  }
  if constexpr (PF) line_load_tw<L, EPT, S>(w, tw, t);
  if constexpr (!FIRST) line_sync<T, std::is_same<V, double>::value>(bar);
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int j = t + q * T;
    const int k = is_pow2(NS) ? (j & (NS - 1)) : (int)((unsigned)j % (unsigned)NS);
    C a[RS];
    if constexpr (FIRST) {
#pragma unroll
      for (int r = 0; r < RS; ++r) a[r] = v[q + r * Q];
    } else {
      const int base = (j - k) * RS + k;
      const int pb = X::at(base, gx);
#pragma unroll
      for (int r = 0; r < RS; ++r) a[r] = buf[X::add(pb, base, r * NS, gx)];
    }
    butterfly<RS, true>(a);
#pragma unroll
    for (int r = 0; r < RS; ++r) v[q + r * Q] = a[r];
  }
  if constexpr (NS > 1) {
    if constexpr (!PF) line_load_tw<L, EPT, S>(w, tw, t);
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int r = 1; r < RS; ++r) v[q + r * Q] = twmul_conj(v[q + r * Q], w[q * (RS - 1) + r - 1]);
  }
}

template <class V, int L, int EPT, bool PF, int... S>
__device__ __forceinline__ void line_fwd_seq(typename Types<V>::C (&v)[EPT], typename Types<V>::C* buf,
                                             const typename Types<V>::W* __restrict__ tw, int t, int gx, int bar,
                                             std::integer_sequence<int, S...>) {
  typename Types<V>::W w[PFCount<L, EPT>::value];
  if constexpr (PF) line_load_tw<L, EPT, 1>(w, tw, t);
  (line_fwd_stage<V, L, EPT, PF, S>(v, buf, tw, t, gx, bar, w), ...);
}
template <class V, int L, int EPT, bool PF, int... S>
__device__ __forceinline__ void line_inv_seq(typename Types<V>::C (&v)[EPT], typename Types<V>::C* buf,
                                             const typename Types<V>::W* __restrict__ tw, int t, int gx, int bar,
                                             std::integer_sequence<int, S...>) {
  typename Types<V>::W w[PFCount<L, EPT>::value];
  (line_inv_stage<V, L, EPT, PF, FFTPlan<L, EPT>::kStages - 1 - S>(v, buf, tw, t, gx, bar, w), ...);
}

// Forward DFT of the line(s) in v (x[t + T m] -> X[t + T m]); the buffer may still
// be read by other threads of the line on entry, and is on exit.
template <class V, int L, int EPT, bool PF>
__device__ __forceinline__ void line_fft_fwd(typename Types<V>::C (&v)[EPT], typename Types<V>::C* buf,
                                             const typename Types<V>::W* __restrict__ tw, int t, int gx, int bar) {
  line_fwd_seq<V, L, EPT, PF>(v, buf, tw, t, gx, bar, std::make_integer_sequence<int, FFTPlan<L, EPT>::kStages>{});
}
// Unnormalised inverse (adjoint).  On entry no other thread may still touch this
// thread's own positions ExPos<P, kStages - 2>::at(t + T m).
template <class V, int L, int EPT, bool PF>
__device__ __forceinline__ void line_fft_inv(typename Types<V>::C (&v)[EPT], typename Types<V>::C* buf,
                                             const typename Types<V>::W* __restrict__ tw, int t, int gx, int bar) {
  line_inv_seq<V, L, EPT, PF>(v, buf, tw, t, gx, bar, std::make_integer_sequence<int, FFTPlan<L, EPT>::kStages>{});
}

// Own position of element t + T m between a forward and an inverse transform.
template <int L, int EPT, int ES>
__device__ __forceinline__ int own_pos(int t, int m, int gx) {
  typedef FFTPlan<L, EPT> P;
  constexpr int S = P::kStages >= 2 ? P::kStages - 2 : 0;
  typedef ExPos<P, S, ES> X;
  if constexpr (P::kStages < 2) return t + P::kT * m;
  else return X::add(X::at(t, gx), t, P::kT * m, gx);
}

}  // namespace psatd
