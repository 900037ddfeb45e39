// pair_push.cuh -- the fused last-axis pass without tensor cores: as k_line_push
// (psatd_kernels.cuh), in FP32 with the components of a line transformed two at a time
// in packed arithmetic (fft_line.cuh).  FP64 transforms them one at a time (every unit
// below is a single).
//
// Components in slot order form units: pairs (c, c + 1) and, where a group has an
// odd count, singles (pair_width).  A unit of a line owns one contiguous region of
// shared memory, w L values (w = its components): the bulk copies stage component
// c at its first half and c + 1 at its second, and the transforms exchange in
// place in that region (pairs as 16-byte elements), so the pass needs no exchange
// buffer beside the staged columns.  A line's threads synchronise only among
// themselves.  After its forward transform a unit holds the spectrum at each
// thread's own positions (own_pos), which the push and the inverse's first
// exchange alone touch.
//
// Bound: latency between the stages at 16 resident warps per SM (shared memory holds
// two CTAs of 2048-point lines), then the L1 / shared-memory data pipe (49 % busy).
// One component per thread -> pairs: 2048^2 TE 84.6 -> 73.7 us (113.5k -> 73.6k
// wavefronts per SM, 46.9 M -> 35.0 M instructions), 256^3 with eleven components 439 ->
// 371 us, 512 x 512 x 1024 9.47 -> 6.83 ms.  FP64 is bound by its units (half an operation
// per cycle and scheduler): 128^2, six components, 97 us with two lines to a one-warp
// CTA, 16 us with a line's two sets of components on SMs of their own, a group each
// component.
//
// The six 2D components are two independent sets, (Ex, Ey, Bz) and (Ez, Bx, By) with
// their sources: a CTA of that layout takes one of them (blockIdx.y) as the TE or TM
// pass over its slots (MAP), with half the shared memory and twice the CTAs (push_sets;
// FP32, 256^2 rho-form step 25.9 -> 19.3 us, 1024 x 512 47.4 -> 41.1).
//
// Component groups (GRP, G = blockDim.z): group j takes the units j, j + G, ...
// (inverse: from G - 1 - j); the block meets before and after the push, whose
// modes the groups split.
#pragma once

#include "fft_line.cuh"
#include "psatd_kernels.cuh"
#include "push_modes.h"

namespace psatd {

// Components of the unit that starts at slot c (slot order: psatd_kernels.cuh).
template <typename R, int LAYOUT>
__device__ __forceinline__ int pair_width(int c) {
  if constexpr (sizeof(R) == 8) return 1;
  else if constexpr (LAYOUT == 2) return c == 2 ? 1 : 2;               // (E0 E1) B2 (J0 J1) (rho rho')
  else if constexpr (LAYOUT == 3) return c == 0 ? 2 : 1;          // (E2 B0) B1 J2
  else return c == 8 ? 1 : 2;                                     // (E0 E1) (E2 B0) (B1 B2) (J0 J1) J2 (rho rho')
}
template <typename R, int LAYOUT>
__host__ __device__ constexpr bool pair_start(int c) {
  return sizeof(R) == 8 ? false : LAYOUT == 2 ? (c == 0 || c == 3 || c == 5) : LAYOUT == 3 ? c == 0 : (c == 0 || c == 2 || c == 4 || c == 6 || c == 9);
}

// The update of one mode whose slot values sit at p2 (pairs) and p1 (singles)
// within the units of this line; us: stride of one component over the block's
// lines, g1 / g2: this line's offset in a single's / pair's unit (bytes).
template <typename R, int LAYOUT, bool PSTD>
__device__ __forceinline__ void push_units(unsigned char* base, int us, int g1, int g2, int p1, int p2,
                                           const CoefReg<R>& f, R mx, R my, R mz,
                                           const PushArgs<R>& a, const typename Types<R>::W* P) {
  typedef typename Types<R>::C C;
  const C Z = mkc(R(0), R(0));
  const int form = a.form;
  const int zmask = a.ndim == 3 ? 7 : 3;
  constexpr int NF = LAYOUT >= 2 ? 3 : 6, NJ = LAYOUT == 2 ? 2 : LAYOUT == 3 ? 1 : 3;
  C s[kMaxComp];
  auto turn = [&](int c, C v, bool back) {  // staggered plans: to the true position and back
    if (P) {
      const int m = slot_stagger<LAYOUT>(c) & zmask;
#pragma unroll
      for (int ax = 0; ax < 3; ++ax)
        if (m & (1 << ax)) v = back ? twmul_conj(v, P[ax]) : twmul(v, P[ax]);
    }
    return v;
  };
#pragma unroll
  for (int c = 0; c < kMaxComp; ++c) {
    if (c >= NF + NJ + (LAYOUT == 3 ? 0 : 2)) break;
    const bool on = c < NF || (c < NF + NJ ? form >= 1 : form == 2);
    if (pair_start<R, LAYOUT>(c)) {
      float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
      if (on) q = *reinterpret_cast<const float4*>(base + c * us + g2 + p2 * 16);
      s[c] = on ? turn(c, mkc(R(q.x), R(q.z)), false) : Z;
      s[c + 1] = on ? turn(c + 1, mkc(R(q.y), R(q.w)), false) : Z;
    } else if (c == 0 || !pair_start<R, LAYOUT>(c - 1)) {
      s[c] = on ? turn(c, *reinterpret_cast<const C*>(base + c * us + g1 + p1 * (int)sizeof(C)), false) : Z;
    }
  }
  R cS_h, cS_l, Sc_h, Sc_l;
  prod2(a.c_h, a.c_l, f.S_h, f.S_l, cS_h, cS_l);
  prod2(a.ic_h, a.ic_l, f.S_h, f.S_l, Sc_h, Sc_l);
  if constexpr (PSTD) {  // J-form or vacuum
    C E[3] = {Z, Z, Z}, B[3] = {Z, Z, Z}, J[3] = {Z, Z, Z};
    if constexpr (LAYOUT == 2) {
      E[0] = s[0]; E[1] = s[1]; B[2] = s[2]; J[0] = s[3]; J[1] = s[4];
    } else if constexpr (LAYOUT == 3) {
      E[2] = s[0]; B[0] = s[1]; B[1] = s[2]; J[2] = s[3];
    } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) { E[i] = s[i]; B[i] = s[3 + i]; J[i] = s[6 + i]; }
    }
    pstd_modes<R>(E, B, J, mx, my, mz, a);
    if constexpr (LAYOUT == 2) {
      s[0] = E[0]; s[1] = E[1]; s[2] = B[2];
    } else if constexpr (LAYOUT == 3) {
      s[0] = E[2]; s[1] = B[0]; s[2] = B[1];
    } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) { s[i] = E[i]; s[3 + i] = B[i]; }
    }
  } else if constexpr (LAYOUT == 2) {
    push_te<R>(s[0], s[1], s[2], s[3], s[4], s[5], s[6], mx, my, f, cS_h, cS_l, Sc_h, Sc_l, a, form);
  } else if constexpr (LAYOUT == 3) {
    push_tm<R>(s[0], s[1], s[2], s[3], mx, my, f, cS_h, cS_l, Sc_h, Sc_l, a, form);
  } else if constexpr (LAYOUT == 1) {
    static_assert(sizeof(R) == 8, "FP32 runs the six 2D components as the TE and TM sets");
    push_te<R>(s[0], s[1], s[5], s[6], s[7], s[9], s[10], mx, my, f, cS_h, cS_l, Sc_h, Sc_l, a, form);
    push_tm<R>(s[2], s[3], s[4], s[8], mx, my, f, cS_h, cS_l, Sc_h, Sc_l, a, form);
  } else {
    C E[3] = {s[0], s[1], s[2]}, B[3] = {s[3], s[4], s[5]};
    const C J[3] = {s[6], s[7], s[8]};
    push_3d<R>(E, B, J, s[9], s[10], mx, my, mz, f, cS_h, cS_l, Sc_h, Sc_l, a, form);
#pragma unroll
    for (int i = 0; i < 3; ++i) { s[i] = E[i]; s[3 + i] = B[i]; }
  }
#pragma unroll
  for (int c = 0; c < NF; ++c) {
    if (pair_start<R, LAYOUT>(c)) {
      const C u = turn(c, s[c], true), w = turn(c + 1, s[c + 1], true);
      *reinterpret_cast<float4*>(base + c * us + g2 + p2 * 16) = make_float4((float)u.x, (float)w.x, (float)u.y, (float)w.y);
    } else if (c == 0 || !pair_start<R, LAYOUT>(c - 1)) {
      *reinterpret_cast<C*>(base + c * us + g1 + p1 * (int)sizeof(C)) = turn(c, s[c], true);
    }
  }
}

// The push of this thread's modes l = t + T (grp + G i), by push_mode_pairs.
template <typename R, int L, int LAYOUT, int EPT, bool STAG, bool PSTD>
__device__ __forceinline__ void push_line_units(unsigned char* base, int us, int g1, int g2, int gx,
                                                const PushArgs<R>& a, const Coef<R>* trow, int t, int grp,
                                                int G, int mxi, int myi, R kpx, R kpy, typename Types<R>::W phx,
                                                typename Types<R>::W phy) {
  typedef FFTPlan<L, EPT> P;
  constexpr int T = P::kT;
  auto coef = [&](int m) -> Coef<R> {
    if constexpr (!PSTD) return trow[coef_entry(t + T * m, L)];
    else return Coef<R>{};
  };
  push_mode_pairs<EPT>(grp, G, coef, [&](int m, const Coef<R>& q) {
    const int l = t + T * m;
    CoefReg<R> f;
    f.C_h = q.C_h; f.C_l = q.C_l; f.S_h = q.S_h; f.S_l = q.S_l;
    f.A1 = q.A1; f.A4 = q.A4; f.B1 = q.B1; f.B2 = q.B2;
    const int p1 = own_pos<L, EPT, 2 * (int)sizeof(R)>(t, m, sizeof(R) == 8 ? gx : 0);
    const int p2 = sizeof(R) == 8 ? 0 : own_pos<L, EPT, 16>(t, m, gx);
    R mx, my, mz;
    if constexpr (STAG) {
      const int ml = l < L / 2 ? l : l - L;
      R kl;
      typename Types<R>::W pl;
      stag_axis(a, a.ndim == 2 ? 1 : 2, ml, kl, pl);
      typename Types<R>::W Ph[3];
      Ph[0] = phx;
      if (a.ndim == 2) {
        mx = kpx; my = kl; mz = R(0);
        Ph[1] = pl;
        Ph[2] = phy;
      } else {
        mx = kpx; my = kpy; mz = kl;
        Ph[1] = phy;
        Ph[2] = pl;
      }
      push_units<R, LAYOUT, PSTD>(base, us, g1, g2, p1, p2, f, mx, my, mz, a, Ph);
    } else {
      const int ml = (l == L / 2) ? 0 : (l < L / 2 ? l : l - L);
      if (a.ndim == 2) {
        mx = a.rx * R(mxi); my = a.ry * R(ml); mz = R(0);
      } else {
        mx = a.rx * R(mxi); my = a.ry * R(myi); mz = a.rz * R(ml);
      }
      push_units<R, LAYOUT, PSTD>(base, us, g1, g2, p1, p2, f, mx, my, mz, a, nullptr);
    }
  });
}

// Slot of component c of the TE (MAP 1) or TM (MAP 2) set of the six-component layout
// (E0 E1 E2 B0 B1 B2 J0 J1 J2 rho rho'); MAP 0: the slot itself.
template <int MAP>
__device__ __forceinline__ int set_slot(int c) {
  return MAP == 1 ? (c < 2 ? c : c == 2 ? 5 : c < 5 ? c + 3 : c + 4) : MAP == 2 ? (c < 3 ? c + 2 : 8) : c;
}

// Body of one CTA: line block bx (tb lines; line g of the block handled by the
// threads (t, g, grp)); mbar / phase: the stage mbarrier and the parity of its
// next phase.  Returns false when a failed index check left the phase unused.
template <typename R, int L, int LAYOUT, int EPT, bool GRP, int MAP = 0>
__device__ __forceinline__ bool line_pair_body(const PushArgs<R>& a_in, const typename Types<R>::W* __restrict__ tw, int bx,
                                               int t, int g, int tb, int grp, int G, unsigned char* smem_raw,
                                               uint32_t mbar, uint32_t phase) {
  const PushArgs<R> a = a_in;  // a private copy: its scalars stay in registers
  const int n_in = MAP == 1 ? 3 + 2 * a.form : MAP == 2 ? 3 + (a.form >= 1 ? 1 : 0) : a.n_in;
  const int n_out = MAP ? 3 : a.n_out;
  typedef typename Types<R>::C C;
  typedef typename Types<R>::W W;
  typedef FFTPlan<L, EPT> P;
  constexpr int CS = (int)sizeof(C);
  constexpr int T = P::kT;
  // twiddles one stage ahead where a stage's fit beside two transforms' elements
  constexpr bool PF = EPT <= 12;
  if constexpr (!GRP) {
    grp = 0;
    G = 1;
  }
  const int tid = (grp * tb + g) * T + t, nthr = T * tb * G;
  const int line0 = bx * tb, line = line0 + g;
  const bool valid = line < a.nlines;
  if (a.tab_ext) {  // checked mode: the line's columns of every slot and its coefficient row
    int mx_c, my_c, row_c;
    line_modes(a, valid ? line : 0, mx_c, my_c, row_c);
    const bool bad = (valid && (int64_t)(line + 1) * L > a.cs) ||
                     (int64_t)(row_c + 1) * a.tab_row > a.tab_ext || row_c < 0;
    if (cta_out_of_bounds(bad, a.chk_err)) return false;
  }
  const int us = tb * L * CS;  // stride of one component over the block's lines
  const int g1 = g * L * CS, g2 = 2 * g1;
  const int gx = line_gx<P>(g), gx1 = CS == 16 ? gx : 0;  // pairs', singles'
  const int bar = 1 + g * G + grp;
  C* spec = static_cast<C*>(a.spec);
  // stage every input slot of the block's lines: one bulk copy per line and slot,
  // issued by the first warp, completing on the stage mbarrier; lines past the
  // last are zero-filled
  const int nv = a.nlines - line0 < tb ? a.nlines - line0 : tb;  // valid lines of the block
  if (!valid)
    for (int c = 0, w; c < n_in; c += w) {
      w = pair_width<R, LAYOUT>(c);
      float4* dst = reinterpret_cast<float4*>(smem_raw + c * us + w * g1);
      for (int i = t + grp * T; i < w * L * CS / 16; i += G * T) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  __syncthreads();  // the mbarrier is initialised; the zeros are visible
  if (tid < 32) {
    constexpr uint32_t bytes = (uint32_t)(L * CS);
    if (tid == 0) {
      fence_async_smem();
      mbar_arrive_expect_tx(mbar, (uint32_t)(nv * n_in) * bytes);
    }
    __syncwarp();
    const int step = nthr < 32 ? nthr : 32;
    for (int i = tid; i < nv * n_in; i += step) {
      const int gl = i / n_in, c = i - gl * n_in;
      const bool second = c > 0 && pair_start<R, LAYOUT>(c - 1);
      const int c0 = second ? c - 1 : c;
      const int w = pair_width<R, LAYOUT>(c0);
      bulk_copy_g2s(smem_u32(smem_raw + c0 * us + (gl * w + (second ? 1 : 0)) * (L * CS)),
                    spec + set_slot<MAP>(c) * a.cs + (int64_t)(line0 + gl) * L, bytes, mbar);
    }
  }
  int mxi, myi, rowi;
  line_modes(a, valid ? line : 0, mxi, myi, rowi);
  R kpx = R(0), kpy = R(0);
  W phx{}, phy{};
  if (a.stag) {
    stag_axis(a, 0, mxi, kpx, phx);
    if (a.ndim == 3) stag_axis(a, 1, myi, kpy, phy);
  }
  const Coef<R>* trow = a.tab + (int64_t)rowi * a.tab_row;
  // the push's coefficient entries: start bringing them into L2 now
#pragma unroll
  for (int m = grp; m < EPT; m += G) {
    const int l = t + T * m;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(trow + coef_entry(l, L)));
  }
  // bounded wait; on expiry the error word is set and one more bounded wait lets
  // copies still in flight land before the buffers are used
  if (!mbar_wait(mbar, phase, kWaitIters)) {
    int* err = a.err ? a.err : a.chk_err;
    if (err) atomicOr(err, kErrStageWait);
    mbar_wait(mbar, phase, kWaitIters);
  }

#pragma unroll 1
  for (int c = 0, u = 0, w; c < n_in; c += w, ++u) {
    w = pair_width<R, LAYOUT>(c);
    if (GRP && u % G != grp) continue;
    if constexpr (sizeof(R) == 4) {
      if (w == 2) {
        const float2* s0 = reinterpret_cast<const float2*>(smem_raw + c * us + g2);
        C2* buf = reinterpret_cast<C2*>(smem_raw + c * us + g2);
        C2 v[EPT];
#pragma unroll
        for (int m = 0; m < EPT; ++m) {
          const float2 x = s0[t + T * m], y = s0[L + t + T * m];
          v[m] = C2{F2{x.x, y.x}, F2{x.y, y.y}};
        }
        line_fft_fwd<F2, L, EPT, PF>(v, buf, tw, t, gx, bar);
#pragma unroll
        for (int m = 0; m < EPT; ++m) buf[own_pos<L, EPT, 16>(t, m, gx)] = v[m];
        continue;
      }
    }
    C* buf = reinterpret_cast<C*>(smem_raw + c * us + g1);
    C v[EPT];
#pragma unroll
    for (int m = 0; m < EPT; ++m) v[m] = buf[t + T * m];
    line_fft_fwd<R, L, EPT, PF>(v, buf, tw, t, gx1, bar);
#pragma unroll
    for (int m = 0; m < EPT; ++m) buf[own_pos<L, EPT, CS>(t, m, gx1)] = v[m];
  }
  if (G > 1) __syncthreads();  // every group's spectra are in their units

  if (a.scheme == 0) {
    if (a.stag)
      push_line_units<R, L, LAYOUT, EPT, true, false>(smem_raw, us, g1, g2, gx, a, trow, t, grp, G, mxi, myi, kpx, kpy, phx, phy);
    else
      push_line_units<R, L, LAYOUT, EPT, false, false>(smem_raw, us, g1, g2, gx, a, trow, t, grp, G, mxi, myi, kpx, kpy, phx, phy);
  } else {
    if (a.stag)
      push_line_units<R, L, LAYOUT, EPT, true, true>(smem_raw, us, g1, g2, gx, a, trow, t, grp, G, mxi, myi, kpx, kpy, phx, phy);
    else
      push_line_units<R, L, LAYOUT, EPT, false, true>(smem_raw, us, g1, g2, gx, a, trow, t, grp, G, mxi, myi, kpx, kpy, phx, phy);
  }
  if (G > 1) __syncthreads();  // every mode is pushed

#pragma unroll 1
  for (int c = 0, u = 0, w; c < n_out; c += w, ++u) {
    w = pair_width<R, LAYOUT>(c);
    if (GRP && u % G != G - 1 - grp) continue;
    C* dst = spec + set_slot<MAP>(c) * a.cs + (int64_t)line * L;
    [[maybe_unused]] const int64_t next = (set_slot<MAP>(c + 1) - set_slot<MAP>(c)) * a.cs;  // a pair's second
    if constexpr (sizeof(R) == 4) {
      if (w == 2) {
        C2* buf = reinterpret_cast<C2*>(smem_raw + c * us + g2);
        C2 v[EPT];
#pragma unroll
        for (int m = 0; m < EPT; ++m) v[m] = buf[own_pos<L, EPT, 16>(t, m, gx)];
        line_fft_inv<F2, L, EPT, PF>(v, buf, tw, t, gx, bar);
        if (valid) {
#pragma unroll
          for (int m = 0; m < EPT; ++m) {
            dst[t + T * m] = make_float2(v[m].x.a, v[m].y.a);
            dst[next + t + T * m] = make_float2(v[m].x.b, v[m].y.b);
          }
        }
        continue;
      }
    }
    C* buf = reinterpret_cast<C*>(smem_raw + c * us + g1);
    C v[EPT];
#pragma unroll
    for (int m = 0; m < EPT; ++m) v[m] = buf[own_pos<L, EPT, CS>(t, m, gx1)];
    line_fft_inv<R, L, EPT, PF>(v, buf, tw, t, gx1, bar);
    if (valid) {
#pragma unroll
      for (int m = 0; m < EPT; ++m) dst[t + T * m] = v[m];
    }
  }
  return true;
}

// Grid (line blocks, sets: 2 for the six 2D components), block (T, lines per CTA,
// component groups); up to 512 threads (128 registers), or without groups (GRP false) 256,
// or one line's threads where these are more (4096 points by 8 elements).  FP32 groups are
// whole warps: with several, T times the lines per CTA is a multiple of 32.
template <typename R, int L, int LAYOUT, int EPT, bool GRP>
__global__ void __launch_bounds__(GRP || EPT == 4 || FFTPlan<L, EPT>::kT > 256 ? 512 : 256)
k_line_pair(PushArgs<R> a, const typename Types<R>::W* __restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t stage_mbar;
  pass_begin();
  const uint32_t mbar = smem_u32(&stage_mbar);
  if (threadIdx.x == 0 && threadIdx.y == 0 && threadIdx.z == 0) mbar_init(mbar, 1);
  auto body = [&](auto lay, auto map) {
    line_pair_body<R, L, decltype(lay)::value, EPT, GRP, decltype(map)::value>(
        a, tw, (int)blockIdx.x, (int)threadIdx.x, (int)threadIdx.y, (int)blockDim.y, (int)threadIdx.z, (int)blockDim.z,
        smem_raw, mbar, 0u);
  };
  if constexpr (LAYOUT == 1) {
    if (sizeof(R) == 4 || gridDim.y == 2) {
      if (blockIdx.y == 0) body(std::integral_constant<int, 2>{}, std::integral_constant<int, 1>{});
      else body(std::integral_constant<int, 3>{}, std::integral_constant<int, 2>{});
      return;
    }
  }
  if constexpr (LAYOUT != 1 || sizeof(R) == 8) body(std::integral_constant<int, LAYOUT>{}, std::integral_constant<int, 0>{});
}

}  // namespace psatd
