// launch_impl.cuh -- templated launchers with the switch over the transform
// length; included by the per-precision translation units.
#pragma once
#include "launch.h"
#include "pair_push.cuh"
#include "pair_rows.cuh"

namespace psatd {

// The FP32 passes without tensor cores run in pairs (pair_rows.cuh, pair_push.cuh).
template <typename R, int TC> constexpr bool kPairs = sizeof(R) == 4 && TC == 0;

// Dynamic shared-memory opt-in (static shared memory adds to the request).  The
// carveout is left to the driver: a maximal shared carveout shrinks the L1 that
// holds the twiddle tables and was measured slower.
template <typename K>
static cudaError_t set_smem(K kern, size_t smem) {
  if (smem > 32 * 1024)
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return cudaSuccess;
}

template <typename R, int TC, int L, bool R2C, bool LOC>
static cudaError_t fwd_T_L_k(const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw, int64_t a, int64_t b,
                           int64_t c, int64_t d, const int64_t* off) {
  typedef typename Types<R>::W W;
  constexpr int T = FFTPlan<L, RowEPT<L, R>::value>::kT;
  cudaError_t e;
  if constexpr (kPairs<R, TC>) {
    const unsigned pairs = g.log_tb > 0 ? 1u << (g.log_tb - 1) : 1u;
    const size_t smem = (size_t)pairs * L * sizeof(C2);
    auto kern = k_fwd_P<L, R2C, LOC>;
    if ((e = set_smem(kern, smem)) != cudaSuccess) return e;
    return launch_pass(g.early, kern, g.grid, dim3(T, pairs), smem, st, io, static_cast<const W*>(tw), a, b, c, d, g.log_tb, off);
  } else {
    if constexpr (row_wide(L, sizeof(R) == 4) && !LOC) {
      if (g.wide) {
        auto kern = k_fwd_T<R, L, R2C, TC, LOC, 16>;
        if ((e = set_smem(kern, g.smem)) != cudaSuccess) return e;
        return launch_pass(g.early, kern, g.grid, dim3(L / 16, 1u << g.log_tb), g.smem, st, io, static_cast<const W*>(tw), a,
                           b, c, d, g.log_tb, off);
      }
    }
    auto kern = k_fwd_T<R, L, R2C, TC, LOC>;
    if ((e = set_smem(kern, g.smem)) != cudaSuccess) return e;
    return launch_pass(g.early, kern, g.grid, dim3(T, 1u << g.log_tb), g.smem, st, io, static_cast<const W*>(tw), a, b, c, d,
                       g.log_tb, off);
  }
  return cudaGetLastError();
}
template <typename R, int TC, int L>
static cudaError_t fwd_T_L(bool r2c, const PassGeom& g, cudaStream_t st, const LineIO& io,
                           const void* tw, int64_t a, int64_t b, int64_t c, int64_t d, const int64_t* off) {
  if (!r2c) return fwd_T_L_k<R, TC, L, false, false>(g, st, io, tw, a, b, c, d, off);
  if constexpr (L <= 2048)
    return io.loc.px ? fwd_T_L_k<R, TC, L, true, true>(g, st, io, tw, a, b, c, d, off)
                     : fwd_T_L_k<R, TC, L, true, false>(g, st, io, tw, a, b, c, d, off);
  else return cudaErrorInvalidValue;
}

template <typename R, int TC, int L, bool C2R, bool LOC>
static cudaError_t inv_T_L_k(const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw, int64_t a, int64_t b,
                           int64_t c, int64_t d, const int64_t* off) {
  typedef typename Types<R>::W W;
  constexpr int T = FFTPlan<L, RowEPT<L, R>::value>::kT;
  cudaError_t e;
  if constexpr (kPairs<R, TC>) {
    const unsigned pairs = g.log_tb > 0 ? 1u << (g.log_tb - 1) : 1u;
    const size_t smem = (size_t)pairs * L * sizeof(C2);
    auto kern = k_inv_P<L, C2R, LOC>;
    if ((e = set_smem(kern, smem)) != cudaSuccess) return e;
    return launch_pass(g.early, kern, g.grid, dim3(T, pairs), smem, st, io, static_cast<const W*>(tw), a, b, c, d, g.log_tb, off);
  } else {
    if constexpr (row_wide(L, sizeof(R) == 4) && !LOC) {
      if (g.wide) {
        auto kern = k_inv_T<R, L, C2R, TC, LOC, 16>;
        if ((e = set_smem(kern, g.smem)) != cudaSuccess) return e;
        return launch_pass(g.early, kern, g.grid, dim3(L / 16, 1u << g.log_tb), g.smem, st, io, static_cast<const W*>(tw), a,
                           b, c, d, g.log_tb, off);
      }
    }
    auto kern = k_inv_T<R, L, C2R, TC, LOC>;
    if ((e = set_smem(kern, g.smem)) != cudaSuccess) return e;
    return launch_pass(g.early, kern, g.grid, dim3(T, 1u << g.log_tb), g.smem, st, io, static_cast<const W*>(tw), a, b, c, d,
                       g.log_tb, off);
  }
  return cudaGetLastError();
}
template <typename R, int TC, int L>
static cudaError_t inv_T_L(bool c2r, const PassGeom& g, cudaStream_t st, const LineIO& io,
                           const void* tw, int64_t a, int64_t b, int64_t c, int64_t d, const int64_t* off) {
  if (!c2r) return inv_T_L_k<R, TC, L, false, false>(g, st, io, tw, a, b, c, d, off);
  if constexpr (L <= 2048)
    return io.loc.px ? inv_T_L_k<R, TC, L, true, true>(g, st, io, tw, a, b, c, d, off)
                     : inv_T_L_k<R, TC, L, true, false>(g, st, io, tw, a, b, c, d, off);
  else return cudaErrorInvalidValue;
}

template <typename R, int TC, int EPT, int L, int LAYOUT, bool GRP>
static auto push_kernel() {
  // radix-16 lines run in groups by default and share one kernel for any count; the others
  // keep a plain kernel, 2 to 4 % faster than the group one with a single group
  if constexpr (TC == 0) return k_line_pair<R, L, LAYOUT, EPT, GRP || (EPT == 16 && sizeof(R) == 4)>;
  else return k_line_push<R, L, LAYOUT, TC, EPT, GRP>;
}

template <typename R, int TC, int EPT, int L, int LS>
static cudaError_t push_L(int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                          const PushArgs<R>& a, const void* tw) {
  typedef typename Types<R>::W W;
  if constexpr (L < EPT || (EPT == 4 && L > 128)) {
    return cudaErrorInvalidValue;
  } else {
    const dim3 block(FFTPlan<L, EPT>::kT, tb, groups);
    // component groups: their own instantiation; FP32 groups are whole warps
    constexpr bool kGrpOk = TC ? EPT == 16 : true;
    if (groups > 1 && (!kGrpOk || (kPairs<R, TC> && (block.x * block.y) % 32 != 0))) return cudaErrorInvalidValue;
    if constexpr (TC == 0) {  // the units alone; the six 2D components: the larger set's
      const bool sets = layout == 1 && push_sets(sizeof(R) == 4, grid.x);
      smem = (size_t)(sets ? 3 + 2 * a.form : a.n_in) * tb * L * 2 * sizeof(R);
      if (sets) grid.y = 2;
    }
    cudaError_t e;
#define PSATD_PUSH_LAUNCH(LAY, GRP)                                            \
  {                                                                            \
    auto kern = push_kernel<R, TC, EPT, L, LAY, GRP>();                        \
    if ((e = set_smem(kern, smem)) != cudaSuccess) return e;                   \
    return launch_pass(a.early != 0, kern, grid, block, smem, st, a, static_cast<const W*>(tw)); \
  }
#define PSATD_PUSH_CASE(LAY)                                                   \
  case LAY: {                                                                  \
    if constexpr (kGrpOk) {                                                    \
      if (groups > 1) PSATD_PUSH_LAUNCH(LAY, true)                             \
      else PSATD_PUSH_LAUNCH(LAY, false)                                       \
    } else {                                                                   \
      PSATD_PUSH_LAUNCH(LAY, false)                                            \
    }                                                                          \
    break;                                                                     \
  }
    if constexpr (LS == 0) {
      switch (layout) {
        PSATD_PUSH_CASE(0)
        PSATD_PUSH_CASE(1)
        default: return cudaErrorInvalidValue;
      }
    } else {
      switch (layout) {
        PSATD_PUSH_CASE(2)
        PSATD_PUSH_CASE(3)
        default: return cudaErrorInvalidValue;
      }
    }
#undef PSATD_PUSH_CASE
#undef PSATD_PUSH_LAUNCH
    return cudaGetLastError();
  }
}

// The tensor-core variants exist from L = 16 on (their first radix-16 stage).
#define PSATD_L_SWITCH(FN, ...)                                   \
  switch (L) {                                                    \
    case 8: if constexpr (!TC) return FN<R, TC, 8>(__VA_ARGS__);  \
            else return cudaErrorInvalidValue;                    \
    case 16: return FN<R, TC, 16>(__VA_ARGS__);                   \
    case 32: return FN<R, TC, 32>(__VA_ARGS__);                   \
    case 64: return FN<R, TC, 64>(__VA_ARGS__);                   \
    case 128: return FN<R, TC, 128>(__VA_ARGS__);                 \
    case 256: return FN<R, TC, 256>(__VA_ARGS__);                 \
    case 512: return FN<R, TC, 512>(__VA_ARGS__);                 \
    case 1024: return FN<R, TC, 1024>(__VA_ARGS__);               \
    case 2048: return FN<R, TC, 2048>(__VA_ARGS__);               \
    case 4096: return FN<R, TC, 4096>(__VA_ARGS__);               \
    default: return cudaErrorInvalidValue;                        \
  }

// Mixed lengths 3 * 2^k (FP32, no tensor-core stages).
#define PSATD_L3_SWITCH(FN, ...)                         \
  switch (L) {                                           \
    case 48: return FN<R, 0, 48>(__VA_ARGS__);           \
    case 96: return FN<R, 0, 96>(__VA_ARGS__);           \
    case 192: return FN<R, 0, 192>(__VA_ARGS__);         \
    case 384: return FN<R, 0, 384>(__VA_ARGS__);         \
    case 768: return FN<R, 0, 768>(__VA_ARGS__);         \
    case 1536: return FN<R, 0, 1536>(__VA_ARGS__);       \
    case 3072: return FN<R, 0, 3072>(__VA_ARGS__);       \
    default: return cudaErrorInvalidValue;               \
  }

// Mixed lengths 5 * 2^k (FP32, no tensor-core stages).
#define PSATD_L5_SWITCH(FN, ...)                         \
  switch (L) {                                           \
    case 80: return FN<R, 0, 80>(__VA_ARGS__);           \
    case 160: return FN<R, 0, 160>(__VA_ARGS__);         \
    case 320: return FN<R, 0, 320>(__VA_ARGS__);         \
    case 640: return FN<R, 0, 640>(__VA_ARGS__);         \
    case 1280: return FN<R, 0, 1280>(__VA_ARGS__);       \
    default: return cudaErrorInvalidValue;               \
  }

template <typename R>
cudaError_t launch_fwd_T5(int L, bool r2c, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sb, int64_t out_sa0, int64_t out_sk, const int64_t* a0_off) {
  PSATD_L5_SWITCH(fwd_T_L, r2c, g, st, io, tw, in_sa0, in_sb, out_sa0, out_sk, a0_off)
}
template <typename R>
cudaError_t launch_inv_T5(int L, bool c2r, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sk, int64_t out_sa0, int64_t out_sb, const int64_t* a0_off) {
  PSATD_L5_SWITCH(inv_T_L, c2r, g, st, io, tw, in_sa0, in_sk, out_sa0, out_sb, a0_off)
}
template <typename R, int LS>
cudaError_t launch_line_push5(int L, int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                              const PushArgs<R>& a, const void* tw) {
  switch (L) {
    case 80: return push_L<R, 0, 20, 80, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 160: return push_L<R, 0, 20, 160, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 320: return push_L<R, 0, 20, 320, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 640: return push_L<R, 0, 20, 640, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 1280: return push_L<R, 0, 20, 1280, LS>(layout, grid, tb, groups, smem, st, a, tw);
    default: return cudaErrorInvalidValue;
  }
}

template <typename R>
cudaError_t launch_fwd_T3(int L, bool r2c, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sb, int64_t out_sa0, int64_t out_sk, const int64_t* a0_off) {
  PSATD_L3_SWITCH(fwd_T_L, r2c, g, st, io, tw, in_sa0, in_sb, out_sa0, out_sk, a0_off)
}
template <typename R>
cudaError_t launch_inv_T3(int L, bool c2r, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sk, int64_t out_sa0, int64_t out_sb, const int64_t* a0_off) {
  PSATD_L3_SWITCH(inv_T_L, c2r, g, st, io, tw, in_sa0, in_sk, out_sa0, out_sb, a0_off)
}
template <typename R, int LS>
cudaError_t launch_line_push3(int L, int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                              const PushArgs<R>& a, const void* tw) {
  switch (L) {
    case 48: return push_L<R, 0, 12, 48, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 96: return push_L<R, 0, 12, 96, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 192: return push_L<R, 0, 12, 192, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 384: return push_L<R, 0, 12, 384, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 768: return push_L<R, 0, 12, 768, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 1536: return push_L<R, 0, 12, 1536, LS>(layout, grid, tb, groups, smem, st, a, tw);
    case 3072: return push_L<R, 0, 12, 3072, LS>(layout, grid, tb, groups, smem, st, a, tw);
    default: return cudaErrorInvalidValue;
  }
}

template <typename R, int TC>
cudaError_t launch_fwd_T(int L, bool r2c, const PassGeom& g, cudaStream_t st, const LineIO& io,
                         const void* tw, int64_t in_sa0, int64_t in_sb, int64_t out_sa0,
                         int64_t out_sk, const int64_t* a0_off) {
  PSATD_L_SWITCH(fwd_T_L, r2c, g, st, io, tw, in_sa0, in_sb, out_sa0, out_sk, a0_off)
}

template <typename R, int TC>
cudaError_t launch_inv_T(int L, bool c2r, const PassGeom& g, cudaStream_t st, const LineIO& io,
                         const void* tw, int64_t in_sa0, int64_t in_sk, int64_t out_sa0,
                         int64_t out_sb, const int64_t* a0_off) {
  PSATD_L_SWITCH(inv_T_L, c2r, g, st, io, tw, in_sa0, in_sk, out_sa0, out_sb, a0_off)
}

template <typename R, int TC, int EPT, int LS>
static cudaError_t push_L_e(int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                            const PushArgs<R>& a, const void* tw, int L) {
#define PUSH_E(LL) push_L<R, TC, EPT, LL, LS>
  switch (L) {
    case 8: if constexpr (!TC) return PUSH_E(8)(layout, grid, tb, groups, smem, st, a, tw);
            else return cudaErrorInvalidValue;
    case 16: return PUSH_E(16)(layout, grid, tb, groups, smem, st, a, tw);
    case 32: return PUSH_E(32)(layout, grid, tb, groups, smem, st, a, tw);
    case 64: return PUSH_E(64)(layout, grid, tb, groups, smem, st, a, tw);
    case 128: return PUSH_E(128)(layout, grid, tb, groups, smem, st, a, tw);
    case 256: return PUSH_E(256)(layout, grid, tb, groups, smem, st, a, tw);
    case 512: return PUSH_E(512)(layout, grid, tb, groups, smem, st, a, tw);
    case 1024: return PUSH_E(1024)(layout, grid, tb, groups, smem, st, a, tw);
    case 2048: return PUSH_E(2048)(layout, grid, tb, groups, smem, st, a, tw);
    case 4096: return PUSH_E(4096)(layout, grid, tb, groups, smem, st, a, tw);
    default: return cudaErrorInvalidValue;
  }
#undef PUSH_E
}

template <typename R, int TC, int EPT, int LS>
cudaError_t launch_line_push(int L, int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                             const PushArgs<R>& a, const void* tw) {
  return push_L_e<R, TC, EPT, LS>(layout, grid, tb, groups, smem, st, a, tw, L);
}

}  // namespace psatd
