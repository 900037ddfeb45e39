// push_modes.h -- which modes of a line the component groups of the fused pass update
// (pair_push.cuh), in code that host compilers take too.
#pragma once

#ifdef __CUDACC__
#define PSATD_HD __host__ __device__ __forceinline__
#else
#define PSATD_HD inline
#endif

namespace psatd {

// Table entry of mode l of a line of L points: |m| along the axis.
PSATD_HD constexpr int coef_entry(int l, int L) { return l <= L / 2 ? l : L - l; }

// Modes t + T m of a thread, m < EPT: group grp of G takes m = grp, grp + G, .. two an
// iteration, coefficients of the next two loaded before the update of this two.  load(m)
// and update(m, q) are called with m < EPT alone: FP64 lines of 4 elements per thread run
// in up to 6 groups, of which the last two have no mode.
template <int EPT, class Load, class Update>
PSATD_HD void push_mode_pairs(int grp, int G, Load load, Update update) {
  if (grp >= EPT) return;
  auto second = [&](int m) { return m + G < EPT ? m + G : m; };
  decltype(load(0)) qn[2] = {load(grp), load(second(grp))};
#ifdef __CUDACC__
#pragma unroll 1
#endif
  for (int m0 = grp; m0 < EPT; m0 += 2 * G) {
    const decltype(load(0)) q[2] = {qn[0], qn[1]};
    const int mn = m0 + 2 * G;
    if (mn < EPT) {
      qn[0] = load(mn);
      qn[1] = load(second(mn));
    }
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int h = 0; h < 2; ++h) {
      const int m = m0 + G * h;
      if (m >= EPT) break;
      update(m, q[h]);
    }
  }
}

}  // namespace psatd
