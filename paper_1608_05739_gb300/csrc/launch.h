// launch.h -- host-side launchers of the PSATD pass kernels, instantiated per
// precision and variant in the rows_* / push_* translation units.  L is the
// transform length along the pass axis (a power of two 8..4096, or 3 * 2^k for
// the *3 launchers); every launcher returns the launch's cudaError_t.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "persist.cuh"
#include "psatd_kernels.cuh"

namespace psatd {

// Launch of a pass that begins with pass_begin().  early: it may be scheduled while its
// predecessor in the stream drains, and waits there for its completion (programmatic
// dependent launch), which hides the launch latency and the drain of the last wave
// between the passes of a step.  The blocks then fill the SMs as the predecessor frees
// them, not evenly, so it pays for passes of many more blocks than fit at once, or short
// ones (the plans' rule: plan_early in capi.cu).
template <class... P, class... A>
static inline cudaError_t launch_pass(bool early, void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                                      cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

struct PassGeom {
  dim3 grid;
  int log_tb;      // lines per CTA = 1 << log_tb
  size_t smem;     // dynamic shared memory bytes
  bool early = false;  // launch_pass
  bool wide = false;   // 16 elements per thread (row_wide lengths)
};

// a0_off: optional device table of per-patch element offsets into the caller's
// arrays (input of launch_fwd_T, output of launch_inv_T); NULL: a0 * stride.
// TC = true: the tensor-core (split-FP16) variants, float data only.
template <typename R, int TC = 0>
cudaError_t launch_fwd_T(int L, bool r2c, const PassGeom& g, cudaStream_t st, const LineIO& io,
                         const void* tw, int64_t in_sa0, int64_t in_sb, int64_t out_sa0,
                         int64_t out_sk, const int64_t* a0_off = nullptr);
template <typename R, int TC = 0>
cudaError_t launch_inv_T(int L, bool c2r, const PassGeom& g, cudaStream_t st, const LineIO& io,
                         const void* tw, int64_t in_sa0, int64_t in_sk, int64_t out_sa0,
                         int64_t out_sb, const int64_t* a0_off = nullptr);
// EPT: 8 or 16 elements per thread (radix-8 / radix-16 stages); TC needs 16.  LS: the
// layouts 0, 1 (LS 0) or 2, 3 (LS 1), a translation unit each.
template <typename R, int TC, int EPT, int LS>
cudaError_t launch_line_push(int L, int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                             const PushArgs<R>& a, const void* tw);

// the same passes for the mixed lengths L = 3 * 2^k (48..3072; R2C / C2R up to 1536), float only
template <typename R>
cudaError_t launch_fwd_T3(int L, bool r2c, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sb, int64_t out_sa0, int64_t out_sk,
                          const int64_t* a0_off = nullptr);
template <typename R>
cudaError_t launch_inv_T3(int L, bool c2r, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sk, int64_t out_sa0, int64_t out_sb,
                          const int64_t* a0_off = nullptr);
template <typename R, int LS>
cudaError_t launch_line_push3(int L, int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                              const PushArgs<R>& a, const void* tw);

// the same passes for the mixed lengths L = 5 * 2^k (80..1280), float only
template <typename R>
cudaError_t launch_fwd_T5(int L, bool r2c, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sb, int64_t out_sa0, int64_t out_sk,
                          const int64_t* a0_off = nullptr);
template <typename R>
cudaError_t launch_inv_T5(int L, bool c2r, const PassGeom& g, cudaStream_t st, const LineIO& io, const void* tw,
                          int64_t in_sa0, int64_t in_sk, int64_t out_sa0, int64_t out_sb,
                          const int64_t* a0_off = nullptr);
template <typename R, int LS>
cudaError_t launch_line_push5(int L, int layout, dim3 grid, int tb, int groups, size_t smem, cudaStream_t st,
                              const PushArgs<R>& a, const void* tw);

// Persistent batch passes (persist.cuh): FAM 0 power-of-two lengths, 1 the 3 * 2^k
// lengths (float, TC = 0).  `grid` CTAs of kPersistThreads threads; *occ (if not
// NULL) receives the CTAs per SM the kernel can keep resident.
template <typename R, int TC, int FAM>
cudaError_t launch_persist_x(bool fwd, int grid, cudaStream_t st, const XClassArgs* cls, const PersistQueue& q,
                             int* occ = nullptr);
template <typename R, int TC, int FAM>
cudaError_t launch_persist_push(int layout, int n_in, int grid, cudaStream_t st, const PushArgs<R>* cls,
                                const void* const* tws, const PersistQueue& q, int* occ = nullptr);

template <typename R>
cudaError_t launch_fdtd(int ndim, int scheme, int64_t nx, int64_t ny, int64_t nz, const double* d,
                        double dt, double c, double eps0, void* const E[3], void* const B[3],
                        const void* const J[3], int nsteps, cudaStream_t st);

}  // namespace psatd
