// push_f64_tetm.cu -- double instantiation of the fused last-axis FFT + PSATD push pass.
#include "launch_impl.cuh"

namespace psatd {
template cudaError_t launch_line_push<double, false, 8, 1>(int, int, dim3, int, int, size_t, cudaStream_t,
                                              const PushArgs<double>&, const void*);
template cudaError_t launch_line_push<double, false, 4, 1>(int, int, dim3, int, int, size_t, cudaStream_t,
                                              const PushArgs<double>&, const void*);
}  // namespace psatd
