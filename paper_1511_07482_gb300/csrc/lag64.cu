// FP64 lag kernels (lag.cuh): a translation unit of their own, compiled beside
// the FP32 ones.
#include "lag.cuh"

namespace kdefft {
template cudaError_t launch_lag<double>(int, int, int, const LagJob<double>&, cudaStream_t);
}  // namespace kdefft
