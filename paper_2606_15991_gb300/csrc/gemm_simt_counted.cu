// FP32 GEMM, the instances that count their writes.
#include "gemm_f32.cuh"

namespace tp {

cudaError_t launch_f32_counted(const SimtArgs& p, int64_t programs, int sms, cudaStream_t st) {
  return launch<true>(p, programs, sms, st);
}

}  // namespace tp
