// 2D FP32 step kernels for N = 5 (one order per translation unit keeps the
// heavily unrolled Gram / Gauss-Jordan code of the orders compiling in parallel).
#include "sl_step2d_launch.cuh"

namespace sl {
cudaError_t launch_step2d_fp32_n5(const Step2DArgs &a, cudaStream_t st) { return launch_step2d_n<5, float>(a, st); }
cudaError_t launch_step2d_batch_fp32_n5(const Batch2DLaunch &b, cudaStream_t st) { return launch_step2d_batch_n<5, float>(b, st); }
cudaError_t preload_step2d_fp32_n5() { return preload_step2d_n<5, float>(); }
}  // namespace sl
