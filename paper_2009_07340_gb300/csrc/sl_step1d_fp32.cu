// 1D step kernels, precision mode SL_FP32: packed from N = 4 on
// (sl_step1d_f2.cuh), scalar at N = 2 and 3 (sl_step1d.cuh), with one and two
// fields per sample alike.  With every node difference formed once, the packed
// kernel is the faster one from N = 4: 30 steps of 2048 sample fields of 256
// elements take, scalar and packed, 121 and 121 us at N = 2, 162 and 166 at 3,
// 199 and 188 at 4, 240 and 239 at 5, 403 and 379 at 8, 1143 and 1044 at 16.
#include "sl_step1d_f2.cuh"

namespace sl {
constexpr int kPackedFrom = 4;

cudaError_t launch_step1d_fp32(const Step1DArgs &a, int N, cudaStream_t st) { return launch_step1d_f2_mode<SL_FP32>(a, N, st); }
size_t step1d_smem_bytes_fp32(int N, int S, int T)
{
    return N < kPackedFrom ? step1d_smem_bytes_t<SL_FP32>(N, S, T) : step1d_f2_smem_bytes<SL_FP32>(N, S, T);
}
cudaError_t launch_step1d_batch_fp32(const Batch1DLaunch &b, int N, cudaStream_t st) { return launch_sl1d_step_kernel_f2_batch_mode<SL_FP32>(b, N, st); }
cudaError_t preload_step1d_fp32()
{
    const cudaError_t e = preload_step1d_seq<SL_FP32>(std::make_integer_sequence<int, kPackedFrom - 2>{});
    return e != cudaSuccess ? e : preload_step1d_f2_seq<SL_FP32, kPackedFrom>(std::make_integer_sequence<int, kMaxN - kPackedFrom + 1>{});
}
}  // namespace sl
