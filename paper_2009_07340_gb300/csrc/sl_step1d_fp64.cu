// 1D step kernels, precision mode SL_FP64: a thread per element, or an
// element's nodes over a group of lanes where the solve is small (the rule of
// split1d_fields; same results).
#include "sl_step1d_split.cuh"

namespace sl {
cudaError_t launch_step1d_fp64(const Step1DArgs &a, int N, cudaStream_t st)
{
    const int S = split1d_fields(N, a.K, a.M, a.ncomp, a.S, a.C, a.T, a.nsm);
    return S > 0 ? launch_split1d(a, N, S, st) : launch_step1d_mode<SL_FP64>(a, N, st);
}
size_t step1d_smem_bytes_fp64(int N, int S, int T) { return step1d_smem_bytes_t<SL_FP64>(N, S, T); }
cudaError_t launch_step1d_batch_fp64(const Batch1DLaunch &b, int N, cudaStream_t st) { return launch_sl1d_step_kernel_batch_mode<SL_FP64>(b, N, st); }
cudaError_t preload_step1d_fp64()
{
    const cudaError_t e = preload_step1d_mode<SL_FP64>();
    return e != cudaSuccess ? e : preload_split1d_seq(std::make_integer_sequence<int, kMaxN - 2>{});
}
}  // namespace sl
