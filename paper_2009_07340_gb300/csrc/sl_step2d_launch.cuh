// sl_step2d_launch.cuh -- the direct kernel's persistent form and the launchers
// of the 2D step: per step and phase the iterative kernel (sl_step2d_fast.cuh),
// then the direct one (sl_step2d.cuh) for the groups it flagged.
#pragma once
#include "sl_step2d_fast.cuh"

namespace sl {

// The direct kernel of one phase (see sl2d_cta): a persistent grid over the
// slot list the iterative kernel left.  With no flagged group it reads the
// list's length and exits; the last CTA to finish empties the list for the
// next launch.
template <int N, typename R, int PHASE, bool BATCH, int NCOMP = 1>
__global__ void __launch_bounds__(Geo2D<N, R, NCOMP>::kBlock, min_ctas2d<N, R>())
    sl2d_direct_kernel(const Step2DArgs a0, const Step2DArgs *__restrict__ args, const long long *__restrict__ prefix,
                       int ninst, int t)
{
    using G = Geo2D<N, R, NCOMP>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R *tab = reinterpret_cast<R *>(smem_raw);
    // node tables depend on N only (every instance of a batch class shares
    // them); computed once per context on the host (node_tables2d)
    const double *tabsrc = BATCH ? args[0].tab : a0.tab;
    const Step2DArgs &L = BATCH ? args[0] : a0;
    const unsigned count = *static_cast<volatile const unsigned *>(L.slot_ctl);
    const long long slot0 = BATCH ? 0 : a0.g0 / G::GPC;  // a launch starts on a slot boundary
    if (blockIdx.x < count) {
        for (int k = threadIdx.x; k < G::kTables; k += blockDim.x) tab[k] = R(tabsrc[k]);
        __syncthreads();
        for (unsigned i = blockIdx.x; i < count; i += gridDim.x) {
            const long long slot = L.slot_list[i];
            sl2d_cta<N, R, PHASE, BATCH, NCOMP>(a0, args, prefix, ninst, t, slot - slot0);
            __syncthreads();  // the slot's shared memory is free again
            if (threadIdx.x == 0) L.slot_mark[slot] = 0u;
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(L.slot_ctl + 1, 1u) == gridDim.x - 1) {  // every other CTA has read the length
            L.slot_ctl[0] = 0u;
            L.slot_ctl[1] = 0u;
        }
    }
}

template <int N, typename R, int NCOMP>
size_t smem2d()
{
    using G = Geo2D<N, R, NCOMP>;
    return sizeof(R) * (((G::kTables + 3) & ~3) + size_t(G::GPC) * G::kGroup);
}

// One phase over groups [g0, g1): for orders with the fast path, the fast
// kernel and then the direct kernel for the groups it flagged.
// CTAs of kernel K resident on the device at once (at least one per SM).
template <auto K>
unsigned resident_ctas(int block, size_t smem)
{
    static std::atomic<int> per_sm{0};  // queried once the kernel has been prepared
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        nsm = 1;
    if (per_sm.load() == 0) {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, K, block, smem) == cudaSuccess && per > 0)
            per_sm.store(per);
        else
            cudaGetLastError();
    }
    return unsigned(std::max(1, nsm) * std::max(1, per_sm.load()));
}

// The iterative kernel runs one CTA per slot of its own geometry; the direct
// kernel (SP lanes per row, fewer groups per CTA) is a persistent grid over
// the slots that one listed, at most one CTA per slot of the launch and no
// more than fit on the device at once.
// The mixed-precision form (an FP64 capacitance factor) exists for the FP32
// remap (one or two fields).
template <typename R>
constexpr bool kHasFac64 = std::is_same<R, float>::value;

template <int N, typename R, int NCOMP, bool BATCH>
cudaError_t launch_phase2d(int phase, long long groups, const Step2DArgs &b, const Step2DArgs *args,
                           const long long *prefix, int ninst, int t, bool f64c, cudaStream_t st,
                           LaunchThrottle *th)
{
    auto one = [&](auto kernel, auto geo, size_t smem, unsigned cap) -> cudaError_t {
        using G = decltype(geo);
        if (th) {
            const cudaError_t e = th->before();
            if (e != cudaSuccess) return e;
        }
        const unsigned grid = std::min(unsigned((groups + G::GPC - 1) / G::GPC), cap);
        kernel<<<grid, unsigned(G::kBlock), smem, st>>>(b, args, prefix, ninst, t);
        return th ? th->after(st) : cudaSuccess;
    };
    using GF = FGeo<N, R>;
    using GD = Geo2D<N, R, NCOMP>;
    constexpr unsigned kAll = ~0u;
    cudaError_t e;
    if (phase == 1) {
        constexpr auto k2 = sl2d_direct_kernel<N, R, 1, BATCH, NCOMP>;
        e = one(sl2d_fast_kernel<N, R, 1, BATCH, NCOMP>, GF{}, FSmem<N, R, 1, false>::bytes, kAll);
        if (e == cudaSuccess)
            e = one(k2, GD{}, smem2d<N, R, NCOMP>(), resident_ctas<k2>(GD::kBlock, smem2d<N, R, NCOMP>()));
    } else {
        constexpr auto k2 = sl2d_direct_kernel<N, R, 2, BATCH, NCOMP>;
        if constexpr (kHasFac64<R>) {
            e = f64c ? one(sl2d_fast_kernel<N, R, 2, BATCH, NCOMP, true>, GF{}, FSmem<N, R, 2, true>::bytes, kAll)
                     : one(sl2d_fast_kernel<N, R, 2, BATCH, NCOMP>, GF{}, FSmem<N, R, 2, false>::bytes, kAll);
        } else {
            e = one(sl2d_fast_kernel<N, R, 2, BATCH, NCOMP>, GF{}, FSmem<N, R, 2, false>::bytes, kAll);
        }
        if (e == cudaSuccess)
            e = one(k2, GD{}, smem2d<N, R, NCOMP>(), resident_ctas<k2>(GD::kBlock, smem2d<N, R, NCOMP>()));
    }
    return e;
}

template <int N, typename R, int NCOMP = 1>
cudaError_t launch_step2d_n(const Step2DArgs &a, cudaStream_t st)
{
    using G = Geo2D<N, R, NCOMP>;
    const long long groups = (long long)a.Kx * a.Ky * a.M;
    // a launch covers at most `chunk` groups (a multiple of the groups per CTA)
    const long long chunk =
        a.chunk > 0 ? std::min(groups, (a.chunk + G::GPC - 1) / G::GPC * G::GPC) : groups;
    Step2DArgs b = a;
    LaunchThrottle *th = a.chunk > 0 ? a.throttle : nullptr;
    for (int t = 0; t < a.nsteps; ++t) {
        for (int phase = 1; phase <= 2; ++phase)  // every group's faces before any remap
            for (long long g0 = 0; g0 < groups; g0 += chunk) {
                b.g0 = g0;
                b.g1 = std::min(groups, g0 + chunk);
                const cudaError_t e = launch_phase2d<N, R, NCOMP, false>(phase, b.g1 - g0, b, nullptr, nullptr, 0, t,
                                                                         a.f64_factor != 0, st, th);
                if (e != cudaSuccess) return e;
            }
    }
    return cudaGetLastError();
}

template <int N, typename R, int NCOMP, bool BATCH>
cudaError_t preload_phases2d()
{
    cudaError_t e = cudaSuccess;
    for (auto k : {sl2d_fast_kernel<N, R, 1, BATCH, NCOMP>, sl2d_direct_kernel<N, R, 1, BATCH, NCOMP>,
                   sl2d_fast_kernel<N, R, 2, BATCH, NCOMP>, sl2d_direct_kernel<N, R, 2, BATCH, NCOMP>})
        if (e == cudaSuccess) e = prepare_kernel(k);
    if constexpr (kHasFac64<R>)
        if (e == cudaSuccess) e = prepare_kernel(sl2d_fast_kernel<N, R, 2, BATCH, NCOMP, true>);
    return e;
}

// Prepares the single-instance kernels of one order for two fields.
template <int N, typename R>
cudaError_t preload_step2d_c2_n()
{
    return preload_phases2d<N, R, 2, false>();
}

// Prepares the kernels of one order (both phases, single and batched).
template <int N, typename R>
cudaError_t preload_step2d_n()
{
    cudaError_t e = preload_phases2d<N, R, 1, false>();
    if (e == cudaSuccess) e = preload_phases2d<N, R, 1, true>();
    return e;
}

// All instances of one order N, `nsteps` steps: per step both phases, each
// one launch (two with the fast path) over every instance's groups.
template <int N, typename R>
cudaError_t launch_step2d_batch_n(const Batch2DLaunch &b, cudaStream_t st)
{
    Step2DArgs none = {};
    for (int t = 0; t < b.nsteps; ++t)
        for (int phase = 1; phase <= 2; ++phase) {
            const cudaError_t e = launch_phase2d<N, R, 1, true>(phase, b.total_groups, none, b.args, b.prefix, b.ninst,
                                                                t, b.f64_factor != 0, st, nullptr);
            if (e != cudaSuccess) return e;
        }
    return cudaGetLastError();
}

}  // namespace sl
