// sl_step1d_split.cuh -- the FP64 1D step with an element's nodes dealt out to
// the lanes of a group: for solves too small to fill the chip.
//
// Bound.  An SM sub-partition completes one FP64 warp instruction in about 64
// clocks, whatever its active lanes, so a solve of few warps takes the time of
// one thread's instruction stream while most sub-partitions idle: with a
// thread per element (sl_step1d.cuh) about 6 N^2 + 22 N FP64 instructions per
// step.  Here a group of G lanes (8 up to N = 8, else 16) holds an element,
// lane j its node j.  The O(N^2) products and recurrences run one node per
// lane; the chains over the nodes (prefix and suffix products, sums) run one
// chain per lane, over operands in shared memory: about 8 N + 50 instructions.
// Every value is formed by the same operations in the same order as in
// sl_step1d.cuh, so that results are bitwise those of that kernel, whichever
// runs.  Measured: a whole
// solve of 256 samples of 8 elements at N = 6, 100 steps, 1.28 -> 0.56 ms; 30
// steps of 100 samples of 3 elements 0.35 -> 0.13 ms at N = 6, 1.81 -> 0.25 at 16.
#pragma once
#include <algorithm>

#include "sl_step1d.cuh"

namespace sl {

template <int N>
struct Split1D {
    static constexpr int G = split1d_lanes(N);  // lanes per element
    // per-element rows of G doubles: delta, F0 - delta, F1 - delta, raw weights,
    // their prefix products, pre0, suf0, pre1, suf1, phi*, E0, E1, r
    enum { DL, FA, FB, RAW, P0, S0, P1, S1, PP, PH, EA, EB, RW, ROWS };
    static constexpr int ES = ROWS * G + 2;  // an odd number of 16 bytes: a warp's elements in different banks
};

template <int N>
size_t split1d_smem(int S, int K, int threads)
{
    return sizeof(double) * (size_t(4) * S * K + size_t(threads / Split1D<N>::G) * Split1D<N>::ES);
}

template <int N>
__global__ void __launch_bounds__(kSplitMaxThreads) sl1d_split_kernel(const Step1DArgs a)
{
    using L = Split1D<N>;
    constexpr int G = L::G;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int K = a.K, S = a.S;
    double *sface = reinterpret_cast<double *>(smem_raw);  // [2 buf][2 side][S][K]
    const int g = threadIdx.x / G, j = threadIdx.x % G;
    double *eb = sface + 4 * S * K + g * L::ES;
    const bool slot = g < S * K;  // groups beyond it compute on zeros and write nothing
    const int sl = slot ? g / K : 0, kl = slot ? g - sl * K : 0;
    const int s = blockIdx.x * S + sl;
    const bool own = slot && s < a.M, active = own && j < N;
    const int jn = j < N ? j : N - 1;  // lanes beyond N repeat the last node

    const double *cf = static_cast<const double *>(a.coef);
    const double al = own ? cf[jn * K + kl] : 0.0, be = own ? cf[(N + jn) * K + kl] : 0.0;
    const double ga = own ? cf[(2 * N + jn) * K + kl] : 0.0;
    const double faL = cf[3 * N * K + kl], faR = cf[3 * N * K + kl + 1];
    const double fbL = cf[3 * N * K + K + 1 + kl], fbR = cf[3 * N * K + K + 1 + kl + 1];
    double z[N];
#pragma unroll
    for (int m = 0; m < N; ++m) z[m] = 4.0 * (a.xi[jn] - a.xi[m]);
    const double F0 = -4.0 * a.xi[jn], F1 = 4.0 * (1.0 - a.xi[jn]);
    double *Qg = static_cast<double *>(a.Q) + ((long long)s * K + kl) * N + jn;
    double q = own ? *Qg : 0.0;
    const int lnb = sl * K + (kl == 0 ? K - 1 : kl - 1), rnb = sl * K + (kl == K - 1 ? 0 : kl + 1);
    // this lane's chain of products (0: pre0, 1: suf0, 2: pre1, 3: suf1, 4 and above: the weights) and of sums
    const double *csrc = eb + G * (j < 2 ? L::FA : j < 4 ? L::FB : L::RAW);
    double *cdst = eb + G * (j == 0 ? L::P0 : j == 1 ? L::S0 : j == 2 ? L::P1 : j == 3 ? L::S1 : L::PP);
    const bool down = j == 1 || j == 3;
    const double *sx = eb + G * (j < 2 ? L::PH : j < 4 ? L::EA : L::EB);
    const double *sy = eb + G * (j == 0 || j == 2 ? L::EA : L::EB);
    bool bad = false;

    double dWn = (own && a.nsteps > 0) ? a.dW[s] : 0.0;
    for (int t = 0; t < a.nsteps; ++t) {
        const double dW = dWn;
        if (own && t + 1 < a.nsteps) dWn = a.dW[(long long)(t + 1) * a.M + s];

        // advance and compositional update relative to the middle node
        const double dl = fma(be, dW, al);
        const double c = __shfl_sync(0xffffffffu, q, N / 2, G);
        const double ph = fma(-ga, q, q - c);
        __syncwarp();  // the previous step's reads of these rows are done
        eb[L::DL * G + j] = dl;
        eb[L::FA * G + j] = F0 - dl;
        eb[L::FB * G + j] = F1 - dl;
        eb[L::PH * G + j] = ph;
        __syncwarp();
        double w = 1.0;
#pragma unroll
        for (int m = 0; m < N; ++m) {
            const double d = z[m] + (dl - eb[L::DL * G + m]);
            w *= m == jn ? 1.0 : d;
        }
        eb[L::RAW * G + j] = w;
        __syncwarp();
        {
            double acc = csrc[down ? N - 1 : 0];
            if (j < 5) cdst[down ? N - 1 : 0] = acc;
#pragma unroll
            for (int m = 1; m < N; ++m) {
                const int i = down ? N - 1 - m : m;
                acc *= csrc[i];
                if (j < 5) cdst[i] = acc;
            }
        }
        __syncwarp();
        {  // batch inversion of the weights, every lane up to its own
            double inv = 1.0 / eb[L::PP * G + N - 1], at = inv;
#pragma unroll
            for (int m = N - 1; m >= 1; --m) {
                if (m == jn) at = inv;
                inv *= eb[L::RAW * G + m];
            }
            w = jn > 0 ? at * eb[L::PP * G + jn - 1] : inv;
        }
        double E0, E1;
        {
            const double p0 = jn > 0 ? eb[L::P0 * G + jn - 1] : 1.0, s0 = jn < N - 1 ? eb[L::S0 * G + jn + 1] : 1.0;
            const double p1 = jn > 0 ? eb[L::P1 * G + jn - 1] : 1.0, s1 = jn < N - 1 ? eb[L::S1 * G + jn + 1] : 1.0;
            E0 = w * (p0 * s0);
            E1 = w * (p1 * s1);
        }
        eb[L::EA * G + j] = E0;
        eb[L::EB * G + j] = E1;
        __syncwarp();
        double acc = 0.0;  // e0, e1, g00, g01, g11 by lane
#pragma unroll
        for (int m = 0; m < N; ++m) acc = fma(sx[m], sy[m], acc);
        const double e0 = __shfl_sync(0xffffffffu, acc, 0, G), e1 = __shfl_sync(0xffffffffu, acc, 1, G);
        const double g00 = __shfl_sync(0xffffffffu, acc, 2, G), g01 = __shfl_sync(0xffffffffu, acc, 3, G);
        const double g11 = __shfl_sync(0xffffffffu, acc, 4, G);
        const double f0 = c + e0, f1 = c + e1;

        double *fL = sface + ((t & 1) * 2 + 0) * S * K, *fR = sface + ((t & 1) * 2 + 1) * S * K;
        if (slot && j == 0) {
            fL[g] = f0;
            fR[g] = f1;
        }
        __syncthreads();
        double gL, gR;
        {
            const double sigL = __dadd_rn(faL, __dmul_rn(fbL, dW)), sigR = __dadd_rn(faR, __dmul_rn(fbR, dW));
            double left = fR[lnb], right = fL[rnb];
            if (!a.periodic) {
                if (kl == 0) left = a.ghost[2 * t + 0];
                if (kl == K - 1) right = a.ghost[2 * t + 1];
            }
            gL = sigL > 0.0 ? left : f0;
            gR = sigR > 0.0 ? f1 : right;
        }
        double mu0, mu1;
        {
            const double G00 = a.inv_w2 + g00, G01 = g01, G11 = a.inv_w2 + g11;
            const double det = G00 * G11 - G01 * G01;
            const double idet = 1.0 / det;
            const double r0 = f0 - gL, r1 = f1 - gR;
            mu0 = (G11 * r0 - G01 * r1) * idet;
            mu1 = (G00 * r1 - G01 * r0) * idet;
            bad |= !(det > 0.0) || !isfinite(mu0) || !isfinite(mu1);
        }
        const double r = (ph - fma(E0, mu0, E1 * mu1)) * w;
        eb[L::RW * G + j] = r;
        __syncwarp();
        double A = eb[L::RW * G], P = z[0] - eb[L::DL * G];
#pragma unroll
        for (int k = 1; k < N; ++k) {
            const double d = z[k] - eb[L::DL * G + k];
            A = fma(A, d, eb[L::RW * G + k] * P);
            if (k + 1 < N) P *= d;
        }
        q = c + A;
    }
    if (active) {
        *Qg = q;
        if (bad) atomicOr(a.err, 1);
    }
}

template <int N>
cudaError_t launch_split1d_n(Step1DArgs a, int S, cudaStream_t st)
{
    const int threads = (S * a.K * Split1D<N>::G + 31) / 32 * 32;
    a.S = S;
    sl1d_split_kernel<N><<<unsigned((a.M + S - 1) / S), threads, split1d_smem<N>(S, a.K, threads), st>>>(a);
    return cudaGetLastError();
}

inline cudaError_t launch_split1d(const Step1DArgs &a, int N, int S, cudaStream_t st)
{
    switch (N) {
    case 3: return launch_split1d_n<3>(a, S, st);
    case 4: return launch_split1d_n<4>(a, S, st);
    case 5: return launch_split1d_n<5>(a, S, st);
    case 6: return launch_split1d_n<6>(a, S, st);
    case 7: return launch_split1d_n<7>(a, S, st);
    case 8: return launch_split1d_n<8>(a, S, st);
    case 9: return launch_split1d_n<9>(a, S, st);
    case 10: return launch_split1d_n<10>(a, S, st);
    case 11: return launch_split1d_n<11>(a, S, st);
    case 12: return launch_split1d_n<12>(a, S, st);
    case 13: return launch_split1d_n<13>(a, S, st);
    case 14: return launch_split1d_n<14>(a, S, st);
    case 15: return launch_split1d_n<15>(a, S, st);
    case 16: return launch_split1d_n<16>(a, S, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int... I>
cudaError_t preload_split1d_seq(std::integer_sequence<int, I...>)
{
    cudaError_t e = cudaSuccess;
    auto one = [&](auto f) {
        if (e == cudaSuccess) e = prepare_kernel(f);
    };
    (one(sl1d_split_kernel<I + 3>), ...);
    return e;
}

}  // namespace sl
