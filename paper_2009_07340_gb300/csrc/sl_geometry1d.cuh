// sl_geometry1d.cuh -- which kernel a 1D solve runs on and how its sample fields
// are dealt out to CTAs: host arithmetic on sizes only.
#pragma once
#include <algorithm>

namespace sl {

constexpr int kMaxThreads1D = 256;  // elements (threads) per CTA in the 1D kernel
constexpr int kMaxCluster1D = 8;    // CTAs per sample field (portable cluster size)
constexpr int kSplitMaxThreads = 512;

// Lanes per element of the split kernel (five at least: its chains).
constexpr int split1d_lanes(int N) { return N <= 8 ? 8 : 16; }

// Launch geometry of the 1D step: C CTAs per sample field (a cluster above
// max_threads elements), T thread slots per field in each, S fields per CTA.
//
// S: the step is bound by the arithmetic of the warps an SM is given, so the
// rule takes the S that leaves the most loaded SM the fewest warps, counting
// whole warps (a CTA of S K threads pads to one) and whole CTAs per SM; of
// equal ones the largest (fewer coefficient tables).  A small solve spreads
// over the SMs that way: 256 samples of 8 elements are 64 one-warp CTAs
// instead of 8 of 256 threads (a whole solve of 100 FP64 steps at N = 6 on the
// thread-per-element kernel 1.30 ms instead of 2.65), and 10000 samples of 20 elements take 8 fields (160 threads, no
// padding) instead of 12 (4 % faster at N = 9).
// C: the fewest warps over the field's CTAs for the same reason; of equal
// ones the smallest cluster.  777 elements take 5 CTAs of 156 slots
// instead of 4 of 195 (501 fields, mixed, N = 11: 11 % faster).
inline void geometry1d(int K, int M, int nsm, int max_threads, int &S, int &C, int &T)
{
    auto warps = [](int threads) { return (threads + 31) / 32; };
    C = (K + max_threads - 1) / max_threads;
    if (C > 1) {
        for (int c = C + 1; c <= kMaxCluster1D; ++c)
            if (c * warps((K + c - 1) / c) < C * warps((K + C - 1) / C)) C = c;
        T = (K + C - 1) / C;
        S = 1;
        return;
    }
    T = K;
    S = 1;
    long long best = -1;
    for (int s = 1; s <= max_threads / K && s <= M; ++s) {
        const long long ctas = (M + s - 1) / s, load = (ctas + nsm - 1) / nsm * warps(s * K);
        if (best < 0 || load <= best) {
            best = load;
            S = s;
        }
    }
}

// Fields per CTA of the split kernel (sl_step1d_split.cuh), 0 where the thread-per-element kernel is
// the faster one: by the FP64 instructions per step of the most loaded SM,
// where up to four warps (one per sub-partition) take the time of one.
// At the line, 30 steps, thread per element and split: 31 elements of 150
// samples at N = 6 353 and 234 us, at N = 16 1813 and 882; 8 of 1000 at N = 8
// 555 and 477, at N = 16 1811 and 1536; on its other side 16 of 1000 take 610 us
// at N = 8, one element per thread.
//
// N = 2 stays with the thread-per-element kernel: fewer instructions there, and
// never more warps than eight lanes per element take.
inline int split1d_fields(int N, int K, int M, int ncomp, int S1, int C1, int T1, int nsm)
{
    const int G = split1d_lanes(N);
    if (N < 3 || ncomp != 1 || C1 != 1 || K * G > kSplitMaxThreads) return 0;
    auto load = [=](int S, int threads) {
        const long long ctas = (M + S - 1) / S, warps = (ctas + nsm - 1) / nsm * ((threads + 31) / 32);
        return std::max(4ll, warps);
    };
    int best_S = 0;
    long long best = (6ll * N * N + 22 * N) * load(S1, S1 * T1);
    for (int S = 1; S * K * G <= kSplitMaxThreads && S <= M; ++S) {
        const long long cost = (8ll * N + 60) * load(S, S * K * G);
        if (cost < best) {
            best = cost;
            best_S = S;
        }
    }
    return best_S;
}

}  // namespace sl
