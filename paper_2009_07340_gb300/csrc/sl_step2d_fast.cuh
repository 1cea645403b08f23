// sl_step2d_fast.cuh -- the iterative (tensor-preconditioned) solves of the 2D
// step, every order and precision; what they do not finish goes to the direct
// kernel of sl_step2d.cuh.
//
// Method.  Within an element the particles of a sample move almost alike (one
// Wiener increment per sample, fields that vary little across an element), so
// the advected basis V is close to a tensor product V0 of two 1D
// advected-basis matrices: with x~_a the mean x of particle column a and y~_b
// the mean y of particle row b, V0[(b,a)][(j,i)] = h_i(x~_a) h_j(y~_b).  Its
// inverse is the tensor product of the 1D interpolation matrices Wx[i][a] =
// l~_a(xi_i) (the Lagrange basis on the x~, evaluated at the nodes) and Wy.
// Phase 1 iterates alpha += V0^{-1} (phi* - V alpha).  Phase 2 iterates
// q += G0^{-1} S^T (rhs - S q) on the stacked system S = [V; w B], with
// G0 = V0^T (I + w^2 E0^T E0) V0, E0 = B V0^{-1}, applied in the stable order
// V0^{-1} (I - E0^T C^{-1} E0) V0^{-T}, C = w^{-2} I + E0 E0^T (4N x 4N,
// assembled from 1D products, its null directions filled up, and inverted by
// its 4N row threads).  Both
// converge to the direct solution.  A group whose tensor factors are
// ill-conditioned (||Wx|| ||Wy|| above kCond: particles far outside the
// element) or whose iteration has not converged is flagged.
//
// Precision.  The preconditioner (Wx, Wy, C^{-1} and every pass through them)
// is FP32 in every mode: it sets how fast the iteration converges, not what
// it converges to.  The FP32 modes iterate on FP32 residuals.  SL_FP64 keeps
// the iterate, the basis and the residual in FP64 and solves for corrections
// by the FP32 iteration on the scaled residual (iterative refinement, as for
// a factor of lower precision: Wilkinson): each outer step gains five to six
// digits, so two or three FP64 residuals replace the seven to eight whole
// FP64 iterations of an FP64 preconditioner.  FP64 runs at 1/64 of the FP32
// rate on GB300 and bounds the FP64 kernels.
//
// Mapping.  A group of W warps per element-sample.  Up to N = 8 one warp (two
// nodes per lane from N = 6): its stages are ordered by __syncwarp instead of
// a named barrier, row operands are loaded once for both nodes, and the
// thread's row of C^{-1} stays in registers.  With one thread per node, two
// warps and a named barrier per stage at N = 8, the kernel waited on barriers
// and shared memory (43 % of the issue slots used; now 71 %, the shared-memory
// pipe 79 % busy in phase 2).  Measured, with the FP32 preconditioner and this
// mapping against FP64 passes and that one: 64 x 64 elements, N = 8, FP32, two
// steps of 64 samples at half the node-gap step 11.15 ms, now 5.73; 32 x 32,
// N = 6, FP64, one step of 32 samples 6.63 ms, now 1.86; 32 x 32, N = 5, FP32,
// two steps of 64 samples with new fields 0.85 ms, now 0.72; 19 x 23, N = 12,
// FP32, one step of 101 samples 2.97 ms, now 2.33.
// Above N = 8 the 4N face points need more than one warp: two, with two nodes
// per lane, up to N = 11 (a warp per 32 nodes, three or four, took 28.7, 35.1
// and 44.0 ns per element-sample at N = 9, 10, 11 on 32 x 32 elements of 16
// samples, now 25.5, 30.9 and 38.9), five at N = 12 (three nodes per lane in
// two warps spill: 60.1 against 59.0 ns).
#pragma once
#include "sl_step2d.cuh"

namespace sl {

template <int N, typename R>
struct FGeo {
    static constexpr int n = N * N;
    static constexpr bool kF64 = sizeof(R) == 8;
    // warps per group (FP64: one thread per node; its FP64 work is bound by
    // the FP64 pipe however it is dealt out)
    static constexpr int W = kF64 ? (n + 31) / 32 : (N <= 8 ? 1 : N <= 11 ? 2 : 5);
    static constexpr int TG = 32 * W;  // threads per group
    // lanes that hold nodes: whole rows of N where that needs no more slots, so
    // that a thread's nodes share their column i
    static constexpr int La0 = TG / N * N;
    static constexpr int La = (n + La0 - 1) / La0 == (n + TG - 1) / TG ? La0 : TG;
    static constexpr int NS = (n + La - 1) / La;  // nodes per thread: tig, tig + La, ...
    static constexpr int GPC = W == 1 ? 4 : (W == 2 ? 2 : 1);  // groups per CTA
    static constexpr int kBlock = GPC * TG;
    static constexpr int F = 4 * N;  // face points
    static_assert(F <= TG, "a thread per face point");
    __host__ __device__ static constexpr int r4(int v) { return (v + 3) & ~3; }
    // row stride for rows read by 16-byte loads of consecutive lanes: an odd
    // number of 16-byte units, so that eight rows fall in different banks
    __host__ __device__ static constexpr int odd4(int v) { return (((v + 3) / 4) | 1) * 4; }
    static constexpr int RS = r4(N);     // rows [j][i] of a node field
    static constexpr int NR = odd4(N);   // rows read across lanes
    static constexpr int NTP = odd4(n);  // rows of the particles' basis values by node
    static constexpr int kCB = 4;                       // pivot block of C's inversion
    static constexpr bool kRowsOneWarp = F <= 32;
    static constexpr int CR = odd4(F);                  // published pivot rows
    // per-group shared memory (floats)
    static constexpr int kW = N * NR;                   // one N x N table
    static constexpr int oW = 0;                        // Wx, Wx^T, Wy, Wy^T
    static constexpr int oG = oW + 4 * kW;              // l~(0), l~(1) in x, then in y: [4][RS]
    static constexpr int oDb = oG + 4 * RS;             // mean displacements [2][RS]
    static constexpr int oRed = oDb + 2 * RS;           // [2][W][2] maxima
    static constexpr int oA = oRed + r4(4 * W);         // node field
    static constexpr int oB = oA + N * NR;              // node field, transposed rows
    static constexpr int oVec = oB + N * NR;            // iterate, rows of RS; a transposed field meanwhile
    static constexpr int oRes = oVec + N * NR;          // residual: particles, then face points
    // (at least the published rows of C's inversion, which these hold before the iteration)
    static constexpr int oEnd1 = oRes + r4(n) + F > oA + 2 * kCB * CR ? oRes + r4(n) + F : oA + 2 * kCB * CR;
    static constexpr int oM = oEnd1;                    // Mx = Wx Wx^T, My
    static constexpr int oU = oM + 2 * kW;              // hvx, hvy; r / mu; M mu ([4][RS] each); u [4N]
    static constexpr int oH = oU + 12 * RS + F;         // hxT, hyT [N][NTP]
    // rows of C^{-1}: in the thread's registers up to N = 8; above, FP32's two
    // nodes per thread need those, and the rows are kept here
    static constexpr bool kCShared = !kF64 && N > 8 && W == 2;
    static constexpr int oC = oH + 2 * N * NTP;
    static constexpr int oEnd2 = oC + (kCShared ? F * CR : 0);
    // FP64 buffers (doubles): the iterate; phase 2 also the particles' y basis
    // by node, their x basis times the residual ([N][NT64] each) and the face residuals
    static constexpr int NT64 = ((n + 1) / 2 | 1) * 2;  // rows an odd number of 16 bytes apart
    static constexpr int kX64 = kF64 ? N * RS : 0;
    static constexpr int kZ64 = kF64 ? 2 * N * NT64 + F : 0;
    // per-CTA tables: Z [N][N], lambda, h0, h1, -4 xi, 4 (1 - xi)
    static constexpr int kTab = r4(N * N + 5 * N);
};

template <int N, typename R, int PHASE, bool FAC64>
struct FSmem {
    using G = FGeo<N, R>;
    // FAC64 (the mixed form's FP64 factor), after the group's buffers:
    // [4][N][N], [4][2][N], [8][N] and 88 doubles, then [4][N][N], [4N][4] and 56 floats
    static constexpr int kFac64 = FAC64 ? G::r4(2 * (4 * N * N + 16 * N + 88) + 4 * N * N + 16 * N + 56) : 0;
    static constexpr int kGroup =
        G::r4((PHASE == 1 ? G::oEnd1 : G::oEnd2 + 2 * G::kZ64) + 2 * G::kX64 + kFac64);
    static constexpr int kTabs = (G::kF64 ? 3 : 1) * G::kTab;  // FP64: the tables in FP64, then in FP32
    static constexpr size_t bytes = sizeof(float) * (size_t(kTabs) + size_t(G::GPC) * kGroup);
};

// ---- FP64 helpers (integer exponent arithmetic: GB300's FP64 pipe is the
// bound of the FP64 kernels)
// e with |x| in [2^(e-1), 2^e) (x normal); above 1023 for infinity and NaN.
__device__ __forceinline__ int exponent_of(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1022; }
// x 2^k, k clamped to the normal range.
__device__ __forceinline__ double scale2(double x, int k)
{
    return x * __hiloint2double((min(max(k, -1022), 1023) + 1023) << 20, 0);
}
// Conversions on the integer pipe (the conversion instructions run at the
// FP64 rate): exact for normal floats and zero; to float rounded to nearest,
// ties away, for values in its normal range.  Infinity and NaN become huge
// numbers, subnormal floats wrong small ones: both only mislead the
// preconditioner, whose iteration then fails and leaves the group to the
// direct solve.
__device__ __forceinline__ double wide(float x)
{
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    return __hiloint2double(int((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), int(b << 29));
}
__device__ __forceinline__ float narrow(double x)
{
    const unsigned hi = unsigned(__double2hiint(x)), lo = unsigned(__double2loint(x));
    const unsigned m = hi & 0x7fffffffu;
    if (m < 0x38100000u || m >= 0x47e00000u) return m < 0x38100000u ? 0.f : float(x);
    const unsigned v = ((m - 0x38000000u) << 3) + (lo >> 29) + ((lo >> 28) & 1u);
    return __uint_as_float((hi & 0x80000000u) | v);
}
// 1 / x by two Newton-Raphson steps from the hardware's approximation (four
// FP64 FMA), within one unit in the last place of the quotient; the division
// where the approximation's range ends.
__device__ __forceinline__ double rcp64(double x)
{
    const unsigned m = unsigned(__double2hiint(x)) & 0x7fffffffu;
    if (m < 0x20000000u || m > 0x5ff00000u) return 1.0 / x;
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

// Row tig of C^{-1} (creg, threads tig < 4N) from C's structure, the factors in FP64 (the mixed form).  C = w^-2 I +
// [[Gx (x) My, Cxy], [Cxy^T, Gy (x) Mx]] with Gx = [gx_s . gx_s'] (2 x 2), My =
// Wy Wy^T and Cxy of rank 4 (its (s, s') blocks are hvy_s' hvx_s^T).  The
// Kronecker blocks invert through the eigenvectors Q of Gx and Gy:
// (w^-2 I + Gx (x) My)^{-1} = sum_t q_t q_t^T (x) (w^-2 I + lambda_t My)^{-1},
// four N x N inverses; the coupling enters by block elimination and the
// Woodbury identity on the Schur complement, with 4 x 4 matrices
// P = A^T Cxx^{-1} A, Qm = B^T Cyy^{-1} B (Cxy = A B^T) and T = P^{-1} - Qm.
// The N x N and 4 x 4 inverses and the products that form P and Qm run in
// FP64; the entries are assembled from them in FP32.  Same result as the
// inverse of the dense C (checked in a NumPy model with these conventions).
// GB300 runs FP64 at 2 lanes per clock per SM, so a warp-wide FP64 instruction
// costs the same whatever its active lanes: the small FP64 steps spread their
// work over the lanes of warp 0, and reciprocals are four FMA (rcp64).
// Conversions run at the FP64 rate too and take the integer pipe instead:
// with them and a reciprocal from a conversion the mixed form took 18.0, 28.9
// and 78.1 ns per element-sample at N = 4, 8, 11, now 14.6, 24.2 and 64.0.
template <int N, int W, int TG, int NR, int RS>
__device__ __forceinline__ void factor64_2d(double *xd, int tig, int lane, int wig, int bar_id, const float *gt,
                                            const float *Mx, const float *My, const float *u4, float wi2,
                                            float (&creg)[4 * N])
{
    constexpr int F = 4 * N;
    auto sync = [&]() {
        if constexpr (W == 1) __syncwarp();
        else group_sync(bar_id, TG);
    };
    double *Ainv = xd;                 // [4][N][N]: (w^-2 I + lx_t My)^{-1}, t = 0, 1; then the y side
    double *piv64 = Ainv + 4 * N * N;  // [4][2][N] pivot rows of their Gauss-Jordan
    double *yz = piv64 + 8 * N;        // [8][N]: y_{t,tp} = Ainv_t hvy_tp, z_{t,tg} = Ainv_{2+t} hvx_tg
    double *sm64 = yz + 8 * N;         // Qx [2][2], lx [2], Qy [2][2], ly [2], then warp-0 scratch
    float *A32 = reinterpret_cast<float *>(sm64 + 88);  // [4][N][N] Ainv in FP32
    float *Z32 = A32 + 4 * N * N;                       // [4N][4]: rows of Cxx^{-1} A, Cyy^{-1} B
    float *s32 = Z32 + 16 * N;                          // Qx [4], Qy [4], Mxx [16], M1 [16], Ti [16]
    const float *hvx = u4, *hvy = u4 + 2 * RS;  // hvx[s RS + i] = (Wx gx_s)_i, hvy[s RS + j] = (Wy gy_s)_j
    double *w64 = sm64 + 12;  // warp-0 scratch: [6] Gram entries, then [16] dots, [3][16] 4 x 4 matrices
    if (wig == 0) {  // the 2 x 2 eigen-decompositions (a Jacobi rotation each)
        if (lane < 6) {  // lane 3 d + e: d = 0 x, 1 y; e = 0: g0.g0, 1: g0.g1, 2: g1.g1
            const int d = lane / 3, e = lane - 3 * d;
            const float *ga = gt + (2 * d + (e == 2)) * RS, *gb = gt + (2 * d + (e != 0)) * RS;
            double acc = 0.0;
#pragma unroll
            for (int m = 0; m < N; ++m) acc = fma(wide(ga[m]), wide(gb[m]), acc);
            w64[lane] = acc;
        }
        __syncwarp();
        if (lane < 2) {
            const int d = lane;
            const double g00 = w64[3 * d], g01 = w64[3 * d + 1], g11 = w64[3 * d + 2];
            double cs = 1.0, sn = 0.0, l0 = g00, l1 = g11;
            if (g01 != 0.0) {
                const double tau = (g11 - g00) * (0.5 * rcp64(g01));
                const double tn = (tau >= 0.0 ? 1.0 : -1.0) * rcp64(fabs(tau) + sqrt(fma(tau, tau, 1.0)));
                cs = rcp64(sqrt(fma(tn, tn, 1.0)));
                sn = tn * cs;
                l0 = fma(-tn, g01, g00);
                l1 = fma(tn, g01, g11);
            }
            double *q = sm64 + 6 * d;  // Q = [[cs, sn], [-sn, cs]]: column t the eigenvector of l_t
            q[0] = cs;
            q[1] = sn;
            q[2] = -sn;
            q[3] = cs;
            q[4] = l0;
            q[5] = l1;
            s32[4 * d + 0] = narrow(cs);
            s32[4 * d + 1] = narrow(sn);
            s32[4 * d + 2] = narrow(-sn);
            s32[4 * d + 3] = narrow(cs);
        }
    }
    sync();
    {  // the four N x N inverses, Gauss-Jordan in FP64, each matrix's rows in one warp
        constexpr bool kOneWarp = F <= 32;
        int mat = -1, r = 0;
        if constexpr (kOneWarp) {
            if (tig < F) mat = tig / N, r = tig % N;
        } else {
            if (wig < 2 && lane < 2 * N) mat = 2 * wig + lane / N, r = lane % N;
        }
        double arow[N];
        if (mat >= 0) {
            const double lam = sm64[(mat >> 1) * 6 + 4 + (mat & 1)];
            const float *M = (mat < 2 ? My : Mx) + r * NR;  // My for the x faces, Mx for the y faces
#pragma unroll
            for (int j = 0; j < N; ++j) arow[j] = j == r ? fma(lam, wide(M[j]), wide(wi2)) : lam * wide(M[j]);
        }
        if (kOneWarp ? wig == 0 : wig < 2) {  // uniform per warp
#pragma unroll
            for (int k = 0; k < N; ++k) {
                // the pivot row publishes itself unscaled; every row then takes
                // one FMA per entry (the pivot row from zero), so that the
                // warp's FP64 instructions are not split by the pivot's scaling
                double *pr = piv64 + ((mat < 0 ? 0 : mat) * 2 + (k & 1)) * N;
                if (mat >= 0 && r == k)
#pragma unroll
                    for (int j = 0; j < N; ++j) pr[j] = arow[j];
                __syncwarp();
                if (mat >= 0) {
                    const double pinv = rcp64(pr[k]);
                    const bool own = r == k;
                    const double coef = own ? pinv : -arow[k] * pinv;
#pragma unroll
                    for (int j = 0; j < N; ++j)
                        arow[j] = j == k ? coef : fma(coef, pr[j], own ? 0.0 : arow[j]);
                }
            }
        }
        if (mat >= 0)
#pragma unroll
            for (int j = 0; j < N; ++j) {
                Ainv[(mat * N + r) * N + j] = arow[j];
                A32[(mat * N + r) * N + j] = narrow(arow[j]);
            }
    }
    sync();
    for (int e2 = tig; e2 < 8 * N; e2 += TG) {  // y and z, FP64
        const int v = e2 / N, k = e2 - v * N;
        const int mat = v < 4 ? v >> 1 : 2 + ((v - 4) >> 1);
        const float *h = v < 4 ? hvy + (v & 1) * RS : hvx + (v & 1) * RS;
        double acc = 0.0;
#pragma unroll
        for (int k2 = 0; k2 < N; ++k2) acc = fma(Ainv[(mat * N + k) * N + k2], wide(h[k2]), acc);
        yz[e2] = acc;
    }
    sync();
    if (wig == 0) {  // P, Qm and the 4 x 4 algebra, FP64, one entry per lane
        double *dyz = w64 + 6;  // [16]: dy[t][a1][a2] = hvy_a1 . y_{t,a2} at 4t + 2a1 + a2, dz at 8 + ...
        double *Pm = dyz + 16;  // [16] P, then P^{-1}, then T^{-1}
        double *Qm = Pm + 16;   // [16]
        double *QT = Qm + 16;   // [16] Qm T^{-1}
        if (lane < 16) {
            const bool isz = lane >= 8;
            const int t = (lane >> 2) & 1, a1 = (lane >> 1) & 1, a2 = lane & 1;
            const float *h = isz ? hvx + a1 * RS : hvy + a1 * RS;
            const double *v = yz + ((isz ? 4 : 0) + 2 * t + a2) * N;
            double acc = 0.0;
#pragma unroll
            for (int k = 0; k < N; ++k) acc = fma(wide(h[k]), v[k], acc);
            dyz[lane] = acc;
        }
        __syncwarp();
        const int e = lane & 15, i4 = e >> 2, j4 = e & 3;
        {
            const double *Qx = sm64, *Qy = sm64 + 6;
            const int sg = i4 >> 1, sp = i4 & 1, tg = j4 >> 1, tp = j4 & 1;
            double v = 0.0;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const double qa = lane < 16 ? Qx[2 * sg + t] : Qy[2 * sp + t], qb = lane < 16 ? Qx[2 * tg + t] : Qy[2 * tp + t];
                const double dv = lane < 16 ? dyz[4 * t + 2 * sp + tp] : dyz[8 + 4 * t + 2 * sg + tg];
                v = fma(qa * qb, dv, v);
            }
            (lane < 16 ? Pm : Qm)[e] = v;
        }
        __syncwarp();
        auto inv4w = [&](double *A) {  // in place, one entry per lane (both half-warps alike)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double p = A[5 * k], aik = A[4 * i4 + k], akj = A[4 * k + j4], aij = A[e];
                __syncwarp();
                const double pinv = rcp64(p);
                const bool ri = i4 == k, cj = j4 == k;
                const double f = ri ? pinv : -aik * pinv;  // row k: pinv akj; others: aij - aik pinv akj
                const double v = cj ? f : fma(f, akj, ri ? 0.0 : aij);
                if (lane < 16) A[e] = v;
                __syncwarp();
            }
        };
        inv4w(Pm);
        if (lane < 16) Pm[e] -= Qm[e];  // T = P^{-1} - Qm
        __syncwarp();
        inv4w(Pm);                      // T^{-1}
        double qt = 0.0;
#pragma unroll
        for (int m = 0; m < 4; ++m) qt = fma(Qm[4 * i4 + m], Pm[4 * m + j4], qt);
        if (lane < 16) QT[e] = qt;
        __syncwarp();
        double mxx = Qm[e];
#pragma unroll
        for (int m = 0; m < 4; ++m) mxx = fma(QT[4 * i4 + m], Qm[4 * m + j4], mxx);
        if (lane < 16) {
            s32[8 + e] = narrow(mxx);                                // Mxx = Qm + Qm T^-1 Qm
            s32[24 + e] = narrow((i4 == j4 ? 1.0 : 0.0) + QT[e]);    // M1 = I + Qm T^-1
            s32[40 + e] = narrow(Pm[e]);                             // T^-1
        }
    }
    if (tig < F) {  // row tig of Cxx^{-1} A (x faces) or Cyy^{-1} B (y faces)
        const int f = tig, s = (f / N) & 1, k = f % N;
        const bool fx = f < 2 * N;
        const double *Qd = fx ? sm64 : sm64 + 6;
#pragma unroll
        for (int a1 = 0; a1 < 2; ++a1)
#pragma unroll
            for (int a2 = 0; a2 < 2; ++a2) {
                double acc = 0.0;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const double q = Qd[2 * s + t] * Qd[2 * (fx ? a1 : a2) + t];
                    acc = fma(q, yz[fx ? (2 * t + a2) * N + k : (4 + 2 * t + a1) * N + k], acc);
                }
                Z32[4 * f + 2 * a1 + a2] = narrow(acc);
            }
    }
    sync();
    if (tig < F) {  // row tig of C^{-1}, assembled in FP32
        const int s = (tig / N) & 1, k = tig % N;
        const bool fx = tig < 2 * N;
        const float4 zr4 = *reinterpret_cast<const float4 *>(Z32 + 4 * tig);
        const float zr[4] = {zr4.x, zr4.y, zr4.z, zr4.w};
        const float *Mxx = s32 + 8, *M1 = s32 + 24, *Tinv = s32 + 40;
        float rr[4], rp[4];  // the row's coefficients for its own block and the other
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float a1 = 0.f, a2 = 0.f;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                a1 = fmaf(zr[m], fx ? Mxx[4 * m + j] : Tinv[4 * m + j], a1);
                a2 = fmaf(zr[m], fx ? M1[4 * m + j] : M1[4 * j + m], a2);
            }
            rr[j] = a1;
            rp[j] = -a2;
        }
        const float *Q32 = fx ? s32 : s32 + 4;
        float cq[2][2];  // Q[s][t] Q[s2][t]
#pragma unroll
        for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
            for (int t = 0; t < 2; ++t) cq[s2][t] = Q32[2 * s + t] * Q32[2 * s2 + t];
        const float *Ab = A32 + (fx ? 0 : 2) * N * N + k * N;  // row k of the block's inverses t = 0, 1
#pragma unroll
        for (int g2 = 0; g2 < F; ++g2) {
            const int s2 = (g2 / N) & 1, k2 = g2 % N;
            const bool same = fx == (g2 < 2 * N);
            const float4 z2 = *reinterpret_cast<const float4 *>(Z32 + 4 * g2);
            float v = (same ? rr[0] : rp[0]) * z2.x;
            v = fmaf(same ? rr[1] : rp[1], z2.y, v);
            v = fmaf(same ? rr[2] : rp[2], z2.z, v);
            v = fmaf(same ? rr[3] : rp[3], z2.w, v);
            if (same) {
                v = fmaf(cq[s2][0], Ab[k2], v);
                v = fmaf(cq[s2][1], Ab[N * N + k2], v);
            }
            creg[g2] = v;
        }
    }
}

// CTAs per SM the register budget is sized for.
template <int N, typename R, int PHASE>
constexpr int fast_ctas()
{
    constexpr int warps = FGeo<N, R>::kBlock / 32;
    return FGeo<N, R>::kF64 ? (N <= 8 ? 16 / warps : 12 / warps) : 16 / warps;
}

// Gauss-node basis at a particle, h_i(x) = lambda_i prod_{m != i} (x - zeta_m),
// x - zeta_m = Z[m] + d (node difference plus displacement).
template <int N, typename T>
__device__ __forceinline__ void particle_basis(const T *Z, const T *lam, T d, T (&h)[N])
{
    T f[N];
#pragma unroll
    for (int m = 0; m < N; ++m) f[m] = Z[m] + d;
    T pre = T(1);
#pragma unroll
    for (int m = 0; m < N; ++m) {
        h[m] = pre;
        pre *= f[m];
    }
    T suf = T(1);
#pragma unroll
    for (int m = N - 1; m >= 0; --m) {
        h[m] *= suf * lam[m];
        suf *= f[m];
    }
}

// sum_m w[m] v[m] of two rows of N floats in shared memory (16-byte aligned).
template <int N>
__device__ __forceinline__ void load_rowf(const float *p, float (&v)[N])
{
#pragma unroll
    for (int m = 0; m < N; m += 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p + m);
        v[m] = q.x;
        if (m + 1 < N) v[m + 1] = q.y;
        if (m + 2 < N) v[m + 2] = q.z;
        if (m + 3 < N) v[m + 3] = q.w;
    }
}
template <int N>
__device__ __forceinline__ float dotf(const float (&w)[N], const float (&v)[N])
{
    float t = 0.f;
#pragma unroll
    for (int m = 0; m < N; ++m) t = fmaf(w[m], v[m], t);
    return t;
}

// (V x) at a particle: sum_j hy[j] sum_i hx[i] x[j][i], x in rows of RS.
template <int N, int RS, typename T>
__device__ __forceinline__ T apply_v(const T *x, const T (&hx)[N], const T (&hy)[N])
{
    T s = T(0);
#pragma unroll
    for (int j = 0; j < N; ++j) {
        T t = T(0);
        if constexpr (sizeof(T) == 4) {
            float v[N];
            load_rowf<N>(x + j * RS, v);
            t = dotf<N>(hx, v);
        } else {
#pragma unroll
            for (int i = 0; i < N; i += 2) {  // RS is a multiple of 4: rows are 16-byte aligned
                const double2 v = *reinterpret_cast<const double2 *>(x + j * RS + i);
                t = fma(hx[i], v.x, t);
                if (i + 1 < N) t = fma(hx[i + 1], v.y, t);
            }
        }
        s = fma(hy[j], t, s);
    }
    return s;
}

template <int N, typename R, int PHASE, bool BATCH, int NCOMP, bool FAC64>
__device__ __forceinline__ void sl2d_fast_group(const Step2DArgs &a0, const Step2DArgs *__restrict__ args,
                                                const long long *__restrict__ prefix, int ninst, int t)
{
    using G = FGeo<N, R>;
    using S = FSmem<N, R, PHASE, FAC64>;
    constexpr int n = G::n, W = G::W, TG = G::TG, La = G::La, NS = G::NS, F = G::F, RS = G::RS, NR = G::NR;
    constexpr bool kPair = !G::kF64;
    constexpr bool kSameI = La % N == 0;  // a thread's nodes share their column
    using State = typename std::conditional<kPair, float2, double>::type;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    const R *sZ = reinterpret_cast<const R *>(smem_raw);  // the tables in the state's precision
    const R *slam = sZ + N * N, *sh0 = slam + N, *sh1 = sh0 + N;
    float *ftab = reinterpret_cast<float *>(smem_raw) + (G::kF64 ? 2 * G::kTab : 0);
    const float *fZ = ftab, *flam = fZ + N * N, *fh0 = flam + N, *fh1 = fh0 + N, *fX0 = fh1 + N, *fX1 = fX0 + N;
    const int grp = threadIdx.x / TG, tig = threadIdx.x - grp * TG;
    const int lane = threadIdx.x & 31, wig = tig >> 5, bar_id = 1 + grp;
    float *gb = reinterpret_cast<float *>(smem_raw) + S::kTabs + grp * S::kGroup;
    double *x64 = reinterpret_cast<double *>(gb + (PHASE == 1 ? G::oEnd1 : G::oEnd2));
    float *Wx = gb + G::oW, *WxT = Wx + G::kW, *Wy = WxT + G::kW, *WyT = Wy + G::kW;
    float *gt = gb + G::oG;    // [4][RS]
    float *db = gb + G::oDb;   // [2][RS]
    unsigned *red = reinterpret_cast<unsigned *>(gb + G::oRed);
    float *fA = gb + G::oA, *fB = gb + G::oB, *vec = gb + G::oVec, *res = gb + G::oRes;
    (void)sh0, (void)sh1, (void)x64;

    auto sync = [&]() {
        if constexpr (W == 1) __syncwarp();
        else group_sync(bar_id, TG);
    };

    const long long ggid = (BATCH ? 0 : a0.g0) + (long long)blockIdx.x * G::GPC + grp;
    int inst = 0;
    if constexpr (BATCH) {
        if (ggid >= prefix[ninst]) return;  // the whole group
        int lo = 0, hi = ninst - 1;         // last instance with prefix[i] <= ggid
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (prefix[mid] <= ggid) lo = mid;
            else hi = mid - 1;
        }
        inst = lo;
    } else {
        if (ggid >= a0.g1) return;
    }
    const Step2DArgs &a = BATCH ? args[inst] : a0;
    const long long gid = BATCH ? ggid - prefix[inst] : ggid;
    const int Kx = a.Kx, Ky = a.Ky, E = Kx * Ky;
    // 32-bit division where it holds the group
    const int s = gid < 0x80000000ll ? int(unsigned(gid) / unsigned(E)) : int(gid / E);
    const int e = int(gid - (long long)s * E);
    const int kx = e % Kx, ky = e / Kx;

    // ---- the thread's nodes (particles): state, displacement, basis
    int ci[NS], ip[NS], jp[NS];
    bool on[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int c = tig + k * La;
        on[k] = tig < La && c < n;
        ci[k] = on[k] ? c : 0;
        ip[k] = ci[k] % N;
        jp[k] = ci[k] / N;
    }
    State *Qg = reinterpret_cast<State *>(a.Q);
    R ch[NCOMP], cl[NCOMP], ph[NCOMP][NS];
    long long qoff[NCOMP];
    R hx[NS][N], hy[NS][N];
    float dxf[NS], dyf[NS];
    {
        const long long V = (long long)E * n;
        const R dWx = R(a.dW[((long long)t * a.M + s) * 2 + 0]);
        const R dWy = R(a.dW[((long long)t * a.M + s) * 2 + 1]);
        const R *cf = static_cast<const R *>(a.coef);
#pragma unroll
        for (int cc = 0; cc < NCOMP; ++cc) {
            qoff[cc] = (((long long)s * NCOMP + cc) * E + e) * n;
            const State cv = Qg[qoff[cc] + n / 2];
            if constexpr (kPair) {
                ch[cc] = cv.x;
                cl[cc] = cv.y;
            } else {
                ch[cc] = cv;
                cl[cc] = R(0);
            }
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const long long pe = (long long)e * n + ci[k];
            // displacement 4 (u dt + b dW) / h as one explicit FMA of the step's
            // coefficients (the same rounding in the batched and single kernels)
            const R dx = fma(cf[2 * V + pe], dWx, cf[pe]);
            const R dy = fma(cf[3 * V + pe], dWy, cf[V + pe]);
            const R gam = cf[4 * V + pe];
#pragma unroll
            for (int cc = 0; cc < NCOMP; ++cc) {
                const State qv = Qg[qoff[cc] + ci[k]];
                if constexpr (kPair) {
                    const float dq = (qv.x - ch[cc]) + (qv.y - cl[cc]);
                    ph[cc][k] = dq - __fmul_rn(gam, qv.x);
                } else {
                    ph[cc][k] = (qv - ch[cc]) - __dmul_rn(gam, qv);
                }
            }
            particle_basis<N, R>(sZ + ip[k] * N, slam, dx, hx[k]);
            particle_basis<N, R>(sZ + jp[k] * N, slam, dy, hy[k]);
            dxf[k] = float(dx);
            dyf[k] = float(dy);
        }
    }
    // FP32 basis of the FP32 iteration (FP64: formed in FP32 by itself; conversions
    // of 2N values per particle would run at the FP64 rate)
    float hxf_[G::kF64 ? NS : 1][N], hyf_[G::kF64 ? NS : 1][N];
    if constexpr (G::kF64) {
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            particle_basis<N, float>(fZ + ip[k] * N, flam, dxf[k], hxf_[k]);
            particle_basis<N, float>(fZ + jp[k] * N, flam, dyf[k], hyf_[k]);
        }
    }
    auto hxf = [&](int k) -> const float(&)[N] { if constexpr (G::kF64) return hxf_[k]; else return hx[k]; };
    auto hyf = [&](int k) -> const float(&)[N] { if constexpr (G::kF64) return hyf_[k]; else return hy[k]; };

    using FaceT = typename std::conditional<kPair, float2, double>::type;
    FaceT *faces = reinterpret_cast<FaceT *>(a.faces);

    // ---- upwinded face values g (Eq. bnd_update) of face point tig, phase 2
    R gf[NCOMP];
#pragma unroll
    for (int cc = 0; cc < NCOMP; ++cc) gf[cc] = R(0);
    if constexpr (PHASE == 2) {
        if (tig < F) {
            const int side = tig / N, f = tig - side * N;
            const bool xface = side < 2, high = side & 1;
            int e_face = e;  // element whose low face is this interface
            if (side == 1) e_face = ky * Kx + (kx + 1 == Kx ? 0 : kx + 1);
            if (side == 3) e_face = (ky + 1 == Ky ? 0 : ky + 1) * Kx + kx;
            // a face on a Dirichlet domain boundary: the ghost value takes the
            // place of the missing neighbour (low side at x = lo / y = lo, high
            // side at x = hi / y = hi); the faces x = hi, y = hi have their own
            // coefficients
            const bool dir = !a.periodic;
            const bool ghost_low = dir && ((side == 0 && kx == 0) || (side == 2 && ky == 0));
            const bool ghost_high = dir && ((side == 1 && kx == Kx - 1) || (side == 3 && ky == Ky - 1));
            const double dW = a.dW[((long long)t * a.M + s) * 2 + (xface ? 0 : 1)];
            R af, bf;
            if (ghost_high) {
                const long long hidx = side == 1 ? (long long)ky * N + f : (long long)Ky * N + (long long)kx * N + f;
                af = R(a.faceUhi[hidx] * a.dt);
                bf = R(a.faceBhi[hidx]);
            } else {
                const R *fc = static_cast<const R *>(a.coef) + 5ll * E * n;  // [2][2 E N]: u dt, sqrt(2 D)
                const long long fidx = (long long)(xface ? 0 : 1) * E * N + (long long)e_face * N + f;
                af = fc[fidx];
                bf = fc[2ll * E * N + fidx];
            }
            bool from_low;  // take the value from the element on the low side
            if constexpr (kPair) from_low = fmaf(bf, float(dW), af) > 0.f;
            else from_low = __dadd_rn(af, __dmul_rn(bf, dW)) > 0.0;
            int e_low = e, e_high = high ? e_face : e;
            if (side == 0) e_low = ky * Kx + (kx == 0 ? Kx - 1 : kx - 1);
            if (side == 2) e_low = (ky == 0 ? Ky - 1 : ky - 1) * Kx + kx;
#pragma unroll
            for (int cc = 0; cc < NCOMP; ++cc) {  // (two fields: periodic meshes only, no ghosts)
                const long long fb = ((long long)s * NCOMP + cc) * E;
                FaceT gv;
                if (from_low && ghost_low)  // left [Ky][N] or bottom [Kx][N] boundary values
                    gv = ghost_face2d<FaceT>(a.ghost[t * a.ghost_w + (side == 0 ? (long long)ky * N + f
                                                                            : 2LL * Ky * N + (long long)kx * N + f)]);
                else if (!from_low && ghost_high)  // right [Ky][N] or top [Kx][N]
                    gv = ghost_face2d<FaceT>(a.ghost[t * a.ghost_w + (side == 1 ? (long long)Ky * N + (long long)ky * N + f
                                                                            : 2LL * Ky * N + (long long)Kx * N +
                                                                                  (long long)kx * N + f)]);
                else
                    gv = from_low ? faces[(fb + e_low) * F + (xface ? N : 3 * N) + f]
                                  : faces[(fb + e_high) * F + (xface ? 0 : 2 * N) + f];
                if constexpr (kPair) gf[cc] = (gv.x - ch[cc]) + (gv.y - cl[cc]);
                else gf[cc] = gv - ch[cc];
            }
        }
    }

    // ---- 1D factors
#pragma unroll
    for (int k = 0; k < NS; ++k)
        if (on[k]) {
            fA[jp[k] * NR + ip[k]] = dxf[k];
            fB[jp[k] * NR + ip[k]] = dyf[k];
            if constexpr (PHASE == 2) {
                float *hxT = gb + G::oH, *hyT = hxT + N * G::NTP;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    hxT[i * G::NTP + ci[k]] = hxf(k)[i];
                    hyT[i * G::NTP + ci[k]] = hyf(k)[i];
                }
            }
        }
    sync();
    if (tig < 2 * N) {  // mean x displacement of particle column, mean y displacement of row
        const bool y = tig >= N;
        const int i = y ? tig - N : tig;
        float sum = 0.f;
#pragma unroll
        for (int m = 0; m < N; ++m) sum += y ? fB[i * NR + m] : fA[m * NR + i];
        db[(y ? RS : 0) + i] = sum / float(N);
    }
    sync();
    // every difference is a node difference plus a displacement difference; the
    // quotients within a few ulp (pdiv): they set the convergence only
#pragma unroll
    for (int k = 0; k < NS; ++k)
        if (on[k]) {
            const int i = jp[k], a2 = ip[k];  // entry [i][a2]
            float nx = 1.f, dx_ = 1.f, ny = 1.f, dy_ = 1.f;
            const float bx = db[a2], by = db[RS + a2];
#pragma unroll
            for (int m = 0; m < N; ++m) {
                const float mx = db[m], my = db[RS + m], zi = fZ[i * N + m], za = fZ[a2 * N + m];
                const bool skip = m == a2;
                nx *= skip ? 1.f : zi - mx;
                dx_ *= skip ? 1.f : za + (bx - mx);
                ny *= skip ? 1.f : zi - my;
                dy_ *= skip ? 1.f : za + (by - my);
            }
            const float wx = pdiv(nx, dx_), wy = pdiv(ny, dy_);
            Wx[i * NR + a2] = wx;
            WxT[a2 * NR + i] = wx;
            Wy[i * NR + a2] = wy;
            WyT[a2 * NR + i] = wy;
        }
    if (PHASE == 2 && tig < F) {  // the tilde basis at the faces
        const int s2 = tig / N, a2 = tig - s2 * N;
        const float *d1 = db + (s2 < 2 ? 0 : RS), *X = (s2 & 1) ? fX1 : fX0;
        const float b1 = d1[a2];
        float num = 1.f, den = 1.f;
#pragma unroll
        for (int m = 0; m < N; ++m) {
            const bool skip = m == a2;
            num *= skip ? 1.f : X[m] - d1[m];
            den *= skip ? 1.f : fZ[a2 * N + m] + (b1 - d1[m]);
        }
        gt[s2 * RS + a2] = pdiv(num, den);
    }
    sync();

    // group maximum of a non-negative float per thread (NaN compares above all)
    auto warp_max = [&](float v) { return __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(v))); };
    int rbuf = 0;
    // publishes the group's maxima of |d| and |x|; `maxima` reads them after a sync
    unsigned kd1 = 0, kx1 = 0;
    auto publish = [&](float d, float x) {
        rbuf ^= 1;
        kd1 = warp_max(d);
        kx1 = warp_max(x);
        if constexpr (W > 1) {
            if (lane == 0) {
                red[rbuf * 2 * W + 2 * wig] = kd1;
                red[rbuf * 2 * W + 2 * wig + 1] = kx1;
            }
        }
    };
    auto maxima = [&](float &md, float &mx) {
        unsigned d = kd1, x = kx1;
        if constexpr (W > 1) {
            d = x = 0u;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                d = max(d, red[rbuf * 2 * W + 2 * w]);
                x = max(x, red[rbuf * 2 * W + 2 * w + 1]);
            }
        }
        md = __uint_as_float(d);
        mx = __uint_as_float(x);
    };

    // group maximum of a binary exponent (-5000: none)
    auto group_top = [&](int top) {
        unsigned m = __reduce_max_sync(0xffffffffu, unsigned(top + 5000));
        if constexpr (W > 1) {
            rbuf ^= 1;
            if (lane == 0) red[rbuf * 2 * W + 2 * wig] = m;
            sync();
            m = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) m = max(m, red[rbuf * 2 * W + 2 * w]);
        }
        return int(m) - 5000;
    };

    // conditioning of the tensor factors, L = ||Wx||_inf ||Wy||_inf, against the
    // largest tried: where what the iteration accepts within its corrections is as
    // exact as its residual; above, the direct solve.  Phase 2 (which squares the
    // conditioning) stops converging first, the mixed form's C^{-1}, rounded with
    // its null directions (see below), before the others.  One step on 64 x 64
    // elements of N = 8 at half the node-gap step with face jumps of 1e-3, off from
    // FP64 relative to a group's own maximum: FP32 2.3e-9 rms (at most 1.7e-8) at L
    // 64 to 160 and 6.3e-9 (6.7e-8) at 160 to 300; mixed 5.6e-7 (1.1e-5) at 128 to
    // 160; the direct solve 2.5e-10.  A step of 64 samples takes 2.62 ms with the
    // FP32 limit at 300, 3.25 at 160.  FP64, the whole node-gap step against the
    // oracle: at most 3e-14 up to L = 512, 1.6e-13 at 512 to 1024 (the direct solve
    // 3.4e-14).  At N <= 4, where a direct solve is cheap, FP64's ill-conditioned go
    // there at once.
    constexpr float kCond = kPair ? (PHASE == 1 ? 512.0f : FAC64 ? 160.0f : 300.0f)
                                  : N <= 4 ? 100.0f : PHASE == 1 ? 4096.0f : 512.0f;
    constexpr int kIters = 8;
    constexpr int kOuter = 24;  // FP64: corrections (ill-conditioned groups gain a digit or less in each)
    constexpr float kShrink = 0.45f;  // and the slowest progress at which that many suffice
    bool done = false;
    float cond = 0.f;
    {
        float sx = 0.f, sy = 0.f;
        if (tig < N) {
#pragma unroll
            for (int m = 0; m < N; ++m) {
                sx += fabsf(Wx[tig * NR + m]);
                sy += fabsf(Wy[tig * NR + m]);
            }
        }
        publish(sx, sy);
        if constexpr (W > 1) sync();
        float mx, my;
        maxima(mx, my);
        cond = mx * my;
        done = cond <= kCond;
    }

    if (done) {
        // Stopping of the FP32 iteration: the last correction d below 1e-6 of
        // max|x| + |c|.  The remaining error is d rho / (1 - rho) at a contraction
        // rate rho.  rho is not estimated from the corrections: the first ones are
        // smooth, and their quotient promises a contraction that the worst-
        // conditioned directions do not have.  Stopping on d^2 / d_before <= 1e-7 as
        // well left one step of the groups of L 16 to 64 (see kCond) off by 1.6e-8
        // rms instead of 2.4e-9, and the FP32 mean after 500 steps 1.8e-5 from FP64
        // instead of 5.6e-6.
        auto settled = [&](float d, float scale) { return d < INFINITY && d <= 1e-6f * scale; };
        // FP64: an FP32 correction is iterated to 1e-7 of itself (1e-8 estimated;
        // what that leaves, the next residual shows).  The outer iteration stops
        // when the last correction is below 1e-13 of max|x| + |c|; corrections
        // shrink by kShrink or more, so that the remaining error is below it too.
        // No estimate from two corrections here either: the directions that FP32
        // resolves shrink by five digits a correction and hide the slow ones.
        // With one (d^2 / d_before <= 1e-14), a step at the node-gap bound left
        // groups of L 64 to 512 up to 1.6e-10 (N = 8) and 1e-8 (N = 10) from the
        // solution.  Below that, where the third correction is rounding, both rules
        // take three.
        auto inner_settled = [&](float d, float before, float scale) {
            return d < INFINITY && (d <= 1e-7f * scale || (before > 0.f && d < 0.5f * before && d * (d / before) <= 1e-8f * scale));
        };
        auto refined = [&](float d, float scale) { return d < INFINITY && d <= 1e-13f * scale; };

        if constexpr (PHASE == 1) {
            float wxr[NS][N], wyr[NS][N];  // the rows of Wx and Wy this thread applies
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (k == 0 || !kSameI) load_rowf<N>(Wx + ip[k] * NR, wxr[k]);
                load_rowf<N>(Wy + jp[k] * NR, wyr[k]);
            }
            // x (at the thread's nodes) solving V x = rhs (at its particles); the
            // iterate stays in vec.  scale0: what the stopping test adds to max|x|.
            auto solve = [&](const float (&rhs)[NS], float (&x)[NS], const float scale0, float &mx) -> bool {
                float r[NS], before = 0.f;
#pragma unroll
                for (int k = 0; k < NS; ++k) {
                    x[k] = 0.f;
                    r[k] = rhs[k];
                }
                for (int it = 0; it < kIters; ++it) {
#pragma unroll
                    for (int k = 0; k < NS; ++k)
                        if (on[k]) fA[jp[k] * RS + ip[k]] = r[k];
                    sync();
                    // V0^{-1} r: [(b, i)] = sum_a Wx[i][a] r[(b, a)] (stored at [i][b]), then sum_b Wy[j][b] [(b, i)]
#pragma unroll
                    for (int k = 0; k < NS; ++k)
                        if (on[k]) {
                            float v[N];
                            load_rowf<N>(fA + jp[k] * RS, v);
                            fB[ip[k] * NR + jp[k]] = dotf<N>(wxr[kSameI ? 0 : k], v);
                        }
                    sync();
                    float dm = 0.f, xm = 0.f;
                    {
                        float v[N];
#pragma unroll
                        for (int k = 0; k < NS; ++k) {
                            if (k == 0 || !kSameI) load_rowf<N>(fB + ip[k] * NR, v);
                            const float d = dotf<N>(wyr[k], v);
                            if (on[k]) {
                                x[k] += d;
                                vec[jp[k] * RS + ip[k]] = x[k];
                                dm = fmaxf(dm, fabsf(d));
                                xm = fmaxf(xm, fabsf(x[k]));
                                if (!(fabsf(d) < INFINITY)) dm = INFINITY;  // NaN too: never settles
                            }
                        }
                    }
                    publish(dm, xm);
                    sync();
                    float md;
                    maxima(md, mx);
                    if (kPair ? settled(md, mx + scale0) : inner_settled(md, before, mx)) return true;
                    // (FP64: a correction that stopped shrinking is left to the next residual)
                    if (!kPair && it > 0 && !(md < 0.5f * before)) return md < INFINITY;
                    before = md;
                    if (it + 1 < kIters)
#pragma unroll
                        for (int k = 0; k < NS; ++k) r[k] = rhs[k] - apply_v<N, RS, float>(vec, hxf(k), hyf(k));
                }
                return !kPair;
            };
            for (int cc = 0; cc < NCOMP && done; ++cc) {
                R xr[NS];
                if constexpr (kPair) {
                    float mx;
                    done = solve(ph[cc], xr, fabsf(ch[cc]), mx);
                } else {
                    // FP64 residual, FP32 corrections
                    double rd[NS];
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        xr[k] = 0.0;
                        rd[k] = ph[cc][k];
                    }
                    float before = 0.f;
                    int e0 = 0;
                    done = false;
                    for (int o = 0; o < kOuter; ++o) {
                        // scaled by a power of two: max |r| in [1/2, 1)
                        int top = -5000;
#pragma unroll
                        for (int k = 0; k < NS; ++k)
                            if (on[k] && rd[k] != 0.0) top = max(top, exponent_of(rd[k]));
                        top = group_top(top);
                        if (top == -5000) {  // zero residual
                            done = true;
                            break;
                        }
                        if (top > 1023) break;  // infinity or NaN
                        if (o == 0) e0 = top;
                        float rf[NS], xf[NS];
#pragma unroll
                        for (int k = 0; k < NS; ++k) rf[k] = float(scale2(rd[k], -top));
                        float mx;
                        if (!solve(rf, xf, 0.f, mx)) break;
                        float xm = 0.f;
#pragma unroll
                        for (int k = 0; k < NS; ++k) {
                            xr[k] += scale2(double(xf[k]), top);
                            if (on[k]) xm = fmaxf(xm, fabsf(float(scale2(xr[k], -e0))));
                        }
                        publish(0.f, xm);
                        if constexpr (W > 1) sync();
                        float mz, ms;
                        maxima(mz, ms);
                        const float d = ldexpf(mx, max(top - e0, -140));
                        const float scale = ms + float(scale2(fabs(ch[cc]), -e0));
                        if (refined(d, scale)) {
                            done = true;
                            break;
                        }
                        if (o > 0 && !(d < kShrink * before)) break;  // not converging
                        before = d;
#pragma unroll
                        for (int k = 0; k < NS; ++k)
                            if (on[k]) x64[jp[k] * RS + ip[k]] = xr[k];
                        sync();
#pragma unroll
                        for (int k = 0; k < NS; ++k) rd[k] = ph[cc][k] - apply_v<N, RS, double>(x64, hx[k], hy[k]);
                    }
                }
                if (!done) break;
                // phase 2 starts from it; the face values of the interpolant
#pragma unroll
                for (int k = 0; k < NS; ++k)
                    if (on[k]) {
                        static_cast<R *>(a.alpha)[qoff[cc] + ci[k]] = xr[k];
                        if constexpr (G::kF64) x64[jp[k] * RS + ip[k]] = xr[k];
                    }
                if constexpr (G::kF64) sync();
                if (tig < F) {
                    const int side = tig / N, f = tig - side * N;
                    const R *xv;
                    if constexpr (G::kF64) xv = x64;
                    else xv = vec;
                    const R *hb = (side & 1) ? sh1 : sh0;
                    R v = R(0);
#pragma unroll
                    for (int m = 0; m < N; ++m) v = fma(hb[m], side < 2 ? xv[f * RS + m] : xv[m * RS + f], v);
                    FaceT out;
                    if constexpr (kPair) {
                        two_sum2d(ch[cc], v, out.x, out.y);
                        out.y += cl[cc];
                    } else {
                        out = ch[cc] + v;
                    }
                    faces[(((long long)s * NCOMP + cc) * E + e) * F + tig] = out;
                }
                if (cc + 1 < NCOMP) sync();  // vec is read before the next field writes it
            }
        } else {
            float *Mx = gb + G::oM, *My = Mx + G::kW;
            float *u4 = gb + G::oU, *mu4 = u4 + 4 * RS, *mm4 = mu4 + 4 * RS, *uu4 = mm4 + 4 * RS;
            const int fseg = tig / N * RS, fk = tig % N;  // face point tig: its side's row, its place there
            const float *hxT = gb + G::oH, *hyT = hxT + N * G::NTP;
            const float wb = float(a.w), wi2 = 1.f / (wb * wb);
            // products for C: Mx = Wx Wx^T, My = Wy Wy^T (kept for the iteration), and
            // hvx[s][i] = sum_a Wx[i][a] gx_s[a] at u4[s RS + i], hvy[s][j] = sum_b Wy[j][b] gy_s[b] at u4[(2 + s) RS + j]
#pragma unroll
            for (int k = 0; k < NS; ++k)
                if (on[k]) {
                    float p[N], q[N];
                    load_rowf<N>(Wx + jp[k] * NR, p);
                    load_rowf<N>(Wx + ip[k] * NR, q);
                    Mx[jp[k] * NR + ip[k]] = dotf<N>(p, q);
                    load_rowf<N>(Wy + jp[k] * NR, p);
                    load_rowf<N>(Wy + ip[k] * NR, q);
                    My[jp[k] * NR + ip[k]] = dotf<N>(p, q);
                }
            if (tig < F) {
                const int s2 = tig / N, k = tig - s2 * N;
                float p[N], q[N];
                load_rowf<N>((s2 < 2 ? Wx : Wy) + k * NR, p);
                load_rowf<N>(gt + s2 * RS, q);
                u4[fseg + fk] = dotf<N>(p, q);
            }
            sync();
            float creg[F];  // thread tig < 4N: row tig of C, then of C^{-1}
            if constexpr (!FAC64) {
                // C's rows are held by a thread each, assembled from the 1D products
                // and inverted in place (symmetric positive definite, eigenvalues >= w^-2).
                // E0 E0^T has four null directions, one per corner: the corner's value
                // along its x face is that along its y face, whatever the field.  There
                // C is w^-2 alone, and an FP32 inverse of it as it stands loses digits in
                // every direction.  u = E0 t has no part in them and E0^T takes none back,
                // so that any multiple of them may be added to C: 4 L, the size of
                // E0 E0^T (a model converged as well with the mean of its diagonal, less
                // well with a tenth of it).  With it FP32 at L 128 to 160 is off by 2.2e-9
                // rms where it was by 3.6e-7 (see kCond).  Groups left to the direct solve
                // at N = 8, a tenth of the node-gap step, without and with it: w = 10 FP64
                // 20 % and none, FP32 16 % and 0.4 %; w = 30 97 % and none, 84 % and 2 %
                // (FP64 867 and 101 ns per element-sample).
                const float kap = 4.f * cond;
                const bool fx = tig < 2 * N;
                const int s2 = (tig / N) & 1;
#pragma unroll
                for (int j = 0; j < F; ++j) creg[j] = 0.f;
                if (tig < F) {
                    float g[N], gv[N], gg0, gg1;
                    load_rowf<N>(gt + fseg, g);
                    load_rowf<N>(gt + (fx ? 0 : 2) * RS, gv);
                    gg0 = dotf<N>(g, gv);
                    load_rowf<N>(gt + (fx ? 1 : 3) * RS, gv);
                    gg1 = dotf<N>(g, gv);
                    float mw[N], h0[N];  // the row of M along this face; this side's hv
                    load_rowf<N>((fx ? My : Mx) + fk * NR, mw);
                    load_rowf<N>(u4 + (fx ? s2 : 2 + s2) * RS, h0);
                    const float a0 = u4[(fx ? 2 : 0) * RS + fk], a1 = u4[(fx ? 3 : 1) * RS + fk];
                    const float t0 = kap * fh0[fk], t1 = kap * fh1[fk];  // corner directions: entry fk of this face
                    const float *hs = s2 ? fh1 : fh0;
#pragma unroll
                    for (int k2 = 0; k2 < N; ++k2) {
                        float d0 = gg0 * mw[k2], d1 = gg1 * mw[k2];  // sides 0, 1 of the same direction
                        const float v = fmaf(t0, fh0[k2], t1 * fh1[k2]);
                        d0 += s2 ? 0.f : v;
                        d1 += s2 ? v : 0.f;
                        const float c0 = fmaf(-t0, hs[k2], a0 * h0[k2]), c1 = fmaf(-t1, hs[k2], a1 * h0[k2]);  // of the other
                        creg[k2] = fx ? d0 : c0;
                        creg[N + k2] = fx ? d1 : c1;
                        creg[2 * N + k2] = fx ? c0 : d0;
                        creg[3 * N + k2] = fx ? c1 : d1;
                    }
#pragma unroll
                    for (int j = 0; j < F; ++j) creg[j] += j == tig ? wi2 : 0.f;
                }
                // Block Gauss-Jordan inversion in place with 4 x 4 pivot blocks (every
                // pivot block of an SPD matrix is SPD: no pivoting).  Step K: the pivot
                // rows publish themselves; after one barrier every thread inverts the
                // pivot block P in registers and forms the coefficients w: pivot row t
                // takes row t of P^{-1}, any other row w = -C[r][K] P^{-1}; then
                // C[r][j] <- C[r][j] + sum_m w_m C[K_m][j] outside the block (the pivot
                // rows start from 0 instead of C[r][j]) and C[r][K] <- w.  The columns
                // are rotated by a block in every step, so that the pivot block is
                // always the first and one loop body serves all steps: unrolled, the
                // steps overran the instruction cache (3.3 of 8.2 warps per issue
                // waited for instructions at N = 8).
                constexpr int CB = G::kCB, CR = G::CR;
                if (!G::kRowsOneWarp || wig == 0) {  // uniform per warp; above one warp, every thread
                    float *pb = fA;
#pragma unroll 1
                    for (int K = 0; K < F; K += CB) {
                        const int t0 = tig - K;
                        const bool pivot = t0 >= 0 && t0 < CB;
                        if (pivot)
#pragma unroll
                            for (int j = 0; j < F; j += 4)
                                *reinterpret_cast<float4 *>(pb + t0 * CR + j) =
                                    make_float4(creg[j], creg[j + 1], creg[j + 2], creg[j + 3]);
                        if constexpr (G::kRowsOneWarp) __syncwarp();
                        else group_sync(bar_id, TG);
                        if (tig < F) {
                            float Pm[CB][CB];  // the pivot block, then its inverse
#pragma unroll
                            for (int t2 = 0; t2 < CB; ++t2) {
                                const float4 q = *reinterpret_cast<const float4 *>(pb + t2 * CR);
                                Pm[t2][0] = q.x, Pm[t2][1] = q.y, Pm[t2][2] = q.z, Pm[t2][3] = q.w;
                            }
#pragma unroll
                            for (int p = 0; p < CB; ++p) {
                                const float d = pdiv(1.f, Pm[p][p]);
#pragma unroll
                                for (int m = 0; m < CB; ++m) Pm[p][m] = m == p ? d : Pm[p][m] * d;
#pragma unroll
                                for (int q2 = 0; q2 < CB; ++q2)
                                    if (q2 != p) {
                                        const float l = Pm[q2][p];
#pragma unroll
                                        for (int m = 0; m < CB; ++m)
                                            Pm[q2][m] = m == p ? -l * d : fmaf(-l, Pm[p][m], Pm[q2][m]);
                                    }
                            }
                            float w[CB];
#pragma unroll
                            for (int m = 0; m < CB; ++m) {
                                float other = 0.f, own = 0.f;
#pragma unroll
                                for (int t2 = 0; t2 < CB; ++t2) {
                                    other = fmaf(-creg[t2], Pm[t2][m], other);
                                    own = t0 == t2 ? Pm[t2][m] : own;
                                }
                                w[m] = pivot ? own : other;
                            }
#pragma unroll
                            for (int j = CB; j < F; j += 4) {
                                float v[CB][4];
#pragma unroll
                                for (int m = 0; m < CB; ++m) {
                                    const float4 q = *reinterpret_cast<const float4 *>(pb + m * CR + j);
                                    v[m][0] = q.x, v[m][1] = q.y, v[m][2] = q.z, v[m][3] = q.w;
                                }
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    float acc = pivot ? 0.f : creg[j + i];
#pragma unroll
                                    for (int m = 0; m < CB; ++m) acc = fmaf(w[m], v[m][i], acc);
                                    creg[j + i - CB] = acc;  // rotated
                                }
                            }
#pragma unroll
                            for (int m = 0; m < CB; ++m) creg[F - CB + m] = w[m];
                        }
                        pb = pb == fA ? fA + CB * CR : fA;
                    }
                }
                sync();  // the last step's published rows are read before the iteration overwrites them
            } else {
                factor64_2d<N, W, TG, NR, RS>(reinterpret_cast<double *>(gb + G::oEnd2), tig, lane, wig, bar_id, gt, Mx, My,
                                              u4, wi2, creg);
            }

            float *crow = gb + G::oC + (tig < F ? tig : 0) * G::CR;
            if constexpr (G::kCShared) {
                if (tig < F)
#pragma unroll
                    for (int j = 0; j < F; j += 4)
                        *reinterpret_cast<float4 *>(crow + j) = make_float4(creg[j], creg[j + 1], creg[j + 2], creg[j + 3]);
            }

            // S^T res at the thread's nodes
            auto transposed = [&](float (&z)[NS]) {
#pragma unroll
                for (int k = 0; k < NS; ++k) z[k] = 0.f;
#pragma unroll
                for (int p = 0; p < n; p += 4) {
                    const float4 r4v = *reinterpret_cast<const float4 *>(res + p);
                    float4 hr = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        if (k == 0 || !kSameI) {
                            const float4 xv = *reinterpret_cast<const float4 *>(hxT + ip[k] * G::NTP + p);
                            hr = make_float4(xv.x * r4v.x, xv.y * r4v.y, xv.z * r4v.z, xv.w * r4v.w);
                        }
                        const float4 yv = *reinterpret_cast<const float4 *>(hyT + jp[k] * G::NTP + p);
                        z[k] = fmaf(hr.x, yv.x, z[k]);
                        if (p + 1 < n) z[k] = fmaf(hr.y, yv.y, z[k]);
                        if (p + 2 < n) z[k] = fmaf(hr.z, yv.z, z[k]);
                        if (p + 3 < n) z[k] = fmaf(hr.w, yv.w, z[k]);
                    }
                }
                const float *rf = res + G::r4(n);
#pragma unroll
                for (int k = 0; k < NS; ++k) {
                    const int i = ip[k], j = jp[k];
                    float zf = fh0[i] * rf[j];
                    zf = fmaf(fh1[i], rf[N + j], zf);
                    zf = fmaf(fh0[j], rf[2 * N + i], zf);
                    zf = fmaf(fh1[j], rf[3 * N + i], zf);
                    z[k] = fmaf(wb, zf, z[k]);
                }
            };
            // d = G0^{-1} z at the thread's nodes (vec is overwritten)
            auto precondition = [&](const float (&z)[NS], float (&d)[NS]) {
#pragma unroll
                for (int k = 0; k < NS; ++k)
                    if (on[k]) {
                        fA[jp[k] * NR + ip[k]] = z[k];
                        vec[ip[k] * NR + jp[k]] = z[k];
                    }
                sync();
                // V0^{-T} z, first pass: [(j, a)] = sum_i Wx[i][a] z[(j, i)] (stored at [a][j]).
                // With it, the face rows' u = E0 V0^{-T} z comes from z directly: since
                // the rows of E0 are outer products, u on x face s at node k is
                // (My rx_s)_k with rx_s[j] = sum_i hvx_s[i] z[(j, i)], and on y face s
                // (Mx ry_s)_k with ry_s[i] = sum_j hvy_s[j] z[(j, i)]: first r, here
                {
                    float w[N];
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        if (k == 0 || !kSameI) load_rowf<N>(WxT + ip[k] * NR, w);
                        float v[N];
                        load_rowf<N>(fA + jp[k] * NR, v);
                        const float tv = dotf<N>(w, v);
                        if (on[k]) fB[ip[k] * NR + jp[k]] = tv;
                    }
                }
                if (tig < F) {
                    float h[N], v[N];
                    load_rowf<N>(u4 + fseg, h);
                    load_rowf<N>((tig < 2 * N ? fA : vec) + fk * NR, v);
                    mu4[fseg + fk] = dotf<N>(h, v);
                }
                sync();
                // second pass: t[(b, a)] = sum_j Wy[j][b] [(j, a)]; and u from r
                {
                    float v[N];
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        if (k == 0 || !kSameI) load_rowf<N>(fB + ip[k] * NR, v);
                        float w[N];
                        load_rowf<N>(WyT + jp[k] * NR, w);
                        const float tv = dotf<N>(w, v);
                        if (on[k]) fA[jp[k] * NR + ip[k]] = tv;
                    }
                }
                if (tig < F) {
                    float m[N], v[N];
                    load_rowf<N>((tig < 2 * N ? My : Mx) + fk * NR, m);
                    load_rowf<N>(mu4 + fseg, v);
                    uu4[tig] = dotf<N>(m, v);
                }
                sync();
                // V0^{-1} t, first pass: [(b, i)] = sum_a Wx[i][a] t[(b, a)] (stored at [i][b]);
                // and mu = C^{-1} u
                {
                    float w[N];
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        if (k == 0 || !kSameI) load_rowf<N>(Wx + ip[k] * NR, w);
                        float v[N];
                        load_rowf<N>(fA + jp[k] * NR, v);
                        const float tv = dotf<N>(w, v);
                        if (on[k]) fB[ip[k] * NR + jp[k]] = tv;
                    }
                }
                if (tig < F) {
                    float m = 0.f, m2 = 0.f;
#pragma unroll
                    for (int j = 0; j < F; j += 4) {
                        const float4 uv = *reinterpret_cast<const float4 *>(uu4 + j);
                        float4 cv;
                        if constexpr (G::kCShared) cv = *reinterpret_cast<const float4 *>(crow + j);
                        else cv = make_float4(creg[j], creg[j + 1], creg[j + 2], creg[j + 3]);
                        m = fmaf(cv.x, uv.x, m);
                        m2 = fmaf(cv.y, uv.y, m2);
                        m = fmaf(cv.z, uv.z, m);
                        m2 = fmaf(cv.w, uv.w, m2);
                    }
                    mu4[fseg + fk] = m + m2;  // r was last read in the previous stage
                }
                sync();
                // M mu: My mu_x,s and Mx mu_y,s
                if (tig < F) {
                    float m[N], v[N];
                    load_rowf<N>((tig < 2 * N ? My : Mx) + fk * NR, m);
                    load_rowf<N>(mu4 + fseg, v);
                    mm4[fseg + fk] = dotf<N>(m, v);
                }
                sync();
                // second pass, less V0^{-1} E0^T mu, which at node (i, j) is
                // sum_s (My mu_x,s)_j hvx_s[i] + hvy_s[j] (Mx mu_y,s)_i
                {
                    float v[N];
#pragma unroll
                    for (int k = 0; k < NS; ++k) {
                        const int i = ip[k], j = jp[k];
                        if (k == 0 || !kSameI) load_rowf<N>(fB + i * NR, v);
                        float w[N];
                        load_rowf<N>(Wy + j * NR, w);
                        float corr = mm4[j] * u4[i];
                        corr = fmaf(mm4[RS + j], u4[RS + i], corr);
                        corr = fmaf(u4[2 * RS + j], mm4[2 * RS + i], corr);
                        corr = fmaf(u4[3 * RS + j], mm4[3 * RS + i], corr);
                        d[k] = dotf<N>(w, v) - corr;
                    }
                }
            };
            // B x at face point tig, x in rows of RS
            auto face_row = [&](const auto *x, const auto *h0, const auto *h1) {
                const int side = tig / N, f = tig - side * N;
                const auto *hb = (side & 1) ? h1 : h0;
                auto v = x[0] * 0;
                v = 0;
#pragma unroll
                for (int m = 0; m < N; ++m) v = fma(hb[m], side < 2 ? x[f * RS + m] : x[m * RS + f], v);
                return v;
            };
            R q[NCOMP][NS];
            for (int cc = 0; cc < NCOMP && done; ++cc) {
                // phase 1's interpolant: the remap differs from it only by the face correction
#pragma unroll
                for (int k = 0; k < NS; ++k)
                    q[cc][k] = on[k] ? static_cast<const R *>(a.alpha)[qoff[cc] + ci[k]] : R(0);
                if constexpr (kPair) {
                    const float cref = fabsf(ch[cc]), gw = wb * gf[cc];
                    float before = 0.f;
                    done = false;
                    for (int it = 0; it < kIters; ++it) {
#pragma unroll
                        for (int k = 0; k < NS; ++k)
                            if (on[k]) vec[jp[k] * RS + ip[k]] = q[cc][k];
                        sync();
                        if (it > 0) {
                            float md, mx;
                            maxima(md, mx);
                            if (settled(md, mx + cref)) {
                                done = true;
                                break;
                            }
                            if (it > 3 && !(md < 0.75f * before)) break;  // not converging: left to the direct solve
                            before = md;
                        }
                        // stacked residual: particles phi* - V q, face points w (g - c) - w B q
#pragma unroll
                        for (int k = 0; k < NS; ++k) {
                            const float vq = apply_v<N, RS, float>(vec, hxf(k), hyf(k));
                            if (on[k]) res[ci[k]] = ph[cc][k] - vq;
                        }
                        if (tig < F) res[G::r4(n) + tig] = gw - wb * face_row((const float *)vec, fh0, fh1);
                        sync();
                        float z[NS], d[NS], dm = 0.f, xm = 0.f;
                        transposed(z);
                        precondition(z, d);
#pragma unroll
                        for (int k = 0; k < NS; ++k)
                            if (on[k]) {
                                q[cc][k] += d[k];
                                dm = fmaxf(dm, fabsf(d[k]));
                                xm = fmaxf(xm, fabsf(q[cc][k]));
                                if (!(fabsf(d[k]) < INFINITY)) dm = INFINITY;  // NaN too: never settles
                            }
                        publish(dm, xm);
                    }
                    if (!done) {  // the last correction
                        sync();
                        float md, mx;
                        maxima(md, mx);
                        done = settled(md, mx + cref);
                    }
                    if (cc + 1 < NCOMP) sync();
                } else {
                    // FP64 gradient z = S^T (rhs - S q) (the residual itself does not
                    // vanish at the solution), FP32 corrections G d = z.  The
                    // interpolant satisfies V alpha = phi* to rounding, so the first
                    // residual is that of the face rows alone; every later one is complete.
                    const double wd = a.w;
                    double *hyT64 = x64 + G::kX64, *hxr64 = hyT64 + N * G::NT64, *rf64 = hxr64 + N * G::NT64;
                    if (cc == 0)
#pragma unroll
                        for (int k = 0; k < NS; ++k)
                            if (on[k])
#pragma unroll
                                for (int j = 0; j < N; ++j) hyT64[j * G::NT64 + ci[k]] = hy[k][j];
                    float before = 0.f;
                    int e0 = 0;
                    done = false;
                    for (int o = 0; o < kOuter; ++o) {
#pragma unroll
                        for (int k = 0; k < NS; ++k)
                            if (on[k]) x64[jp[k] * RS + ip[k]] = q[cc][k];
                        sync();
                        if (o > 0)
#pragma unroll
                            for (int k = 0; k < NS; ++k) {
                                const double r = ph[cc][k] - apply_v<N, RS, double>(x64, hx[k], hy[k]);
                                if (on[k])
#pragma unroll
                                    for (int i = 0; i < N; ++i) hxr64[i * G::NT64 + ci[k]] = hx[k][i] * r;
                            }
                        if (tig < F) rf64[tig] = wd * (gf[cc] - face_row((const double *)x64, sh0, sh1));
                        sync();
                        double zd[NS];
                        int top = -5000;
#pragma unroll
                        for (int k = 0; k < NS; ++k) {
                            const int i = ip[k], j = jp[k];
                            double zf = sh0[i] * rf64[j];
                            zf = fma(sh1[i], rf64[N + j], zf);
                            zf = fma(sh0[j], rf64[2 * N + i], zf);
                            zf = fma(sh1[j], rf64[3 * N + i], zf);
                            zf *= wd;
                            if (o > 0) {
                                double z2 = 0.0;  // a second chain
#pragma unroll
                                for (int p = 0; p < n; p += 2) {
                                    const double2 xv = *reinterpret_cast<const double2 *>(hxr64 + i * G::NT64 + p);
                                    const double2 yv = *reinterpret_cast<const double2 *>(hyT64 + j * G::NT64 + p);
                                    zf = fma(xv.x, yv.x, zf);
                                    if (p + 1 < n) z2 = fma(xv.y, yv.y, z2);
                                }
                                zf += z2;
                            }
                            zd[k] = zf;
                            if (on[k] && zf != 0.0) top = max(top, exponent_of(zf));
                        }
                        top = group_top(top);
                        if (top == -5000) {  // zero gradient
                            done = o > 0;
                            if (done) break;
                            continue;
                        }
                        if (top > 1023) break;  // infinity or NaN
                        if (before == 0.f) e0 = top;
                        float zs[NS], xf[NS], dprev = 0.f, dmax = 0.f;
#pragma unroll
                        for (int k = 0; k < NS; ++k) {
                            zs[k] = float(scale2(zd[k], -top));
                            xf[k] = 0.f;
                        }
                        bool ok = false;
                        for (int it = 0; it < kIters; ++it) {
                            float z[NS], d[NS], dm = 0.f, xm = 0.f;
#pragma unroll
                            for (int k = 0; k < NS; ++k) z[k] = zs[k];
                            if (it > 0) {  // z - S^T S xf
#pragma unroll
                                for (int k = 0; k < NS; ++k) {
                                    const float v = apply_v<N, RS, float>(vec, hxf(k), hyf(k));
                                    if (on[k]) res[ci[k]] = -v;
                                }
                                if (tig < F) res[G::r4(n) + tig] = -wb * face_row((const float *)vec, fh0, fh1);
                                sync();
                                float zt[NS];
                                transposed(zt);
#pragma unroll
                                for (int k = 0; k < NS; ++k) z[k] += zt[k];
                            }
                            precondition(z, d);
#pragma unroll
                            for (int k = 0; k < NS; ++k)
                                if (on[k]) {
                                    xf[k] += d[k];
                                    vec[jp[k] * RS + ip[k]] = xf[k];
                                    dm = fmaxf(dm, fabsf(d[k]));
                                    xm = fmaxf(xm, fabsf(xf[k]));
                                    if (!(fabsf(d[k]) < INFINITY)) dm = INFINITY;
                                }
                            publish(dm, xm);
                            sync();
                            float md;
                            maxima(md, dmax);
                            ok = md < INFINITY;
                            if (!ok || inner_settled(md, dprev, dmax)) break;
                            if (it > 0 && !(md < 0.5f * dprev)) break;  // left to the next residual
                            dprev = md;
                        }
                        if (!ok) break;
                        float xm = 0.f;
#pragma unroll
                        for (int k = 0; k < NS; ++k) {
                            q[cc][k] += scale2(double(xf[k]), top);
                            if (on[k]) xm = fmaxf(xm, fabsf(float(scale2(q[cc][k], -e0))));
                        }
                        publish(0.f, xm);
                        if constexpr (W > 1) sync();
                        float mz, ms;
                        maxima(mz, ms);
                        const float d = ldexpf(dmax, max(top - e0, -140));
                        const float scale = ms + float(scale2(fabs(ch[cc]), -e0));
                        if (o > 0 && refined(d, scale)) {
                            done = true;
                            break;
                        }
                        if (o > 1 && !(d < kShrink * before)) break;  // not converging
                        before = d;
                    }
                    if (cc + 1 < NCOMP) sync();
                }
            }
            if (done)
#pragma unroll
                for (int cc = 0; cc < NCOMP; ++cc)
#pragma unroll
                    for (int k = 0; k < NS; ++k)
                        if (on[k]) {
                            if constexpr (kPair) {
                                float hi, lo;
                                two_sum2d(ch[cc], q[cc][k], hi, lo);
                                Qg[qoff[cc] + ci[k]] = make_float2(hi, lo + cl[cc]);
                            } else {
                                Qg[qoff[cc] + ci[k]] = ch[cc] + q[cc][k];
                            }
                        }
        }
    }
    // a group the iteration did not finish goes to the direct solve
    if (tig == 0) {
        a.fb[gid] = done ? 0 : 1;
        if (!done) {
            if (a.fbcount) atomicAdd(a.fbcount + (PHASE - 1), 1ull);
            // its direct-kernel CTA slot, listed once however many of its groups are flagged
            const Step2DArgs &L = BATCH ? args[0] : a0;
            const long long slot = ggid / Geo2D<N, R, NCOMP>::GPC;
            if (atomicExch(L.slot_mark + slot, 1u) == 0u) L.slot_list[atomicAdd(L.slot_ctl, 1u)] = unsigned(slot);
        }
    }
}

template <int N, typename R, int PHASE, bool BATCH, int NCOMP = 1, bool FAC64 = false>
__global__ void __launch_bounds__(FGeo<N, R>::kBlock, fast_ctas<N, R, PHASE>())
    sl2d_fast_kernel(const Step2DArgs a0, const Step2DArgs *__restrict__ args, const long long *__restrict__ prefix,
                     int ninst, int t)
{
    using G = FGeo<N, R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // node tables depend on N only (every instance of a batch class shares
    // them); computed once per context on the host (node_tables2d)
    const double *src = BATCH ? args[0].tab : a0.tab;
    R *tab = reinterpret_cast<R *>(smem_raw);
    for (int k = threadIdx.x; k < N * N + 5 * N; k += G::kBlock) {
        const double v = src[k];
        tab[k] = R(v);
        if constexpr (G::kF64) reinterpret_cast<float *>(smem_raw)[2 * G::kTab + k] = float(v);
    }
    __syncthreads();
    sl2d_fast_group<N, R, PHASE, BATCH, NCOMP, FAC64>(a0, args, prefix, ninst, t);
}

}  // namespace sl
