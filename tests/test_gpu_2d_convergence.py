"""What the iterations of the 2D step accept is as exact as their residual,
whatever the conditioning of a group's tensor factors: one step of rough
states (face jumps of 1e-3) group by group, by L = ||Wx||_inf ||Wy||_inf, the
FP32 forms against the FP64 kernels and those against the oracle; and the
moments after the whole horizon of the 64 x 64 workload."""

import numpy as np
import pytest

import sl_inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sl():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_07340_gb300 import build

    build.build()
    import paper_2009_07340_gb300 as sl

    return sl


def _nodes(N):
    return 0.5 * (1 - np.cos((np.arange(N) + 0.5) * np.pi / N))


def _conditioning(pb, dW):
    """L of every element-sample [M][E] (rotation drift, sinsin diffusion), from
    the mean displacements of the particle columns and rows."""
    N, K = pb["N"], pb["K"][0]
    xi, h = _nodes(N), 1.0 / K
    g = (np.arange(K)[:, None] + xi).ravel() * h
    X, Y = np.meshgrid(g, g, indexing="xy")  # [y][x]
    w, cx, cy = pb["drift"][1]
    D0, a, p, q = pb["diffusion"][1]
    u = (-w * (Y - cy), w * (X - cx))
    b = np.sqrt(2 * D0 * (1 + a * np.sin(p * np.pi * X) * np.sin(q * np.pi * Y)))
    out = []
    for s in range(dW.shape[0]):
        L = 1.0
        for d in (0, 1):
            disp = ((u[d] * pb["dt"] + b * dW[s, d]) / h).reshape(K, N, K, N)  # [ky][j][kx][i]
            xt = xi + (disp.mean(axis=1) if d == 0 else disp.mean(axis=3).transpose(0, 2, 1))  # [ky][kx][N]
            num = xi[:, None] - xt[..., None, :]
            den = xt[..., :, None] - xt[..., None, :]
            W = np.ones(xt.shape[:-1] + (N, N))  # the Lagrange basis on xt at the nodes
            for k in range(N):
                for m in range(N):
                    if m != k:
                        W[..., :, k] *= num[..., :, m] / den[..., k, m][..., None]
            L = L * np.abs(W).sum(-1).max(-1)
        out.append(L.ravel())
    return np.array(out)


def _rough_states(pb):
    """[M][E][j][i]: 1 and a linear part per element, a jump at every face."""
    N, E, xi = pb["N"], pb["K"][0] ** 2, _nodes(pb["N"])
    c = 1e-3 * np.random.default_rng(N).uniform(-0.5, 0.5, size=(3, pb["M"], E, 1, 1))
    return 1 + c[0] + c[1] * xi[None, :] + c[2] * xi[:, None]


# Tolerances, relative to a group's own maximum.  An accepted group's error is
# d rho / (1 - rho) with the last correction d <= 1e-6 of it.  Up to L = 64 the
# contraction rate rho of the remap is at most 0.14 (a spectral radius that a
# dense model of such elements gave at the whole node-gap step): 1.6e-7, and
# 2.8e-8 for the faces (0.027); together 2e-7.  From 64 to the limit (300, the
# mixed form 160) rho may reach 0.5 (eight corrections from 1e-3 to 1e-6 need
# 0.37), d for the worst: 1e-6 for the root mean square.  Above it the direct
# solve is exact to rounding.
@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("N,K,M", [(4, 64, 24), (6, 64, 12), (8, 64, 12), (10, 32, 16)])
def test_accepted_groups_are_converged(sl, precision, N, K, M):
    pb = I.config3(M=M, steps=1, K=K, N=N, dt=1e-9)
    q0 = _rough_states(pb)
    got = {}
    for prec in ("fp64", precision):
        with sl.Solver(pb, prec) as s:
            s.set_samples(0, q0)
            pb["dt"] = 0.5 * s.dt_max
            dW = s.wiener(0, 1, dt=pb["dt"])[0]
            s.step(dt=pb["dt"], steps=1)
            got[prec] = s.samples().reshape(M, K * K, N * N)
            direct = s.fallbacks
    L = _conditioning(pb, dW)
    err = np.abs(got[precision] - got["fp64"]).max(-1) / np.abs(got["fp64"]).max(-1)
    limit = 300 if precision == "fp32" else 160
    low, mid, high = L <= 64, (L > 64) & (L <= limit), L > limit
    # the iteration is what is tested: only groups above the limit, and a few
    # near it that need more than its corrections, go to the direct solve
    assert (L > limit * 1.001).sum() <= direct[1] <= (L > limit * 0.999).sum() + 0.05 * mid.sum()
    assert err[low].max() <= 2e-7
    assert mid.sum() == 0 or np.sqrt((err[mid] ** 2).mean()) <= 1e-6
    assert high.sum() == 0 or err[high].max() <= 2e-7


# FP64: corrections shrink by 0.45 or more, the last is below 1e-13: 0.8e-13 of
# the group remains in its faces and in its remap, which answers a face error
# by a few times (its Lebesgue constant); rounding at a condition of L adds
# L 2^-53 = 5e-13 at L = 4096.  1e-12 in all.
@pytest.mark.parametrize("N", [4, 6, 8, 10])
def test_fp64_groups_are_refined_to_the_end(sl, orc, N):
    K, M = 16, 16
    pb = I.config3(M=M, steps=1, K=K, N=N, dt=1e-9)
    q0 = _rough_states(pb)
    with sl.Solver(pb, "fp64") as s:
        pb["dt"] = s.dt_max  # the whole node-gap bound: L over three orders of magnitude
        s.set_samples(0, q0)
        dW = s.wiener(0, 1, dt=pb["dt"])[0]
        s.step(dt=pb["dt"], steps=1)
        got = s.samples().reshape(M, K * K, N * N)
        direct = s.fallbacks
    ref = orc.run(pb, state_in=q0, want_states=True, nthreads=16, ns=M)["states"].reshape(got.shape)
    L = _conditioning(pb, dW)
    err = np.abs(got - ref).max(-1) / np.abs(ref).max(-1)
    assert direct[1] < 0.5 * L.size  # most groups are the iteration's
    assert err[L <= 4096].max() <= 1e-12


# A boundary weight does not hinder the FP64 and FP32 iterations: the null
# directions of the face rows (one per corner), where the capacitance matrix is
# w^-2 alone, are filled up before its FP32 inversion.  Rough states at a fifth
# of the node-gap step (L below 100): nearly every group is iterated.  FP64 as
# above.  FP32: the last correction is below 1e-6 and rho at most 0.5, in the
# faces and in the remap: 2e-6.
@pytest.mark.parametrize("w", [10.0, 30.0])
@pytest.mark.parametrize("N,K", [(5, 16), (8, 16), (11, 12)])
def test_boundary_weights_converge(sl, orc, N, K, w):
    M = 16
    pb = I.with_(I.config3(M=M, steps=1, K=K, N=N, dt=1e-9), bc_weight=w)
    q0 = _rough_states(pb)
    ref = None
    for prec, tol in (("fp64", 1e-12), ("fp32", 2e-6)):
        with sl.Solver(pb, prec) as s:
            s.set_samples(0, q0)
            pb["dt"] = 0.2 * s.dt_max
            s.step(dt=pb["dt"], steps=1)
            got = s.samples().reshape(M, K * K, N * N)
            direct = s.fallbacks
        if ref is None:
            ref = orc.run(pb, state_in=q0, want_states=True, nthreads=16, ns=M)["states"].reshape(got.shape)
        assert direct[1] <= 0.01 * M * K * K, prec
        assert (np.abs(got - ref).max(-1) / np.abs(ref).max(-1)).max() <= tol, prec


def test_whole_horizon_of_the_64x64_workload(sl):
    # 500 steps at half the node-gap step, where errors of single groups add up:
    # FP32 and mixed means within the tolerance of the FP32 forms of FP64's
    pb = I.config3(M=16, steps=500, dt=I.DT_CFG3_HALF)
    mean = {}
    for prec in ("fp64", "fp32", "mixed"):
        with sl.Solver(pb, prec) as s:
            s.step()
            mean[prec] = s.moments()[0]
    scale = np.abs(mean["fp64"]).max()
    for prec in ("fp32", "mixed"):
        assert np.abs(mean[prec] - mean["fp64"]).max() / scale <= 1e-5, prec
