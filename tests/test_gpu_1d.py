"""GPU parity of the 1D path against the FP64 CPU oracle, through the C ABI.

Bars: Philox words / FP64 Wiener increments bit-exact; SL_FP64 moments and
per-sample states within 1e-10 of the oracle (relative to max |mean|);
SL_MIXED / SL_FP32 moments within 1e-5.
"""

import numpy as np
import pytest

import sl_inputs as I

pytestmark = pytest.mark.gpu

FP64_TOL = 1e-10
MIXED_TOL = 1e-5


@pytest.fixture(scope="module")
def sl():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_07340_gb300 import build

    build.build()
    import paper_2009_07340_gb300 as sl

    return sl


def _rel(a, b, scale=None):
    scale = np.abs(b).max() if scale is None else scale
    return float(np.abs(np.asarray(a) - np.asarray(b)).max() / scale)


@pytest.mark.parametrize("dim,step0", [(1, 0), (1, 123456), (2, 7), (1, 2 ** 32 - 3)])
def test_wiener_bit_exact(sl, orc, dim, step0):
    pb = I.config1() if dim == 1 else I.with_(I.config3(M=37, K=2, N=3))
    pb = I.with_(pb, M=37)
    dt = 1.7e-4
    with sl.Solver(pb) as s:
        got = s.wiener(step0, 3, dt)
    want = orc.wiener(pb["seed"], dim, 37, step0, 3, dt)
    assert got.shape == want.shape
    assert np.array_equal(got.view(np.uint64), want.view(np.uint64))


def _run_pair(sl, orc, pb, precision="fp64", nthreads=8, states=4):
    ref = orc.run(pb, want_states=True, nthreads=nthreads, ns=pb["M"])
    with sl.Solver(pb, precision) as s:
        s.step()
        mean, m2 = s.moments()
        st = s.samples(0, states)
    M = pb["M"]
    rm, rq = ref["sum"] / M, ref["sumsq"] / M
    scale = np.abs(rm).max()
    return (_rel(mean, rm, scale), _rel(m2, rq),
            _rel(st, ref["states"][:states], scale))


def test_config1_fp64_full(sl, orc):
    e_mean, e_m2, e_st = _run_pair(sl, orc, I.config1())
    assert e_mean <= FP64_TOL and e_m2 <= FP64_TOL and e_st <= FP64_TOL


@pytest.mark.parametrize("N", [4, 8, 12, 16])
def test_config2_shape_fp64(sl, orc, N):
    # config-2 fields and dt on a 48-element mesh, 61 samples, 40 steps
    pb = I.config2(N=N, M=61, steps=40, K=48)
    e_mean, e_m2, e_st = _run_pair(sl, orc, pb)
    assert e_mean <= FP64_TOL and e_m2 <= FP64_TOL and e_st <= FP64_TOL


@pytest.mark.parametrize("K,N,M", [(1, 5, 9), (2, 2, 33), (3, 3, 5), (7, 7, 70), (13, 9, 3),
                                   (100, 6, 5), (256, 16, 3), (257, 5, 3), (300, 8, 2), (1000, 4, 2)])
def test_ragged_shapes_and_clusters_fp64(sl, orc, K, N, M):
    pb = I.config2(N=N, M=M, steps=12, K=K)
    pb["dt"] = 0.5 * orc.dt_max(pb)
    e_mean, e_m2, e_st = _run_pair(sl, orc, pb, states=M)
    assert e_mean <= FP64_TOL and e_st <= FP64_TOL


@pytest.mark.parametrize("precision", ["mixed", "fp32"])
@pytest.mark.parametrize("N", [4, 8, 16])
def test_config2_shape_mixed(sl, orc, precision, N):
    pb = I.config2(N=N, M=64, steps=200, K=64)
    e_mean, _, _ = _run_pair(sl, orc, pb, precision)
    assert e_mean <= MIXED_TOL


# At N=16 and dt = 7.33e-7 (the Eq. (1d_timestep) node-gap bound of that
# order) the step amplifies perturbations by ~0.85 % per step (pinned on the
# oracle alone in test_oracle_physics.py::test_amplification_at_the_bound):
# over 1000 steps any rounding difference grows ~5000x, so two correct FP64
# implementations with different operation orders end ~5e-10 apart.  The
# 1e-10 bar is applied where the step is stable (half that dt, or the first
# 300 steps); the full horizon at the bound uses the amplified bound 2e-9.
FP64_TOL_AT_BOUND = 2e-9


@pytest.mark.parametrize("N,frac,steps,tol", [(16, 1.0, 1000, FP64_TOL_AT_BOUND), (16, 1.0, 300, FP64_TOL),
                                              (16, 0.5, 1000, FP64_TOL), (12, 1.0, 1000, FP64_TOL)])
def test_config2_full_size_fp64_sampled(sl, orc, N, frac, steps, tol):
    # the full workload (K=256, M=4096) in the launch configuration of the
    # benchmark; the oracle recomputes samples 0 and 4095 one by one, and the
    # device moments must equal the mean of all device samples
    pb = I.config2(N=N, steps=steps)
    pb["dt"] = frac * I.DT_CFG2
    with sl.Solver(pb, "fp64") as s:
        s.step()
        mean, m2 = s.moments()
        st = s.samples()
    for sidx in (0, pb["M"] - 1):
        ref = orc.run(pb, s0=sidx, ns=1, want_states=True)["states"][0]
        assert _rel(st[sidx], ref) <= tol
    assert _rel(mean, st.mean(0)) <= 1e-13
    assert _rel(m2, (st ** 2).mean(0)) <= 1e-13


@pytest.mark.parametrize("precision", ["mixed", "fp32"])
@pytest.mark.parametrize("N,frac", [(16, 0.5), (12, 1.0), (8, 1.0), (4, 1.0)])
def test_config2_full_size_mixed_vs_fp64(sl, orc, precision, N, frac):
    # the full workload in the benchmark's launch configuration: the moments
    # against the FP64 GPU path (itself pinned to the oracle above), and the
    # first and last samples against the oracle recomputing them one by one
    pb = I.config2(N=N)
    pb["dt"] = frac * I.DT_CFG2
    with sl.Solver(pb, "fp64") as s:
        s.step()
        m64, _ = s.moments()
    with sl.Solver(pb, precision) as s:
        s.step()
        mlo, _ = s.moments()
        first, last = s.samples(0, 1)[0], s.samples(pb["M"] - 1, 1)[0]
    assert _rel(mlo, m64) <= MIXED_TOL
    scale = np.abs(m64).max()
    for sidx, got in ((0, first), (pb["M"] - 1, last)):
        ref = orc.run(pb, s0=sidx, ns=1, want_states=True)["states"][0]
        assert _rel(got, ref, scale) <= MIXED_TOL


def test_restart_and_checkpoint_bitwise(sl):
    pb = I.config2(N=8, M=16, steps=30, K=32)
    with sl.Solver(pb) as a:
        a.step(steps=30)
        full = a.samples()
    with sl.Solver(pb) as b:
        b.step(steps=18)
        b.step(steps=12)
        assert b.step_count == 30
        assert np.array_equal(b.samples(), full)
    with sl.Solver(pb) as c:
        c.step(steps=18)
        ck = c.samples()
    with sl.Solver(pb) as d:
        d.set_samples(0, ck)
        d.step_count = 18
        d.step(steps=12)
        assert np.array_equal(d.samples(), full)


def test_sample_independent_of_batch(sl):
    # a sample's trajectory does not depend on how many samples run with it
    pb = I.config2(N=6, M=5, steps=20, K=20)
    with sl.Solver(pb) as a:
        a.step()
        small = a.samples()
    with sl.Solver(I.with_(pb, M=300)) as b:
        b.step()
        big = b.samples(0, 5)
    assert np.array_equal(small, big)


def test_dt_guard_and_errors(sl, orc):
    pb = I.config2(N=16, M=4, steps=1, K=256)
    with sl.Solver(pb, strict_dt=True) as s:
        assert s.dt_max == pytest.approx(orc.dt_max(pb), rel=1e-12)
        with pytest.raises(sl.SLError) as e:
            s.step(dt=2 * s.dt_max, steps=1)
        assert e.value.code == -2
        s.step(dt=s.dt_max, steps=1)  # at the bound: accepted
        with pytest.raises(sl.SLError):
            s.step(dt=-1.0, steps=1)
        s.moments()


def test_moments_device(sl):
    import torch

    pb = I.config2(N=8, M=33, steps=5, K=16)
    with sl.Solver(pb, stream=torch.cuda.current_stream().cuda_stream) as s:
        s.step()
        mean, m2 = s.moments()
        dm = torch.zeros(s.V, dtype=torch.float64, device="cuda")
        dq = torch.zeros(s.V, dtype=torch.float64, device="cuda")
        s.moments_device(dm, dq)
        torch.cuda.synchronize()
        assert np.array_equal(dm.cpu().numpy(), mean.ravel())
        assert np.array_equal(dq.cpu().numpy(), m2.ravel())


def test_sample_ranges_shard_bitwise(sl):
    # disjoint sample ranges on separate contexts (as on separate GPUs)
    # reproduce the single-context run sample for sample
    pb = I.config2(N=8, M=10, steps=15, K=24)
    with sl.Solver(pb) as a:
        a.step()
        whole = a.samples()
    with sl.Solver(I.with_(pb, M=4)) as b, sl.Solver(I.with_(pb, M=6), sample0=4) as c:
        b.step()
        c.step()
        assert np.array_equal(np.concatenate([b.samples(), c.samples()]), whole)


@pytest.mark.parametrize("K", [1, 3, 8, 32])
@pytest.mark.parametrize("N", range(2, 17))
def test_small_fp64_solves_equal_the_first_samples_of_large_ones(sl, N, K):
    # a small FP64 solve deals an element's nodes out to lanes, a large one
    # has a thread per element: the same operations in the same order.  Five
    # samples (several fields in a block, the last one partly filled) against
    # the first five of 20000 / K^(1/2); periodic, then Dirichlet with a weight.
    pb = I.config2(N=N, M=5, steps=4, K=K)
    pb["dt"] = 1e-6
    large = I.with_(pb, M=int(20000 / K ** 0.5))
    for extra in ({}, {"periodic": False, "bc_weight": 3.0,
                       "ghost": np.stack([np.linspace(0.8, 1.2, 4), np.linspace(1.3, 0.9, 4)], axis=1)}):
        got = []
        for p in (I.with_(pb, **extra), I.with_(large, **extra)):
            with sl.Solver(p, "fp64") as s:
                s.step()
                got.append(s.samples(0, 5))
        assert np.array_equal(got[0], got[1])


def test_one_element_one_sample_of_two_nodes(sl, orc):
    # FP64 N = 2: a block of one thread fills the node tables
    pb = I.config2(N=2, M=1, steps=5, K=1)
    pb["dt"] = 0.5 * orc.dt_max(pb)
    ref = orc.run(pb, want_states=True, ns=1)["states"]
    with sl.Solver(pb, "fp64") as s:
        s.step()
        assert np.abs(s.samples() - ref).max() / np.abs(ref).max() <= FP64_TOL
