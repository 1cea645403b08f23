"""The FP64 reciprocal and the integer-pipe conversions of the 2D kernels
(rcp64, wide, narrow in sl_step2d_fast.cuh) against IEEE division and
conversion over their ranges.  They only precondition an iteration, so that a
wrong one would show as direct solves, not in the results: a small program
built with nvcc runs them alone."""

import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROG = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "sl_step2d_fast.cuh"
__global__ void k_rcp(const double *x, double *y, long n) {
    const long i = blockIdx.x * 256l + threadIdx.x;
    if (i < n) y[i] = sl::rcp64(x[i]);
}
__global__ void k_wide(const float *x, double *y, long n) {
    const long i = blockIdx.x * 256l + threadIdx.x;
    if (i < n) y[i] = sl::wide(x[i]);
}
__global__ void k_narrow(const double *x, float *y, long n) {
    const long i = blockIdx.x * 256l + threadIdx.x;
    if (i < n) y[i] = sl::narrow(x[i]);
}
template <typename A, typename B> int run(void (*k)(const A *, B *, long), const char *in, const char *out) {
    FILE *f = fopen(in, "rb");
    if (!f) return 1;
    fseek(f, 0, SEEK_END);
    const long n = ftell(f) / long(sizeof(A));
    rewind(f);
    std::vector<A> x(n);
    std::vector<B> y(n);
    if (long(fread(x.data(), sizeof(A), n, f)) != n) return 2;
    fclose(f);
    A *dx;
    B *dy;
    if (cudaMalloc(&dx, n * sizeof(A)) || cudaMalloc(&dy, n * sizeof(B))) return 3;
    if (cudaMemcpy(dx, x.data(), n * sizeof(A), cudaMemcpyHostToDevice)) return 4;
    k<<<unsigned((n + 255) / 256), 256>>>(dx, dy, n);
    if (cudaMemcpy(y.data(), dy, n * sizeof(B), cudaMemcpyDeviceToHost)) return 5;
    f = fopen(out, "wb");
    if (!f || long(fwrite(y.data(), sizeof(B), n, f)) != n) return 6;
    return fclose(f);
}
int main(int, char **v) {
    switch (atoi(v[1])) {
    case 0: return run(k_rcp, v[2], v[3]);
    case 1: return run(k_wide, v[2], v[3]);
    default: return run(k_narrow, v[2], v[3]);
    }
}
"""


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    import torch

    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if not torch.cuda.is_available() or nvcc is None:
        pytest.skip("no CUDA device or no nvcc")
    d = tmp_path_factory.mktemp("helpers")
    (d / "h.cu").write_text(PROG)
    subprocess.check_call([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "paper_2009_07340_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), str(d / "h.cu"), "-o", str(d / "h")])

    def call(op, x, out):
        x.tofile(d / "in")
        subprocess.check_call([str(d / "h"), str(op), str(d / "in"), str(d / "out")])
        return np.fromfile(d / "out", dtype=out)

    return call


def _bits64(lo, hi, count, seed):
    """Doubles of both signs, exponents lo to hi (unbiased), random mantissas and
    the all-zero and all-one ones of every exponent."""
    rng = np.random.default_rng(seed)
    e = np.arange(lo, hi + 1)
    man = np.concatenate([rng.integers(0, 1 << 52, size=(len(e), count), dtype=np.uint64),
                          np.tile(np.array([0, 1, (1 << 52) - 1], dtype=np.uint64), (len(e), 1))], axis=1)
    b = ((e + 1023).astype(np.uint64) << np.uint64(52))[:, None] | man
    b = b.ravel()
    return np.concatenate([b, b | np.uint64(1 << 63)]).view(np.float64)


def test_reciprocal(helper):
    # two Newton-Raphson steps from an approximation of 2^-14 or better leave
    # 2^-56 of error beside the last operation's rounding (2^-53 or half a unit
    # in the last place): at most one unit from the rounded quotient
    x = np.concatenate([_bits64(-1022, 1023, 500, 1), [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310]])
    with np.errstate(divide="ignore", over="ignore"):
        ref = 1.0 / x
    got = helper(0, x, np.float64)
    inside = (np.abs(x) >= 2.0 ** -511) & (np.abs(x) < 2.0 ** 512 * (1 + 2.0 ** -20))
    assert np.all(np.abs(got[inside].view(np.int64) - ref[inside].view(np.int64)) <= 1)
    assert np.array_equal(got[~inside], ref[~inside], equal_nan=True)  # the division itself


def test_widening_is_exact(helper):
    rng = np.random.default_rng(2)
    b = (np.arange(1, 255, dtype=np.uint32) << 23)[:, None] | rng.integers(0, 1 << 23, size=(254, 500), dtype=np.uint32)
    b = np.concatenate([b.ravel(), [0, 0x007FFFFF + 1, 0x7F7FFFFF]]).astype(np.uint32)
    x = np.concatenate([b, b | np.uint32(1 << 31)]).view(np.float32)
    assert np.array_equal(helper(1, x, np.float64).view(np.int64), x.astype(np.float64).view(np.int64))


def test_narrowing_rounds_to_nearest_ties_away(helper):
    x = _bits64(-126, 126, 500, 3)
    top = np.uint64(0xFFFFFFFFF0000000)
    ties = ((x.view(np.uint64) & top) & ~np.uint64(1 << 28)) | np.uint64(1 << 28)  # half a unit beyond a float
    x = np.concatenate([x, ties.view(np.float64), (ties - np.uint64(1)).view(np.float64), [0.0, -0.0]])
    got = helper(2, x, np.float32).astype(np.float64)
    ref = x.astype(np.float32).astype(np.float64)  # to nearest, ties to even
    assert np.array_equal(np.abs(got - x), np.abs(ref - x))  # as near (the differences are exact)
    tie = (x.view(np.uint64) & np.uint64((1 << 29) - 1)) == np.uint64(1 << 28)
    assert np.all(np.abs(got[tie]) > np.abs(x[tie])) and np.array_equal(got[~tie], ref[~tie])
    # outside its normal range: zero below, the conversion itself above
    small = np.concatenate([_bits64(-1022, -127, 20, 4), [5e-324]])
    assert np.all(helper(2, small, np.float32) == 0.0)
    large = np.concatenate([_bits64(127, 1023, 20, 5), [np.inf, -np.inf, np.nan]])
    with np.errstate(over="ignore"):
        assert np.array_equal(helper(2, large, np.float32), large.astype(np.float32), equal_nan=True)
