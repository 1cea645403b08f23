"""CPU check of the rule that takes a 1D FP64 solve to the split kernel
(split1d_fields in sl_geometry1d.cuh): on 152 SMs the small solves of
test_small_fp64_solves_equal_the_first_samples_of_large_ones run on it and the
large ones on the thread-per-element kernel, so that the test compares the two
at every order above 2; and its bounds hold over all sizes.  A host program prints the rule."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROG = r"""
#include <cstdio>
#include "sl_geometry1d.cuh"
int main() {
    int N, K, M, ncomp, nsm;
    while (scanf("%d %d %d %d %d", &N, &K, &M, &ncomp, &nsm) == 5) {
        int S, C, T;
        sl::geometry1d(K, M, nsm, sl::kMaxThreads1D, S, C, T);
        printf("%d %d %d %d %d\n", S, C, T, sl::split1d_fields(N, K, M, ncomp, S, C, T, nsm), sl::split1d_lanes(N));
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which(os.environ.get("CXX", "g++"))
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rule")
    (d / "r.cpp").write_text(PROG)
    subprocess.check_call([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2009_07340_gb300", "csrc"),
                           str(d / "r.cpp"), "-o", str(d / "r")])

    def call(cases):
        text = "".join("%d %d %d %d %d\n" % c for c in cases)
        out = subprocess.run([str(d / "r")], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]

    return call


def test_small_solves_are_split_and_large_ones_are_not(rule):
    sizes = [(N, K) for N in range(2, 17) for K in (1, 3, 8, 32)]
    small = rule([(N, K, 5, 1, 152) for N, K in sizes])
    large = rule([(N, K, int(20000 / K ** 0.5), 1, 152) for N, K in sizes])
    for (N, K), s, b in zip(sizes, small, large):
        assert b[3] == 0, (N, K)
        # N = 2: fewer instructions per thread; 32 elements take eight warps of
        # lanes, which pays from N = 5 on (6 N^2 + 22 N against 2 (8 N + 60))
        assert (s[3] > 0) == (N > 2 and (K < 32 or N > 4)), (N, K)


def test_rule_keeps_to_the_kernels_limits(rule):
    cases = [(N, K, M, c, nsm) for N in (2, 3, 8, 9, 16) for K in (1, 2, 31, 33, 64, 65, 256, 257, 2048)
             for M in (1, 2, 7, 500, 20000) for c in (1, 2) for nsm in (1, 132, 152)]
    for (N, K, M, c, nsm), (S, C, T, F, G) in zip(cases, rule(cases)):
        assert C * T >= K and 1 <= S <= M and S * T <= 256 and 1 <= C <= 8
        assert 0 <= F <= M and F * K * G <= 512
        if N < 3 or c != 1 or C != 1:
            assert F == 0
        elif K * M == 1:
            assert F == 1  # the smallest solves always are
