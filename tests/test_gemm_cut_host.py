"""How many CTAs share a tile of the SINT4 GEMM, on the CPU."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "lq_gemm_cut.h"
extern "C" int split(int M, int N, int stages, int ctas, int asked) {
  const int clusters[3] = {74, 34, 15};   // as a B200 holds them
  return pick_split(M, (long long)lq_ceil_div(M, LQ_BM) * lq_ceil_div(N, LQ_BM), stages, ctas, clusters, asked);
}
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "split.cpp").write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2604_18117_b200", "csrc"), "-I", os.path.join(cuda, "include"), str(d / "split.cpp"), "-o",
                    str(d / "split.so")], check=True)
    lib = ctypes.CDLL(str(d / "split.so"))
    return lambda M, K, N, branch=1, ctas=148, asked=0: lib.split(M, N, -(-K // 128) + branch, ctas, asked)


# Timed by four and by eight, each in turn on one card: the faster, where they differ by over 2 %.
@pytest.mark.parametrize("M,K,N,faster", [(384, 872, 640, 4), (512, 872, 264, 4), (384, 896, 512, 4), (384, 1016, 640, 4), (384, 1152, 640, 4),
                                          (128, 864, 1152, 4), (128, 848, 1024, 4), (256, 896, 512, 4), (384, 1240, 640, 4), (384, 1376, 640, 4),
                                          (48, 872, 640, 8), (60, 1152, 512, 8), (128, 1536, 640, 8), (192, 1536, 264, 8), (128, 1536, 128, 8)])
def test_eight_share_a_tile_only_where_that_is_faster(split, M, K, N, faster):
    assert split(M, K, N) == faster


@pytest.mark.parametrize("M,K,N,branch,n", [(1, 1152, 1152, 1, 8), (1, 640, 1152, 1, 4), (60, 640, 1152, 1, 4), (64, 640, 1152, 1, 1), (128, 640, 1152, 1, 1),
                                            (120, 1152, 4608, 1, 2), (256, 1152, 4608, 1, 2), (256, 4608, 1152, 1, 4), (120, 8192, 1152, 1, 8),
                                            (8192, 1152, 1152, 1, 1), (1, 512, 1152, 0, 1)])
def test_the_other_lines_of_the_rule(split, M, K, N, branch, n):
    assert split(M, K, N, branch) == n


@pytest.mark.parametrize("asked", [0, 2, 4, 8])
def test_what_shares_a_tile_has_a_stage_each_and_room(split, asked):
    for ctas in (1, 2, 6, 148):
        for K in (64, 128, 512, 1152, 8192):
            for M in (1, 127, 129, 1000, 32768):
                for N in (8, 1152, 8192):
                    n, units = split(M, K, N, ctas=ctas, asked=asked), -(-M // 128) * -(-N // 128)
                    assert n in (1, 2, 4, 8) and n <= ctas and n <= -(-K // 128) + 1 and (n == 1 or n * units <= ctas)
                    assert asked == 0 or n in (1, asked)
