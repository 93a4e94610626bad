"""How the MX GEMM's launches are cut, on the CPU: where a pair of CTAs keeps its weights in shared memory, and that what it keeps and
the ring beside it fit."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIELDS = ("width", "tiles_n", "pair", "ctas", "stages", "resident", "b_slots", "smem")
SOURCE = """
#include "lq_gemm_mx_cut.h"
extern "C" int cut(int M, int N, int b_wrap, int planes, int branch, int acc, int weight_bits, int out_bytes, int ctas, int width, int* out) {
  lqmx::MxCut c;
  if (!lqmx::plan_mx({M, N, b_wrap, planes, branch != 0, acc != 0, weight_bits, out_bytes}, ctas, width, true, c)) return 0;
  const int v[] = {c.width, c.tiles_n, c.pair, c.ctas, c.stages, c.resident, c.b_slots, c.smem};
  for (int i = 0; i < 8; ++i) out[i] = v[i];
  return 1;
}
"""
# digit planes of the activations, branch, an accumulator of its own, bits of a weight
FORMATS = {"mxint4 none": (1, 0, 0, 6), "mxint4 w8a8": (1, 1, 1, 6), "mxint4 w16a16": (1, 1, 0, 6), "mxfp4": (1, 1, 0, 4), "mxint4a8": (2, 1, 0, 6)}


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    d = tmp_path_factory.mktemp("cut")
    (d / "cut.cpp").write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2604_18117_b200", "csrc"), "-I", os.path.join(cuda, "include"), str(d / "cut.cpp"), "-o", str(d / "cut.so")],
                   check=True)
    lib = ctypes.CDLL(str(d / "cut.so"))

    def get(fmt, M, K, N, out_bytes=2, ctas=148, width=0):
        out = (ctypes.c_int * 8)()
        return dict(zip(FIELDS, out)) if lib.cut(M, N, -(-K // 128), *FORMATS[fmt], out_bytes, ctas, width, out) else None

    return get


# Timed with the weights kept over the time without, each on the same card in turn.
SLOWER = [("mxint4a8", 16384, 1280, 4608, 2, 1.09), ("mxint4a8", 4096, 1280, 2048, 2, 1.08), ("mxint4a8", 2560, 1152, 4608, 2, 1.03),
          ("mxfp4", 16384, 1280, 2048, 2, 1.06), ("mxfp4", 10240, 1152, 7168, 2, 1.10), ("mxfp4", 2560, 768, 2048, 2, 1.04),
          ("mxfp4", 2524, 1112, 7040, 4, 1.11), ("mxint4 w8a8", 10240, 768, 1152, 2, 1.04), ("mxint4 w8a8", 6144, 1152, 1152, 2, 1.02),
          ("mxint4 w8a8", 16208, 896, 8104, 2, 1.20), ("mxint4 w8a8", 7645, 1360, 5776, 2, 1.16), ("mxint4 w8a8", 16384, 768, 7168, 2, 1.04),
          ("mxint4 none", 16384, 1280, 7168, 2, 1.10), ("mxint4 none", 15481, 824, 6488, 4, 1.12), ("mxint4 w16a16", 11501, 1032, 6056, 4, 1.13),
          ("mxint4 w16a16", 12668, 1680, 416, 2, 1.06)]
FASTER = [("mxfp4", 8192, 1152, 3456, 2, 0.95), ("mxfp4", 6144, 768, 3072, 2, 0.89), ("mxint4 w8a8", 8192, 1152, 3456, 2, 0.96),
          ("mxint4 w8a8", 12288, 1024, 2048, 2, 0.95), ("mxint4a8", 8192, 1152, 3456, 2, 0.95), ("mxint4a8", 12288, 768, 3072, 2, 0.92),
          ("mxint4 none", 6144, 768, 1152, 2, 0.93), ("mxint4 none", 16384, 1280, 1152, 2, 0.88), ("mxint4 w16a16", 6144, 1152, 4608, 2, 0.91)]


@pytest.mark.parametrize("fmt,M,K,N,out_bytes,ratio", SLOWER + FASTER)
def test_weights_stay_only_where_that_is_faster(cut, fmt, M, K, N, out_bytes, ratio):
    assert cut(fmt, M, K, N, out_bytes)["resident"] == (ratio < 1)


@pytest.mark.parametrize("fmt", FORMATS)
def test_what_is_kept_and_the_ring_fit(cut, fmt):
    """Every cut's shared memory; a resident one's ring has no more stages than K, whose slots are then free in time."""
    kept = 0
    for K in range(128, 8193, 128):
        for N in (8, 264, 1152, 3456, 8192):
            for M in (1, 129, 2305, 4096, 8192, 16384, 32768):
                c = cut(fmt, M, K, N)
                assert 0 < c["smem"] <= 227 * 1024 and c["stages"] >= 3 and c["ctas"] <= 148
                if c["resident"]:
                    kept += 1
                    assert c["pair"] and 2 * c["stages"] >= K // 128 >= c["stages"] and c["b_slots"] >= K // 128
    assert kept > 10


@pytest.mark.parametrize("fmt,K,width", [("mxint4 none", 1152, 192), ("mxint4 w8a8", 1152, 160), ("mxint4 w16a16", 1032, 192), ("mxfp4", 1152, 192), ("mxint4a8", 1152, 192)])
def test_the_sizes_of_the_gpu_test_reach_the_kept_weights(cut, fmt, K, width):
    assert cut(fmt, 2600, K, 1160, out_bytes=4, ctas=6, width=width)["resident"]
