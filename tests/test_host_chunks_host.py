"""Row chunks of a call from host memory, on the CPU: they cover the rows, and never outnumber the events kept for them."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "lq_internal.h"
#if MOST
#undef LQ_HOST_CHUNKS
#define LQ_HOST_CHUNKS MOST
#endif
#include "lq_host_chunks.h"
extern "C" int chunks(int M, double x, double y, int* out) {
  struct { int end[LQ_HOST_CHUNKS], guard[16]; } s;
  for (int& g : s.guard) g = -7;
  const int n = host_chunks(M, (size_t)x, (size_t)y, s.end);
  for (int g : s.guard)
    if (g != -7) return -1;
  for (int i = 0; i < n && i < LQ_HOST_CHUNKS; ++i) out[i] = s.end[i];
  return n;
}
"""


@pytest.fixture(scope="module", params=[0, 5], ids=["as built", "five"])
def chunks(tmp_path_factory, request):
    d = tmp_path_factory.mktemp("chunks")
    (d / "chunks.cpp").write_text(SOURCE)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-DMOST={request.param}", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2604_18117_b200", "csrc"), "-I", os.path.join(cuda, "include"), str(d / "chunks.cpp"), "-o",
                    str(d / "chunks.so")], check=True)
    lib = ctypes.CDLL(str(d / "chunks.so"))
    lib.chunks.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_void_p]

    def get(M, x, y):
        out = (ctypes.c_int * 16)()
        n = lib.chunks(M, x, y, out)
        assert n >= 1, "written beyond the end"
        return list(out)[:n]

    get.most = request.param or 8
    return get


@pytest.mark.parametrize("x,y", [(1e3, 1e3), (7e6, 7e6), (7e6, 14e6), (5e8, 5e8)])
def test_chunks_cover_the_rows(chunks, x, y):
    for M in [*range(1, 2600), 4096, 5001, 8192, 32768]:
        end = chunks(M, x, y)
        assert len(end) <= chunks.most and end[-1] == M
        assert all(e % 128 == 0 for e in end[:-1]) and all(a < b for a, b in zip([0, *end], end))


# MB of X and Y, the faster number of chunks (timed against each other): more where the way out waits for the way in
@pytest.mark.parametrize("x,y,n", [(9.4, 9.4, 4), (16.8, 21.0, 5), (8.4, 16.8, 8), (5.9, 14.8, 8), (14.4, 21.5, 8), (3.1, 10.6, 8), (8.4, 33.6, 5),
                                   (9.4, 37.7, 5), (4.2, 6.3, 4), (33.6, 67.1, 5)])
def test_the_faster_number_of_chunks(chunks, x, y, n):
    assert len(chunks(4096, 1e6 * x, 1e6 * y)) == min(n, chunks.most)
