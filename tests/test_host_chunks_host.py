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
extern "C" int chunks(int M, double bytes, int* out) {
  struct { int end[LQ_HOST_CHUNKS], guard[16]; } s;
  for (int& g : s.guard) g = -7;
  const int n = host_chunks(M, (size_t)bytes, s.end);
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
    lib.chunks.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_void_p]

    def get(M, bytes):
        out = (ctypes.c_int * 16)()
        n = lib.chunks(M, bytes, out)
        assert n >= 1, "written beyond the end"
        return list(out)[:n]

    get.most = request.param or 8
    return get


@pytest.mark.parametrize("bytes", [1e3, 2e7, 1e9])
def test_chunks_cover_the_rows(chunks, bytes):
    for M in [*range(1, 2600), 4096, 5001, 8192, 32768]:
        end = chunks(M, bytes)
        assert len(end) <= chunks.most and end[-1] == M
        assert all(e % 128 == 0 for e in end[:-1]) and all(a < b for a, b in zip([0, *end], end))
