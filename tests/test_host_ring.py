"""Page-locked memory of the Krylov solves (krylov.hpp), compiled for the host
with fakes of the runtime calls: kernels that an error leaves in flight may
still write it, so the stream is waited for before it is freed."""
import os
import shutil
import subprocess

import pytest

from paper_2507_17053_gb300 import _build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <string>
#include "krylov.hpp"
static std::string calls;
static int events_left = 1 << 30;
extern "C" {
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::malloc(n); calls += "m"; return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); calls += "f"; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  if (events_left-- <= 0) return cudaErrorMemoryAllocation;
  *e = (cudaEvent_t)&calls;
  calls += "e";
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { calls += "d"; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { calls += s == (cudaStream_t)8 ? "S" : "?"; return cudaSuccess; }
}
static int check(const char* want) {
  if (calls != want) std::printf("%s, not %s\n", calls.c_str(), want);
  const int bad = calls != want;
  calls.clear();
  return bad;
}
int main() {
  int bad = 0;
  { sbm::HostRing r((cudaStream_t)8); bad |= r.init(64, 3) != cudaSuccess; }
  bad |= check("meeeSdddf");
  events_left = 1;
  { sbm::HostRing r((cudaStream_t)8); bad |= r.init(64, 3) == cudaSuccess; }
  bad |= check("meSdf");
  { sbm::HostRing r((cudaStream_t)8); }
  bad |= check("");
  return bad;
}
"""


def test_freed_only_after_the_stream(tmp_path):
    try:
        cuda = os.path.join(os.path.dirname(_build._nvcc()), "..", "include")
    except RuntimeError:
        pytest.skip("no CUDA headers")
    src = tmp_path / "ring.cpp"
    src.write_text(SRC)
    exe = str(tmp_path / "ring")
    subprocess.run([shutil.which("g++"), "-std=c++17", f"-I{_build.CSRC}", f"-I{_build.INCLUDE}",
                    f"-I{cuda}", str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
