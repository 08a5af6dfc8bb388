"""A device buffer whose allocation failed holds nothing (csrc/common.cuh, host
code compiled by nvcc with fakes of the library's allocation calls).

Callers grow scratch with `if (buf.n < need) alloc`; a buffer that kept the size it
had asked for would pass that test later with a NULL pointer.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
PROGRAM = r"""
#include <cstdio>
#include "common.cuh"
namespace krr {
static int g_fail = 0;
static char g_mem[64];
void set_error(const char *, ...) {}
cudaError_t pool_malloc(void **p, size_t, cudaStream_t) {
  if (g_fail) { *p = nullptr; return cudaErrorMemoryAllocation; }
  *p = g_mem;
  return cudaSuccess;
}
}
int main() {
  krr::DevBuf<double> b;
  krr::g_fail = 1;
  int bad = b.alloc(8, nullptr) != KRR_ENOMEM || b.n != 0 || b.p;
  krr::g_fail = 0;
  bad |= b.alloc(4, nullptr) != KRR_OK || b.n != 4 || !b.p;
  krr::g_fail = 1;
  bad |= b.alloc(8, nullptr) != KRR_ENOMEM || b.n != 0 || b.p;
  b.p = nullptr;
  return bad;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_failed_allocation_leaves_no_size(tmp_path):
    (tmp_path / "t.cu").write_text(PROGRAM)
    subprocess.run([NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    f"-I{ROOT}/include", f"-I{ROOT}/paper_2304_12465_gb300/csrc",
                    str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")], check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0
