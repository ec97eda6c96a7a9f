"""The buffers of Lorentz-Berthelot evaluations when an allocation fails: none
is kept, so that the next call allocates all of them instead of handing null
pointers to the kernels.  Runs on the CPU: the allocator is the test's own."""
import os
import shutil
import subprocess

import pytest

from paper_1308_4005_gb300 import build as B

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "mls6_internal.h"

int main(int, char** argv) {
  const bool spectral = atoi(argv[1]);
  for (int fail = 1; fail <= 5; ++fail) {  // the failing allocation
    mls6::Plan p;
    p.N = 10;
    p.prec = MLS6_FP32;
    p.spectral = spectral;
    p.lv[1].n[0] = 8; p.lv[1].n[1] = 6; p.lv[1].n[2] = 4;
    p.lv[1].np = 192;
    std::map<void*, size_t> live;
    int count = 0;
    auto alloc = [&](void** q, size_t b) {
      if (++count == fail) { *q = (void*)0x10; return false; }  // what a failure leaves is not read
      *q = malloc(b);
      live[*q] = b;
      return true;
    };
    auto release = [&](void* q) {
      if (!live.erase(q)) printf("released twice or never allocated\n");
      free(q);
    };
    const bool first = mls6::lb_workspace(&p, alloc, release);
    const int need = spectral ? 4 : 2;
    if (first != (fail > need)) printf("first %d fail %d\n", first, fail);
    if (!first && (!live.empty() || p.d_lbw || p.d_lbpot || p.d_lbq || p.d_lbs))
      printf("kept %zu fail %d\n", live.size(), fail);
    if (!mls6::lb_workspace(&p, alloc, release)) printf("second fail %d\n", fail);
    if ((int)live.size() != need || live[p.d_lbw] != 4 * 10 || live[p.d_lbpot] != 4 * 7 * 192 ||
        (spectral && (live[p.d_lbq] != 4 * 7 * 192 || live[p.d_lbs] != 2 * 8 * 7 * 6 * 5 * 4)))
      printf("sizes, fail %d\n", fail);
  }
  printf("done\n");
}
"""


@pytest.mark.parametrize("spectral", [0, 1])
def test_lb_workspace_is_all_or_nothing(tmp_path, spectral):
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc())))
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    exe = str(tmp_path / "t")
    inc = [os.path.join(cuda, "include"), B.CSRC]
    subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-O1", str(src), "-o", exe] +
                   [v for i in inc for v in ("-I", i)], check=True)
    out = subprocess.run([exe, str(spectral)], capture_output=True, text=True, check=True).stdout
    assert out == "done\n"
