"""Which systems take the cluster kernel of the PCG's vector half: by size, preconditioner and storage,
not in a crowded batch, and never where the device has no room for such a cluster (here: no device).
"""
import os
import shutil
import subprocess

import pytest

from paper_2405_03584_gb300 import build

SRC = r"""
#include <cstdio>
#include "state.h"
using namespace ipmk;
static int bad = 0;
static void check(bool got, bool want, const char* what) {
  if (got != want) { std::printf("%s: %d\n", what, (int)got); bad = 1; }
}
static Dev dev(int64_t n, int64_t m, int storage) {
  Dev d{};
  d.n = d.nsys = n; d.m = m; d.storage = storage; d.sm_count = 152; d.cluster = 1;
  return d;
}
int main() {
  const int64_t last = 57344, plain = 16384;
  for (int64_t n : {(int64_t)1, (int64_t)512, (int64_t)513, plain, plain + 1, last, last + 1})
    for (int storage : {ST_F64, ST_F32, ST_BF16, ST_FP8})
      for (int64_t m : {0, 10})
        for (int pc : {PC_JACOBI, PC_JACOBI_LR, PC_DENSE, PC_BLOCK32}) {
          Dev d = dev(n, m, storage);
          const bool lr = pc == PC_JACOBI_LR && m > 0;
          const bool takes = pc <= PC_JACOBI_LR && n <= (lr || storage != ST_F64 ? last : plain);
          check(tail_runs(d, pc), takes, "takes");
          d.crowd = 1;
          check(tail_runs(d, pc), false, "crowded");
          d.aug = 1;
          check(tail_runs(d, pc), takes, "crowded, augmented");
          d.cluster = 0;
          check(tail_runs(d, pc), false, "no room, augmented");
          d = dev(n, m, storage);
          d.cluster = 0;
          check(tail_runs(d, pc), false, "no room");
        }
  int devices = 0;
  if (cudaGetDeviceCount(&devices) != cudaSuccess || devices == 0) {
    cudaGetLastError();
    check(tail_places(dev(1000, 10, ST_F32), PC_JACOBI_LR), false, "places without a device");
  }
  return bad;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_tail_rule(tmp_path):
    lib = build.build()
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(SRC)
    r = subprocess.run([shutil.which("nvcc"), *build.ARCH, *build.FLAGS, "-I" + build.CSRC, str(src), "-o", str(exe), lib,
                        "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[:2000]
