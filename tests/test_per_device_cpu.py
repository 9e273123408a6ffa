"""Launch settings that belong to a device (csrc/per_device.h), on fakes of the CUDA runtime: a process that
uses a second device gets the opt-in to large dynamic shared memory and the cluster count of that device,
and a failed query is tried again."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2609_34077_gb300 import build

HARNESS = r"""
#include "per_device.h"
#include <cstdio>
static int dev = 0, sets[80][2], fail = 0, queries = 0;
static const char *ka = "a", *kb = "b";
extern "C" cudaError_t cudaGetDevice(int* d) { *d = dev; return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError(void) { return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* k, cudaFuncAttribute a, int v) {
  if (fail) return cudaErrorInvalidValue;
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize && v == 70000) ++sets[dev][k == kb];
  return cudaSuccess;
}
extern "C" cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  ++queries;
  if (fail) return cudaErrorInvalidValue;
  *n = int(c->gridDim.x) / 2 - dev;
  return cudaSuccess;
}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  static mcft::SmemOptIn a, b;
  static mcft::ResidentClusters r;
  fail = 1;
  CHECK(a.allow(ka, 70000) == cudaErrorInvalidValue && r.get(ka, 152, 320, 70000) == 0);
  fail = 0;
  for (int round = 0; round < 3; ++round)
    for (dev = 0; dev < 70; ++dev) {  // past the table too
      CHECK(a.allow(ka, 70000) == cudaSuccess && r.get(ka, 152, 320, 70000) == 76 - dev);
      if (dev % 2) CHECK(b.allow(kb, 70000) == cudaSuccess);
    }
  for (int d = 0; d < 70; ++d) {
    CHECK(sets[d][0] == (d < 64 ? 1 : 3));
    CHECK(sets[d][1] == (d % 2 == 0 ? 0 : d < 64 ? 1 : 3));
  }
  CHECK(queries == 1 + 64 + 3 * 6);
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_settings_of_every_device(tmp_path):
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    inc = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_launch_setting_goes_through_it():
    """No kernel file sets a function attribute or counts resident clusters by itself."""
    for f in sorted(os.listdir(build.CSRC)):
        if f != "per_device.h":
            text = open(os.path.join(build.CSRC, f)).read()
            assert not re.search(r"cudaFuncSetAttribute\s*\(|cudaOccupancyMaxActiveClusters\s*\(", text), f
