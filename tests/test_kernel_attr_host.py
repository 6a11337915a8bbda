"""CPU checks of the per-device launch state (csrc/kernel_attr.cuh), compiled as
host code against a fake CUDA runtime with two devices: a kernel's
shared-memory limit is raised on each device that launches it, from any host
thread, and a failed call is not remembered as done."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_05900_gb300", "csrc")

FAKE = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "kernel_attr.cuh"
static thread_local int dev = 0;
static std::atomic<int> sets[2], asks[2];
static bool fail = false;
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = dev; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) {
  if (fail) return cudaErrorInvalidValue;
  ++sets[dev];
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int d) { ++asks[d]; *v = 100 + d; return cudaSuccess; }
}
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
using namespace hotrg;
int main() {
  SmemLimit limit, other;
  fail = true;
  CHECK(limit.raise(nullptr, 1) == cudaErrorInvalidValue);
  fail = false;
  CHECK(limit.raise(nullptr, 1) == cudaSuccess && sets[0] == 1 && sets[1] == 0);
  CHECK(limit.raise(nullptr, 1) == cudaSuccess && sets[0] == 1);
  CHECK(sm_count() == 100 && sm_count() == 100 && asks[0] == 1);
  dev = 1;                                     // a second device gets its own
  CHECK(limit.raise(nullptr, 1) == cudaSuccess && sets[0] == 1 && sets[1] == 1);
  CHECK(sm_count() == 101 && asks[1] == 1);
  CHECK(other.raise(nullptr, 1) == cudaSuccess && sets[1] == 2);
  SmemLimit shared;
  std::atomic<int> bad{0};
  std::vector<std::thread> th;
  for (int t = 0; t < 8; ++t)
    th.emplace_back([&, t] {
      dev = t & 1;
      for (int i = 0; i < 1000; ++i)
        if (shared.raise(nullptr, 1) != cudaSuccess || sm_count() != 100 + dev) ++bad;
    });
  for (auto &t : th) t.join();
  CHECK(bad == 0 && sets[0] >= 2 && sets[1] >= 3);
  printf("ATTR_OK\n");
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_limits_belong_to_the_device(tmp_path):
    from paper_2602_05900_gb300.build import _cuda_home
    src, exe = tmp_path / "fake.cc", tmp_path / "fake"
    src.write_text(FAKE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(_cuda_home(), "include"), str(src),
                    "-o", str(exe), "-pthread"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "ATTR_OK" in r.stdout, r.stdout


def test_launchers_keep_no_state_of_their_own():
    """No launcher remembers per process what belongs to a device."""
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        if f != "kernel_attr.cuh":
            assert "cudaFuncSetAttribute" not in text and "cudaDevAttrMultiProcessorCount" not in text, f
