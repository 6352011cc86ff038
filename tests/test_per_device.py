"""Kernel attributes are set on every device of the process, once each, from any
thread, and again after a failure (a second GPU that was never set up would refuse
the launch).  A fake runtime counts the calls; no GPU is used."""
import glob
import os

from _cxx import run_cxx

PROGRAM = r"""
#include "per_device.h"
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>

static thread_local int device = 0;
static std::atomic<int> sets[100];
static std::atomic<bool> broken{false};
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
  if (broken) return cudaErrorUnknown;
  ++sets[device];
  return cudaSuccess;
}
static void kernel_a(int) {}
static void kernel_b(int) {}

static cudaError_t launch_a() {
  static tn::PerDevice once;
  return tn::allow_smem(once, kernel_a, 100000);
}
static cudaError_t launch_b() {
  static tn::PerDevice once;
  return tn::allow_smem(once, kernel_b, 100000);
}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)

int main() {
  broken = true;
  CHECK(launch_a() == cudaErrorUnknown);
  broken = false;
  for (int d : {0, 1, 3}) {
    device = d;
    for (int i = 0; i < 3; ++i) CHECK(launch_a() == cudaSuccess);
    CHECK(sets[d] == 1);  // (on device 0 after the failure)
    CHECK(launch_b() == cudaSuccess && launch_b() == cudaSuccess);
    CHECK(sets[d] == 2);
  }
  device = 80;  // beyond the table: set by every call
  CHECK(launch_a() == cudaSuccess && launch_a() == cudaSuccess && sets[80] == 2);
  // threads that start together on a fresh device each return with it set
  std::vector<std::thread> ts;
  std::atomic<int> go{0}, bad{0};
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&] {
      device = 5;
      ++go;
      while (go < 8) {}
      if (launch_a() != cudaSuccess || sets[5] < 1) ++bad;
    });
  for (auto& t : ts) t.join();
  CHECK(bad == 0);
  return 0;
}
"""


def test_every_device_is_set_up_once(tmp_path):
    run_cxx(tmp_path, PROGRAM, link=False)


def test_launchers_set_attributes_that_way():
    from paper_2110_14502_gb300 import build as B
    for path in glob.glob(os.path.join(B.CSRC, "*")):
        with open(path) as f:
            if os.path.basename(path) != "per_device.h":
                assert "cudaFuncSetAttribute" not in f.read(), path
