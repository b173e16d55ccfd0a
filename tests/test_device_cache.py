"""What the library remembers per device is asked for on every device.

A process may hold graphs on several devices.  Launch shapes are asked for once per device, and a kernel
whose shared memory exceeds the default needs its attribute set on each of them; otherwise its launch is
refused there.  The CUDA calls are replaced by fakes of two devices that differ, so no GPU is needed.
"""
from __future__ import annotations

import os
import subprocess

import pytest

_FAKES = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <set>

static int g_device = 0, g_occupancy_calls = 0;
static std::set<int> g_opted_in;  // devices whose attribute was set
static const int kSms[3] = {152, 100, 7};
static cudaError_t fake_get_device(int *d) { *d = g_device; return cudaSuccess; }
static cudaError_t fake_attribute(int *v, cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? kSms[d % 3] : 1;
  return cudaSuccess;
}
template <typename F> static cudaError_t fake_func_attribute(F, cudaFuncAttribute, int) {
  g_opted_in.insert(g_device);
  return cudaSuccess;
}
template <typename F> static cudaError_t fake_occupancy(int *n, F, int, size_t smem) {
  ++g_occupancy_calls;
  *n = smem <= 48 * 1024 || g_opted_in.count(g_device) ? 2 : 0;
  return cudaSuccess;
}
#define cudaGetDevice fake_get_device
#define cudaDeviceGetAttribute fake_attribute
#define cudaFuncSetAttribute fake_func_attribute
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake_occupancy
"""

_MAIN = {
    "hm_levels.cu": r"""
namespace hm { int num_sms() { return kSms[g_device % 3]; } uint64_t budget_ms() { return 1; } int32_t filter_min() { return 1; } }
int main() {
  static_assert(sizeof(hm::LvShared) > 48 * 1024, "needs the attribute");
  int bad = 0;
  for (int rep = 0; rep < 2; ++rep)
    for (int d : {0, 1, 2, 0, 200}) {
      g_device = d;
      const int got = hm::lv_grid(hm::lv_kernel(true, false, false), 4);
      if (got != 2 * kSms[d % 3]) bad += std::printf("device %d: grid %d\n", d, got);
      if (!g_opted_in.count(d)) bad += std::printf("device %d: attribute not set\n", d);
    }
  if (g_occupancy_calls > 3 + 2) bad += std::printf("asked %d times\n", g_occupancy_calls);
  std::puts(bad ? "bad" : "ok");
  return bad != 0;
}
""",
    "hm_sort.cu": r"""
int main() {
  int bad = 0;
  for (int d : {0, 1, 2, 0, 200, 1}) {
    g_device = d;
    if (hm::num_sms() != kSms[d % 3]) bad += std::printf("device %d: %d SMs\n", d, hm::num_sms());
  }
  std::puts(bad ? "bad" : "ok");
  return bad != 0;
}
""",
}


@pytest.mark.parametrize("unit", sorted(_MAIN))
def test_launch_shapes_are_per_device(unit, tmp_path):
    from paper_2507_04130_gb300 import _build

    src = tmp_path / "harness.cu"
    src.write_text(f'{_FAKES}\n#include "{unit}"\n{_MAIN[unit]}')
    exe = str(tmp_path / "harness")
    made = subprocess.run([_build._nvcc(), *_build.ARCH, "-O0", "-std=c++17", f"-I{_build.INCLUDE}", f"-I{_build.CSRC}",
                           str(src), "-o", exe], capture_output=True, text=True)
    assert made.returncode == 0, made.stderr
    ran = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert ran.returncode == 0 and ran.stdout.strip() == "ok", ran.stdout + ran.stderr
