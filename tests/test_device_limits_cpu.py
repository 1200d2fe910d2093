"""Launch limits per device (csrc/device_limits.cu, host code) against a fake
CUDA runtime with three devices: a second device gets its own limits and
occupancies, values are looked up once per device, limits are never lowered and
a failed lookup is tried again."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1504_02891_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <utility>
#include "device_limits.h"

static int device, fail_next, set_calls, occ_calls;
static std::map<std::pair<int, const void*>, int> limit;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { *v = 100 + d; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  ++set_calls;
  if (fail_next) { --fail_next; return cudaErrorInvalidValue; }
  limit[{device, f}] = v;
  return cudaSuccess;
}
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int, size_t smem) {
  ++occ_calls;
  if ((size_t)limit[{device, f}] < smem) return cudaErrorInvalidValue;   // as a launch would
  *n = smem > 90000 ? 0 : 2 + device;
  return cudaSuccess;
}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
using namespace gpe;
int main() {
  int a, b, occ = 0;   // two kernels' addresses: &a, &b
  static KernelShape small, large;
  fail_next = 1;
  CHECK(kernel_shape(small, &a, 64, 50000, &occ) == cudaErrorInvalidValue);
  CHECK(kernel_shape(small, &a, 64, 50000, &occ) == cudaSuccess && occ == 2);   // not kept as failed
  for (int turn = 0; turn < 2; ++turn)
    for (device = 0; device < 3; ++device) {
      CHECK(kernel_shape(small, &a, 64, 50000, &occ) == cudaSuccess && occ == 2 + device);
      CHECK(limit[std::make_pair(device, (const void*)&a)] >= 50000);
      CHECK(kernel_shape(large, &a, 64, 70000, &occ) == cudaSuccess && occ == 2 + device);
      CHECK(limit[std::make_pair(device, (const void*)&a)] == 70000);
      CHECK(num_sms() == 100 + device);
    }
  CHECK(set_calls == 1 + 6 && occ_calls == 6);
  device = 1;
  CHECK(raise_smem(&a, 60000) == cudaSuccess && limit[std::make_pair(1, (const void*)&a)] == 70000);   // not lowered
  CHECK(raise_smem(&b, 40000) == cudaSuccess && limit[std::make_pair(1, (const void*)&b)] == 40000);
  static KernelShape none;
  CHECK(kernel_shape(none, &b, 64, 99000, &occ) == cudaSuccess && occ == 1);    // at least one
  device = MAX_DEVICES + 3;                                                     // beyond the table: not kept
  const int before = occ_calls;
  CHECK(kernel_shape(small, &a, 64, 50000, &occ) == cudaSuccess && occ == 2 + device);
  CHECK(kernel_shape(small, &a, 64, 50000, &occ) == cudaSuccess && occ_calls == before + 2);
  CHECK(num_sms() == 100 + device);
  printf("ok\n");
  return 0;
}
"""


def _include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_limits_belong_to_a_device(tmp_path):
    src = tmp_path / "main.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "main"
    inc = [i for i in (_include(), "/usr/local/cuda/include") if os.path.isdir(i)]
    cmd = ["g++", "-std=c++17", *[f"-I{i}" for i in inc], f"-I{CSRC}", str(src), "-x", "c++",
           os.path.join(CSRC, "device_limits.cu"), "-o", str(exe), "-pthread"]
    subprocess.run(cmd, check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "ok\n"


def test_launchers_keep_nothing_per_process():
    """No launcher keeps an occupancy, a limit or an error in a static of its own."""
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f), encoding="utf-8").read())
        for m in re.finditer(r"\bstatic\s+(?:const\s+)?(cudaError_t|size_t|int)\s+(\w+)\s*=[^;]*;", text):
            assert not re.search(r"occ|allowed|smem|raise_smem|nsm|sms", m.group(0)), (f, m.group(0))
        assert not re.search(r"\bstatic const KernelShape\b", text), f
