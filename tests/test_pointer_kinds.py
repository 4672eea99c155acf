"""Which buffers the kernels use in place (csrc/acm_ptr.h), against a stand-in for the
runtime's pointer query: the current device's memory and managed memory only. Another
GPU's memory and host memory have to go through a copy. CPU only.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include "acm_ptr.h"
// pointer value: 1 + 10 * type + device; 0 mod 10 is a pointer the query refuses
extern "C" cudaError_t CUDARTAPI cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  const int v = (int)(intptr_t)p;
  if (v % 10 == 0) return cudaErrorInvalidValue;
  a->type = (cudaMemoryType)(v / 10);
  a->device = v % 10 - 1;
  return cudaSuccess;
}
static int cleared = 0;
extern "C" cudaError_t CUDARTAPI cudaGetLastError(void) { ++cleared; return cudaSuccess; }
static int q(int type, int owner, int dev) { return acm::on_device((void*)(intptr_t)(10 * type + owner + 1), dev); }
int main() {
  printf("%d %d %d %d %d %d %d", q(cudaMemoryTypeDevice, 0, 0), q(cudaMemoryTypeDevice, 1, 1),
         q(cudaMemoryTypeDevice, 1, 0), q(cudaMemoryTypeDevice, 0, 1), q(cudaMemoryTypeManaged, 0, 1),
         q(cudaMemoryTypeHost, 0, 0), q(cudaMemoryTypeUnregistered, 0, 0));
  const int bad = acm::on_device((void*)(intptr_t)20, 0);
  printf(" %d %d\n", bad, cleared);
  return 0;
}
"""


def test_only_the_current_devices_memory_is_used_in_place(tmp_path):
    from paper_2312_15554_gb300 import build
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        inc = "/usr/local/cuda/include"
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-I", os.path.join(build.CSRC), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    #              own own other other managed host unregistered | refused, error cleared
    assert out == ["1", "1", "0", "0", "1", "0", "0", "0", "1"]


def test_every_entry_point_asks_the_same_question():
    """The contexts' and the context-free transform share the one test of a buffer's device."""
    for f in ("acm_api.cu", "acm_static.cu"):
        s = open(os.path.join(ROOT, "paper_2312_15554_gb300", "csrc", f)).read()
        assert "on_device(" in s and "cudaPointerGetAttributes" not in s, f
