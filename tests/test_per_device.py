"""A process that works on a second device: kernel attributes and occupancies are
asked for on each device once (per_device.cuh compiled for the host against a
counting stand-in for the runtime), and no launcher keeps one answer for the
whole process."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_03563_gb300", "csrc")

PROGRAM = r"""
#include "per_device.cuh"
#include <cstdio>
static int device = 0, opted[70], asked[70];
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return device < 0 ? cudaErrorNoDevice : cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v) { opted[device] += v; return cudaSuccess; }
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  asked[device]++;
  *n = device + 1;
  return cudaSuccess;
}
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* k, int t, size_t s, unsigned) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k, t, s);
}
static void kernel() {}
int main() {
  static ps::PerDevice cached;
  for (int round = 0; round < 3; round++)
    for (int d : {0, 1, 63, 65}) {   // past the kept ones the question is repeated
      device = d;
      int n = 0;
      if (ps::resident_blocks(kernel, 256, 1000, cached, &n) != cudaSuccess || n != d + 1) return 1;
    }
  for (int d : {0, 1, 63})
    if (opted[d] != 1000 || asked[d] != 1) return 2;
  if (opted[65] != 3000 || asked[65] != 3) return 3;
  int n = 7;
  device = -1;
  if (ps::resident_blocks(kernel, 256, 1000, cached, &n) == cudaSuccess || n != 7) return 4;
  std::printf("ok\n");
  return 0;
}
"""


def test_each_device_is_asked_once(tmp_path):
    from paper_2605_03563_gb300.build import nvcc
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-I", include, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "ok\n"


def test_no_launcher_keeps_an_answer_for_the_process():
    kept = re.compile(r"static\s+(?:std::atomic<int>|int|size_t|bool)\s+\w+\s*(?:=|\{|;)")
    for f in sorted(os.listdir(CSRC)):
        code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        assert not kept.findall(code), f
