"""Kernel attributes are set on every device that is used, not once a process
(host code only: the device is a stand-in)."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1702_03154_gb300", "csrc")

PROGRAM = r"""
#include <cuda_runtime.h>
static int device;
static cudaError_t stand_in(int *d) { *d = device; return cudaSuccess; }
#define cudaGetDevice stand_in
#include "common.cuh"
int main() {
  static bbh::DeviceOnce once;
  int ran[3] = {0, 0, 0}, fail = 1;
  auto set = [&] { ran[device]++; return fail ? 1 : 0; };
  if (bbh::once_per_device(once, set) != 1) return 1;  // a failure is not kept
  fail = 0;
  for (int round = 0; round < 3; round++)
    for (device = 0; device < 3; device++)
      if (bbh::once_per_device(once, set) != 0) return 2;
  return ran[0] == 2 && ran[1] == 1 && ran[2] == 1 ? 0 : 3;
}
"""


def test_once_on_each_device(tmp_path):
    from paper_1702_03154_gb300 import build_ext
    src, exe = tmp_path / "once.cu", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([build_ext.nvcc()] + build_ext.ARCH + build_ext.NVCC_FLAGS +
                   ["-I" + CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_attributes_are_set_through_it():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        if "cudaFuncSetAttribute" in text:
            assert "once_per_device" in text, path
            assert not re.search(r"static bool \w*attr", text), path
