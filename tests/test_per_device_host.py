"""What a launcher sets once (function attributes) belongs to the device it was set on: per_device.h against a fake of
cudaGetDevice, and no launcher that keeps a flag for the whole process instead.  No GPU."""
import os
import re
import shutil
import subprocess

import pytest

from paper_1312_1476_gb300 import _build

SOURCE = r"""
#include <cassert>
#include <cstdio>
#include "per_device.h"

static int device = 0;
static cudaError_t lookup = cudaSuccess;
extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* d) {
  *d = device;
  return lookup;
}

int main() {
  static gmrf::PerDevice value;
  int calls = 0, v = 0;
  auto form = [&](int* r) {
    ++calls;
    *r = 100 + device;
    return cudaSuccess;
  };
  for (int round = 0; round < 3; ++round)
    for (device = 0; device < 3; ++device) assert(value.get(form, &v) == cudaSuccess && v == 100 + device);
  assert(calls == 3);  // once for each of the three
  device = 3;          // a failure is reported, not kept
  auto fails = [&](int*) { return cudaErrorInvalidValue; };
  assert(value.get(fails, &v) == cudaErrorInvalidValue);
  assert(value.get(form, &v) == cudaSuccess && v == 103 && calls == 4);
  device = 1000;  // beyond the table: formed each time
  assert(value.get(form, &v) == cudaSuccess && value.get(form) == cudaSuccess && v == 1100 && calls == 6);
  lookup = cudaErrorInitializationError;
  assert(value.get(form, &v) == cudaErrorInitializationError && calls == 6);
  std::puts("ok");
}
"""


def test_formed_once_per_device(tmp_path):
    nvcc = shutil.which(_build._nvcc())
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I", cuda, "-I", _build.CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "ok\n"


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(_build.CSRC) if f.endswith((".cu", ".cuh", ".h"))))
def test_no_attribute_behind_a_flag_of_the_process(name):
    with open(os.path.join(_build.CSRC, name)) as f:
        text = f.read()
    for m in re.finditer(r"cudaFuncSetAttribute|cudaOccupancy|set_attribute\(", text):
        before = text[max(0, m.start() - 700):m.start()]
        assert not re.search(r"static\s+(std::)?(atomic<bool>|once_flag|const size_t lim)", before), name
