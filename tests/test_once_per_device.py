"""Kernel attributes belong to a device: they are set once on each, and again where
that failed."""
import subprocess

from paper_2608_06291_gb300 import buildlib

ONCE = r"""
#include "common.cuh"
using namespace bakron;
int main() {
  static OncePerDevice once;
  int calls = 0;
  cudaError_t result = cudaErrorInvalidValue;
  auto set = [&] { ++calls; return result; };
  if (once.on(0, set) != cudaErrorInvalidValue || calls != 1) return 1;
  result = cudaSuccess;
  if (once.on(0, set) != cudaSuccess || calls != 2) return 2;   // again after a failure
  if (once.on(0, set) != cudaSuccess || calls != 2) return 3;   // once
  if (once.on(1, set) != cudaSuccess || calls != 3) return 4;   // another device
  if (once.on(0, set) != cudaSuccess || once.on(1, set) != cudaSuccess || calls != 3) return 5;
  if (once.on(1000, set) != cudaSuccess || once.on(1000, set) != cudaSuccess || calls != 5) return 6;
  return 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cu", tmp_path / "once"
    src.write_text(ONCE)
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, "-std=c++17", "-I", buildlib.CSRC, "-I", buildlib.INCLUDE,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_attribute_is_set_once_per_process():
    """Every cudaFuncSetAttribute of the library's own kernels goes through it."""
    import glob
    import re
    for path in glob.glob(buildlib.CSRC + "/*.cu"):
        with open(path) as f:
            text = f.read()
        if "cudaFuncSetAttribute(" in text and not path.endswith("mma_rate.cu"):   # that one sets it on each call
            assert "OncePerDevice" in text, path
            assert not re.search(r"static bool (?:\w+_)?done = false|bool g_attr_done", text), path
