"""Kernel attributes are set on every device that launches the kernel: they
belong to the device that is current when they are set, so a process-wide
"once" leaves a second device without them."""
import os
import re
import subprocess

from test_pdl_sources import CSRC, sources


def process_wide(text):
    """Initialisers of function-local statics that set a kernel attribute (they
    run once per process)."""
    out = []
    for m in re.finditer(r"static\s+(?:const\s+)?\w+\s+\w+\s*=\s*\[", text):
        end = text.find("}();", m.end())
        if "cudaFuncSetAttribute" in text[m.end():end]:
            out.append(text[m.start():m.end()])
    return out


def test_no_kernel_attribute_is_set_once_per_process():
    text = sources()
    assert "cudaFuncSetAttribute" in text
    assert process_wide(text) == []
    assert process_wide("static const bool once = [] { cudaFuncSetAttribute(k, a, 1); "
                        "return true; }();")


MAIN = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "dp_device.h"
static thread_local int dev = 0;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = dev; return cudaSuccess; }
int main() {
  static dp::PerDevice per;
  std::atomic<int> calls[3] = {{0}, {0}, {0}};
  auto use = [&](int d) { dev = d; return per([&] { ++calls[d]; return 10 * d; }); };
  std::vector<std::thread> t;
  std::atomic<int> bad{0};
  for (int k = 0; k < 12; ++k)
    t.emplace_back([&, k] { for (int r = 0; r < 100; ++r) if (use(k % 3) != 10 * (k % 3)) ++bad; });
  for (auto &h : t) h.join();
  static dp::PerDevice fails;
  int tries = 0;
  dev = 0;
  int a = fails([&] { ++tries; return -3; }), b = fails([&] { ++tries; return 5; });
  int c = fails([&] { ++tries; return 6; });
  std::printf("%d %d %d %d %d %d %d %d\n", (int)bad, (int)calls[0], (int)calls[1], (int)calls[2], a, b,
              c, tries);
}
"""


def test_once_on_each_device(tmp_path):
    """Twelve threads on three (faked) devices: one call a device, its value to
    every thread; a failure is tried again."""
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(MAIN)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-I", f"{cuda}/include",
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert out.split() == ["0", "1", "1", "1", "-3", "5", "5", "2"]
