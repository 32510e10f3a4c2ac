"""What the library does once per device (kernel attributes), on devices that a fake runtime call names."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "device_once.h"
#include <cstdio>
#include <thread>
#include <vector>
static thread_local int g_dev = 0;
extern "C" cudaError_t CUDARTAPI cudaGetDevice(int *d) { *d = g_dev; return g_dev < 0 ? cudaErrorInvalidDevice : cudaSuccess; }
static int calls[64], other;
static void use(int dev) {
  static jolt::DeviceOnce once;
  g_dev = dev;
  once([&] { if (dev >= 0 && dev < 64) ++calls[dev]; else ++other; });
}
int main() {
  for (int round = 0; round < 3; ++round) for (int d : {0, 1, 7, 63}) use(d);
  std::vector<std::thread> ts;
  for (int i = 0; i < 8; ++i) ts.emplace_back([] { use(5); });
  for (auto &t : ts) t.join();
  use(64); use(64); use(-1);
  int total = 0;
  for (int c : calls) total += c;
  std::printf("%d %d %d %d %d %d %d\n", calls[0], calls[1], calls[7], calls[63], calls[5], total, other);
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2607_12550_b200", "csrc"), "-I", os.path.join(cuda, "include"),
                    str(src), "-o", str(exe)], check=True)
    # once on each of five devices; where the device is unknown there is nothing to remember it by
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["1", "1", "1", "1", "1", "5", "3"]


def test_kernel_attributes_are_set_per_device():
    csrc = os.path.join(ROOT, "paper_2607_12550_b200", "csrc")
    for name in os.listdir(csrc):
        text = open(os.path.join(csrc, name)).read()
        if "cudaFuncSetAttribute(" in text and name != "cluster_jacobi.cuh":        # (its helper is called under a DeviceOnce)
            assert "DeviceOnce" in text and "static bool attr" not in text and "static size_t attr" not in text, name
