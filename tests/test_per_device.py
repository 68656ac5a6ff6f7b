"""Per-device set-up: an error stays with the device it was met on, and each device is set up once, from any thread."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <atomic>
#include <thread>
#include <vector>
#include "per_device.cuh"

int main() {
  static qc::PerDevice<int> attrs;
  std::atomic<int> calls[8] = {};
  std::atomic<int> wrong{0};
  std::vector<std::thread> threads;
  for (int t = 0; t < 32; ++t)
    threads.emplace_back([&, t] {
      const int device = t % 8;
      for (int i = 0; i < 100; ++i)
        if (attrs.once(device, [&] { ++calls[device]; return device == 3 ? 7 : 0; }) != (device == 3 ? 7 : 0)) ++wrong;
    });
  for (auto& t : threads) t.join();
  for (auto& c : calls) wrong += c != 1;
  return wrong;
}
"""


def test_an_error_stays_with_its_device(tmp_path):
    source, binary = tmp_path / "per_device.cpp", tmp_path / "per_device"
    source.write_text(PROGRAM)
    include = os.path.join(ROOT, "paper_1805_07941_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-x", "c++", "-I", include, "-o", str(binary), str(source)], check=True)
    assert subprocess.run([str(binary)], timeout=60).returncode == 0


def test_the_library_keeps_no_error_for_all_devices():
    """Every function attribute goes through it: no error variable that outlives a call is shared by the devices."""
    text = open(os.path.join(ROOT, "paper_1805_07941_b200", "csrc", "qconv_api.cu")).read()
    assert "static cudaError_t" not in text
