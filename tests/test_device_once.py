"""Work done once per device (the Schwarz kernels' shared-memory limits): a
second device gets its own, a failure is not kept, threads do it once; and the
limits are not kept by anything that forgets the device. The header is plain
C++ and runs here without a GPU."""
import glob
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_07041_gb300", "csrc")

PROGRAM = r'''
#include "dd_device_once.cuh"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  dd::DeviceOnce once;
  int calls[3] = {0, 0, 0};
  auto on = [&](int dev, int rc) { return once.run(dev, [&] { calls[dev]++; return rc; }); };
  if (on(0, 0) || on(0, 0) || calls[0] != 1) return 1;
  if (on(1, 0) || calls[1] != 1) return 2;                    // another device: its own
  if (on(2, 7) != 7 || on(2, 0) || on(2, 7) || calls[2] != 2) return 3;   // a failure is tried again, a success kept
  dd::DeviceOnce shared;
  std::atomic<int> n{0};
  std::vector<std::thread> t;
  for (int i = 0; i < 16; i++) t.emplace_back([&, i] { shared.run(i % 2, [&] { n++; return 0; }); });
  for (auto &x : t) x.join();
  return n == 2 ? 0 : 4;
}
'''


def test_device_once(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_limits_are_kept_per_device():
    """The Schwarz sources keep no once-flag or limit of their own."""
    for path in glob.glob(os.path.join(CSRC, "dd_sap*")):
        text = open(path).read()
        assert "once_flag" not in text and "static int raised" not in text, path
