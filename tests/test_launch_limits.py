"""What launchers remember of a kernel (csrc/mbo_limits.h) is kept per device, and a
shared-memory limit only grows, whatever the order in which host threads ask."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cassert>
#include <cstdio>
#include <thread>
#include <vector>
#include "mbo_limits.h"
using namespace mbo;
int main() {
  {  // each device has a limit of its own, and a failed call is not remembered
    SmemLimit l;
    int calls = 0;
    auto ok = [&](size_t) { ++calls; return 0; };
    assert(l.raise(0, 48 * 1024, ok) == 0 && calls == 0);
    assert(l.raise(0, 100000, ok) == 0 && calls == 1);
    assert(l.raise(0, 90000, ok) == 0 && calls == 1);
    assert(l.raise(1, 90000, ok) == 0 && calls == 2);
    assert(l.raise(1, 100000, [](size_t) { return 7; }) == 7);
    assert(l.raise(1, 100000, ok) == 0 && calls == 3);
    assert(l.raise(kLimitDevices, 90000, ok) == 0 && calls == 4);
  }
  for (int round = 0; round < 200; ++round) {  // never lowered between a call and the launch after it
    SmemLimit l;
    std::atomic<size_t> device{0};
    std::atomic<bool> low{false};
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i)
      t.emplace_back([&, i] {
        const size_t want = 50000 + 1000 * (size_t)((i * 5 + round) % 8);
        l.raise(0, want, [&](size_t b) {
          std::this_thread::yield();
          device = b;
          return 0;
        });
        std::this_thread::yield();
        if (device < want) low = true;
      });
    for (auto& x : t) x.join();
    assert(!low && device == 57000);
  }
  DeviceCount c;
  int asked = 0;
  auto ask = [&] { return ++asked * 10; };
  assert(c.get(0, ask) == 10 && c.get(1, ask) == 20 && c.get(0, ask) == 10 && asked == 2);
  std::puts("ok");
}
"""


def test_limits_per_device_and_growing(tmp_path):
    src = tmp_path / "limits.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "limits"
    inc = os.path.join(ROOT, "paper_1711_01365_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-UNDEBUG", "-I", inc, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60)
    assert out.stdout.strip() == "ok"
