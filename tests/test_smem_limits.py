"""The kernels' limits of dynamic shared memory (csrc/qis_smem.cuh): a limit is kept per device, never
lowered by a smaller launch from another thread, taken up again after an error, and no launcher sets the
attribute past it."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_00180_gb300", "csrc")

HARNESS = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "qis_smem.cuh"

static std::atomic<long> real[2];   // the limit of the one kernel on two devices, as a driver holds it
static std::atomic<int> sets;
static qis::SmemLimits limits;
static char kernel;

static bool launch(int dev, long bytes) {   // ask, then launch as soon as others may have asked as well
  const int e = limits.raise(dev, &kernel, bytes, [&] {
    std::this_thread::sleep_for(std::chrono::microseconds(200));   // a slow driver call
    real[dev] = bytes;
    ++sets;
    return 0;
  });
  std::this_thread::sleep_for(std::chrono::microseconds(300));
  return e == 0 && real[dev] >= bytes;
}

int main() {
  std::atomic<int> bad{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 4; ++t)
    ts.emplace_back([&, t] {
      for (int k = 0; k < 200; ++k)
        if (!launch(t & 1, 50000 + 1000 * ((t * 7 + k * 3) % 40))) ++bad;
    });
  for (auto& t : ts) t.join();
  if (bad || sets > 80) return std::printf("%d launches above the limit, %d set\n", (int)bad, (int)sets), 1;
  // an error is passed on and the limit asked for again
  char other;
  if (limits.raise(0, &other, 60000, [] { return 7; }) != 7) return std::puts("error lost"), 1;
  int asked = 0;
  limits.raise(0, &other, 60000, [&] { return ++asked, 0; });
  limits.raise(0, &other, 60000, [&] { return ++asked, 0; });
  limits.raise(1, &other, 60000, [&] { return ++asked, 0; });
  return asked == 2 ? 0 : (std::printf("asked %d times\n", asked), 1);
}
"""


def test_limits_only_grow_and_are_per_device(tmp_path):
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_every_launcher_asks_through_the_limits():
    # (qis_noalloc.cu sets fixed sizes once per device, under its own lock)
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        calls = re.findall(r"cudaFuncSetAttribute\(\s*(\w+)", open(path).read())
        name = os.path.basename(path)
        if name == "qis_api.cu":
            assert calls == ["kernel"]
        elif name == "qis_noalloc.cu":
            assert set(calls) == {"k_na_fields", "k_na_select"}
        else:
            assert not calls, name
