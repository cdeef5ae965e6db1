"""State made once per device (csrc/per_device.h), compiled for the host with
g++ (no GPU): with several threads on several devices every device's value is
made exactly once and every caller gets its own device's; a make that throws
is tried again.  And no kernel attribute or device property is remembered any
other way: a flag set once per process leaves the second device of a process
without the shared memory that its kernels ask for."""
import ctypes
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2208_06191_gb300", "csrc")

WRAPPER = r"""
#include "per_device.h"
#include <atomic>
#include <stdexcept>
#include <thread>
#include <vector>
extern "C" int made_once(int devices, int threads, int calls) {
  cbddc::PerDevice<int> state;
  std::vector<std::atomic<int>> made(devices);
  std::atomic<int> wrong{0};
  std::vector<std::thread> pool;
  for (int t = 0; t < threads; ++t)
    pool.emplace_back([&, t] {
      for (int i = 0; i < calls; ++i) {
        const int dev = (i + t) % devices;
        if (state.get(dev, [&] { ++made[dev]; return 100 + dev; }) != 100 + dev) ++wrong;
      }
    });
  for (auto& th : pool) th.join();
  for (auto& m : made)
    if (m != 1) ++wrong;
  return wrong;
}
extern "C" int made_again_after_a_throw() {
  cbddc::PerDevice<bool> state;
  int tries = 0;
  for (int i = 0; i < 3; ++i) {
    try {
      state.get(1, [&]() -> bool {
        if (++tries == 1) throw std::runtime_error("no");
        return true;
      });
    } catch (const std::runtime_error&) {
    }
  }
  return tries;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("per_device")
    src = d / "wrap.cpp"
    src.write_text(WRAPPER)
    so = d / "libper_device.so"
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("devices,threads", [(1, 1), (1, 8), (2, 2), (8, 8)])
def test_made_once_per_device(lib, devices, threads):
    assert lib.made_once(devices, threads, 2000) == 0


def test_made_again_after_a_throw(lib):
    assert lib.made_again_after_a_throw() == 2


def test_nothing_is_remembered_per_process():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        # a mutable flag or number of the process, set at its first use
        assert not re.search(r"static\s+(bool|int)\s+\w+\s*=", text), name
        for m in re.finditer("cudaFuncSetAttribute", text):
            assert "PerDevice" in text[:m.start()].rsplit("template", 1)[-1], name
