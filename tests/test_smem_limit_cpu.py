"""A kernel's shared-memory limit is raised by every handle that needs more,
and handles may be created in several threads: whatever the order in which
threads read and set it, the largest need stays.  smem_limit.cuh is compiled
with the host compiler, the driver's two calls replaced by ones that take
long enough for every thread to get in between."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_04579_gb300", "csrc")
SHIM = r"""
#include <atomic>
#include <chrono>
#include <thread>
#include <vector>
#include "smem_limit.cuh"
// count threads raise one limit to needs[i]; error: what set() returns for a need above 227 KB
extern "C" int raise_all(const int* needs, int count, int* results) {
  std::atomic<int> limit{0}, sets{0};
  std::vector<std::thread> ts;
  for (int i = 0; i < count; ++i)
    ts.emplace_back([&, i] {
      results[i] = gnm::raise_limit(
          [&](int* c) {
            *c = limit;
            std::this_thread::sleep_for(std::chrono::milliseconds(5));
            return 0;
          },
          [&](int v) {
            std::this_thread::sleep_for(std::chrono::milliseconds(v % 7));
            ++sets;
            if (v > 232448) return 1;
            limit = v;
            return 0;
          },
          needs[i]);
    });
  for (auto& t : ts) t.join();
  return limit;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("smem_limit")
    src, out = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(out)],
                   check=True)
    return ctypes.CDLL(str(out))


def run(lib, needs):
    a, r = (ctypes.c_int * len(needs))(*needs), (ctypes.c_int * len(needs))()
    return lib.raise_all(a, len(needs), r), list(r)


@pytest.mark.parametrize("needs", [[100000, 200000], [200000, 100000], list(range(50000, 66000, 1000)),
                                   list(range(66000, 50000, -1000)), [49152] * 8])
def test_the_largest_need_stays(lib, needs):
    for _ in range(3):
        assert run(lib, needs) == (max(needs), [0] * len(needs))


def test_too_much_is_still_an_error_and_changes_nothing(lib):
    limit, results = run(lib, [100000, 300000, 200000])
    assert limit == 200000 and results == [0, 1, 0]
