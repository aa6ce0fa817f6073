"""Settings made once per device when several host threads come first together (plain C++, no GPU): nobody goes on
before the setting is made, it is made once, a failed one is tried again, and no device loses another's mark."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.cuh"

using namespace gep;

int main() {
  constexpr int DEV = 4, THREADS = 16, ROUNDS = 200;
  int wrong = 0;
  for (int round = 0; round < ROUNDS; ++round) {
    DeviceOnce once;
    DeviceValue value;
    std::atomic<int> made[DEV] = {}, calls[DEV] = {}, failed[DEV] = {}, bad{0};
    std::vector<std::thread> t;
    for (int i = 0; i < THREADS; ++i)
      t.emplace_back([&, i]() {
        const int d = i % DEV;
        int rc;
        do {
          rc = once.run(d, [&]() {
            if (d == 1 && failed[d].fetch_add(1) == 0) return -1;
            std::this_thread::sleep_for(std::chrono::microseconds(50));
            calls[d].fetch_add(1);
            made[d].store(1);
            return 0;
          });
        } while (rc != 0);
        if (made[d].load() != 1) bad.fetch_add(1);
        int v = -1;
        value.get(d, &v, [&](int* out) {
          std::this_thread::sleep_for(std::chrono::microseconds(50));
          *out = 10 + d;
          return 0;
        });
        if (v != 10 + d) bad.fetch_add(1);
      });
    for (auto& x : t) x.join();
    wrong += bad.load();
    for (int d = 0; d < DEV; ++d) wrong += calls[d].load() != 1;
  }
  printf("%d\n", wrong);
  return wrong != 0;
}
"""


def test_first_use_from_many_threads(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_1504_06443_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, timeout=120).stdout.strip() == "0"


def test_no_unprotected_state():
    """Function statics of the library's host code are one of the protected kinds."""
    import glob
    import re
    for path in glob.glob(os.path.join(ROOT, "paper_1504_06443_gb300", "csrc", "*.cu*")):
        for line in open(path):
            m = re.match(r"\s+static\s+(?!constexpr|_assert)(.*)", line)
            assert not m or re.match(r"(DeviceOnce|DeviceValue|std::atomic<|thread_local )", m.group(1)), (path, line)
