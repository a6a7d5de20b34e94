"""The per-device table of launch facts (csrc/device_table.h): threads that meet in their first call work a value out once and
all read that one; a failed attempt is handed on and tried again."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "device_table.h"
int main() {
  static he::DeviceTable<3> table;
  std::atomic<int> made{0}, wrong{0};
  std::vector<std::thread> threads;
  for (int i = 0; i < 24; ++i)
    threads.emplace_back([&, i] {
      for (int dev = 0; dev < 2; ++dev)
        for (int item = 0; item < 3; ++item) {
          int v = 0;
          const int rc = table.get(dev, item, &v, [&](int* out) -> int {
            ++made;
            std::this_thread::sleep_for(std::chrono::milliseconds(5));
            *out = item == 2 ? -1 : 100 * dev + item + 1;
            return 0;
          });
          if (rc != 0 || v != (item == 2 ? -1 : 100 * dev + item + 1)) ++wrong;
        }
    });
  for (auto& t : threads) t.join();
  int v = 7, rc1 = table.get(5, 0, &v, [](int* out) -> int { *out = 3; return 9; });
  const bool kept = v == 7;
  int rc2 = table.get(5, 0, &v, [](int* out) -> int { *out = 4; return 0; });
  std::printf("%d %d %d %d %d %d\n", made.load(), wrong.load(), rc1, (int)kept, rc2, v);
}
"""


def test_first_calls_of_many_threads_work_a_value_out_once(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2412_16187_b200", "csrc"), "-o", exe, src], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True, timeout=60).stdout.split()
    assert out == ["6", "0", "9", "1", "0", "4"]
