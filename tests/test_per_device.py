"""Launch settings found once per device (csrc/per_device.h): threads that ask together all get the finished
value, and a failure is not remembered.  Host code only, compiled and run here."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
  static dfmm::PerDevice<int> sms;
  std::atomic<int> calls{0}, wrong{0};
  auto find = [&](int v) {
    ++calls;
    std::this_thread::sleep_for(std::chrono::milliseconds(50));
    return v;
  };
  std::vector<std::thread> t;
  for (int i = 0; i < 32; ++i)
    t.emplace_back([&, i] { if (sms.get(i % 2, [&] { return find(152 + i % 2); }) != 152 + i % 2) ++wrong; });
  for (auto& x : t) x.join();
  int thrown = 0;
  for (int dev : {-1, 64})
    try { sms.get(dev, [&] { return find(1); }); } catch (const std::exception&) { ++thrown; }
  try { sms.get(7, [&]() -> int { throw std::runtime_error("not now"); }); } catch (const std::exception&) { ++thrown; }
  if (sms.get(7, [&] { return find(5); }) != 5) ++wrong;
  std::printf("%d %d %d\n", calls.load(), wrong.load(), thrown);
}
"""


def test_value_is_found_once_and_complete(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", os.path.join(ROOT, "paper_1311_4257_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    assert out == ["3", "0", "3"]
