"""Kernel attributes and SM counts are a device's: a process with contexts on two devices sets and asks them on both."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_01275_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.hpp"
int main() {
  nlmg::DeviceOnce once;
  int calls = 0;
  auto ok = [&] { ++calls; return 0; };
  auto bad = [&] { ++calls; return 7; };
  std::printf("%d ", once.run(0, bad));                  // an error is returned and not remembered
  once.run(0, ok); once.run(0, ok); once.run(0, bad);    // once
  std::printf("%d ", calls);
  once.run(1, ok); once.run(1, ok);                      // the second device has its own
  std::printf("%d ", calls);
  once.run(64, ok); once.run(64, ok); once.run(-1, ok);  // beyond the table: every time
  std::printf("%d ", calls);
  std::atomic<int> n{0};
  nlmg::DeviceOnce many;
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] { for (int i = 0; i < 1000; ++i) many.run(t % 4, [&] { ++n; return 0; }); });
  for (auto& t : ts) t.join();
  std::printf("%d\n", n.load() >= 4 && n.load() <= 8);
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["7", "2", "3", "6", "1"]


def test_attributes_are_set_per_device_and_checked():
    """Every kernel's limit goes through the one helper, which remembers it per device and returns its error."""
    calls = []
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        calls += [name] * text.count("cudaFuncSetAttribute(")
        for m in re.finditer(r"static[^;{]*=\s*\[[^\]]*\]", text):
            body = text[m.start():m.start() + 400].split("}()")[0]
            assert not re.search(r"cuda(FuncSetAttribute|GetDevice|DeviceGetAttribute)", body), name
    assert calls == ["persist.cu"]
