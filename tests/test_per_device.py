"""A kernel's shared-memory limit is raised on every device it is launched on (csrc/idkm_per_device.h), shown with stand-ins
for the device and for the call that raises it."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_07759_b200", "csrc")

PROGRAM = r"""
#include "idkm_per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  idkm::PerDevice limit;
  int raised[70] = {0}, status = 0;
  auto call = [&](int dev) { return limit.once(dev, [&] { ++raised[dev]; return status; }); };
  bool ok = call(0) == 0 && call(0) == 0 && raised[0] == 1;
  ok = ok && call(1) == 0 && raised[1] == 1 && raised[0] == 1;      // a second device is not taken for the first
  status = 7;
  ok = ok && call(2) == 7 && call(2) == 7 && raised[2] == 2;        // a refusal is not remembered
  status = 0;
  ok = ok && call(2) == 0 && call(2) == 0 && raised[2] == 3;
  ok = ok && call(63) == 0 && call(63) == 0 && raised[63] == 1 && call(64) == 0 && call(64) == 0 && raised[64] == 2;
  idkm::PerDevice shared;
  std::atomic<int> calls{0}, bad{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] { for (int i = 0; i < 1000; ++i) bad += shared.once(t % 4, [&] { ++calls; return 0; }) != 0; });
  for (auto& t : ts) t.join();
  ok = ok && bad == 0 && calls >= 4 && calls <= 8;
  std::puts(ok ? "ok" : "wrong");
  return ok ? 0 : 1;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "ok"


def test_no_launcher_remembers_a_limit_for_the_process():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static\s+bool\s+\w*configured", text), name
