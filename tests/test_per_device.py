"""Kernels' shared-memory limits are raised on every device a process uses: the
helper that remembers devices, compiled and run on the CPU, and the sources,
where no launch keeps that setting in a static of the process."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_05279_gb300", "csrc")

PROGRAM = r"""
#include "per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
#define CHECK(c) do { if (!(c)) { std::printf("line %d\n", __LINE__); return 1; } } while (0)
int main() {
  bmg::PerDevice p;
  int calls = 0;
  auto ok = [&] { ++calls; return 0; };
  CHECK(p.once(0, ok) == 0 && p.once(0, ok) == 0 && calls == 1);
  CHECK(p.once(1, ok) == 0 && p.once(63, ok) == 0 && p.once(1, ok) == 0 && calls == 3);   // other devices
  CHECK(p.once(5, [&] { ++calls; return 7; }) == 7 && calls == 4);                        // a failure is not remembered
  CHECK(p.once(5, ok) == 0 && calls == 5 && p.once(5, ok) == 0 && calls == 5);
  CHECK(p.once(64, ok) == 0 && p.once(64, ok) == 0 && calls == 7);                        // past the table: every time
  CHECK(p.once(-1, ok) == 0 && calls == 8);
  bmg::PerDevice q;
  std::atomic<int> n{0}, early{0};
  std::vector<std::thread> t;
  for (int k = 0; k < 8; ++k)
    t.emplace_back([&] {
      bool mine = false;
      q.once(2, [&] { mine = true; n.fetch_add(1); return 0; });
      if (!mine && n.load() == 0) early = 1;
    });
  for (auto& x : t) x.join();
  CHECK(n.load() >= 1 && !early.load() && q.once(2, ok) == 0 && calls == 8);
  return 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cc", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_no_limit_is_kept_for_the_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"cudaFuncSetAttribute", src):
            stmt = src[src.rfind("static ", 0, m.start()):m.start()]
            inside = not re.search(r"\n\}", stmt) and ("= [] {" in stmt or stmt.rstrip().endswith("="))
            assert not inside, (os.path.basename(path), src[m.start():m.start() + 80])
