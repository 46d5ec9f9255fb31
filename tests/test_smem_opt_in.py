"""The opt-in to dynamic shared memory (csrc/smem_opt_in.h) without a GPU: once per device, larger
sizes again, failures not remembered, from many threads; and no launcher keeps a flag of
its own for the whole process."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37029_gb300", "csrc")

MAIN = r"""
#include "smem_opt_in.h"
#include <cstdio>
#include <thread>
#include <vector>
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  static lsp::SmemOptIn once;
  int calls = 0;
  auto ok = [&] { ++calls; return 0; };
  auto fail = [&] { ++calls; return 7; };
  CHECK(once.ensure(0, 100, fail) == 7 && calls == 1);        // not remembered
  CHECK(once.ensure(0, 100, ok) == 0 && calls == 2);
  CHECK(once.ensure(0, 100, fail) == 0 && calls == 2);        // granted
  CHECK(once.ensure(0, 64, fail) == 0 && calls == 2);
  CHECK(once.ensure(0, 101, ok) == 0 && calls == 3);          // more
  CHECK(once.ensure(1, 100, ok) == 0 && calls == 4);          // another device
  CHECK(once.ensure(1, 101, fail) == 7 && calls == 5);
  CHECK(once.ensure(1, 100, fail) == 0 && calls == 5);        // what it had stays
  CHECK(once.ensure(1000, 1, ok) == 0 && once.ensure(1000, 1, ok) == 0 && calls == 7);   // no slot: every time
  static lsp::SmemOptIn shared;
  std::atomic<int> sets{0}, bad{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] {
      for (int i = 0; i < 2000; ++i)
        if (shared.ensure((t + i) % 4, 10, [&] { ++sets; return 0; })) ++bad;
    });
  for (auto& t : ts) t.join();
  CHECK(bad == 0 && sets == 4);
  return 0;
}
"""


def test_opt_in_is_per_device(tmp_path):
    src, exe = tmp_path / "main.cc", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_launcher_takes_the_opt_in():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        assert not re.search(r"cudaFuncSetAttribute", open(path).read()), path
