"""Kernel limits and occupancies are kept per device (csrc/per_device.h), with
devices stood in for by numbers: no GPU is needed, and a test machine has one."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_00970_gb300", "csrc")
PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
  gs2d::PerDevice p, q;
  int made = 0, v = 0;
  auto make = [&](int x) { return [&made, x](int* o) { ++made; *o = x; return 0; }; };
  CHECK(p.get(0, &v, make(304)) == 0 && v == 304 && made == 1);
  CHECK(p.get(0, &v, make(7)) == 0 && v == 304 && made == 1);       // kept
  CHECK(p.get(1, &v, make(264)) == 0 && v == 264 && made == 2);     // the second device's own
  CHECK(p.get(0, &v, make(7)) == 0 && v == 304 && made == 2);
  CHECK(q.get(0, &v, make(5)) == 0 && v == 5 && made == 3);         // another kernel's table
  CHECK(p.get(2, &v, [&](int*) { ++made; return 9; }) == 9);        // a failure is not kept
  CHECK(p.get(2, &v, make(11)) == 0 && v == 11 && made == 5);
  for (int k = 0; k < 2; ++k) CHECK(p.get(64, &v, make(13 + k)) == 0 && v == 13 + k);
  CHECK(p.get(-1, &v, make(1)) == 0 && made == 8);
  gs2d::PerDevice r;
  made = 0;
  std::vector<std::thread> ts;
  for (int k = 0; k < 8; ++k)
    ts.emplace_back([&, k] { int x = 0; for (int i = 0; i < 100; ++i) r.get(k & 1, &x, make(k & 1)); });
  for (auto& t : ts) t.join();
  CHECK(made == 2);
  return 0;
}
"""


def test_values_are_made_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_kernel_attribute_is_set_once_per_process():
    """Every cudaFuncSetAttribute call stands behind a table by device."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"cudaFuncSetAttribute\(", text):
            before = text[max(0, m.start() - 500):m.start()]
            assert re.search(r"limits\.get|(ready|slots|done|done_per_dev)\[dev\]", before), \
                (name, text.count("\n", 0, m.start()) + 1)
