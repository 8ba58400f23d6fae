"""Kernel attributes are set once per CUDA context, not by every bind and every step_static.

The memory of which contexts have them is a small host class; this compiles it with a program
that counts the calls it lets through."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1903_05133_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "context_once.h"
int main() {
  ha::ContextOnce once;
  int a = 0, b = 0;
  auto set_a = [&] { ++a; return 0; };
  auto set_b = [&] { ++b; return 0; };
  for (int i = 0; i < 5; ++i)
    if (once.run(7, 1, set_a) || once.run(7, 2, set_b)) return 1;
  if (a != 1 || b != 1) return 2;                       // once each in context 7
  for (int i = 0; i < 3; ++i) once.run(8, 1, set_a);
  if (a != 2 || b != 1) return 3;                       // again in another context
  for (int i = 0; i < 3; ++i) once.run(0, 1, set_a);
  if (a != 5) return 4;                                 // context unknown: every time
  int fails = 0;
  auto fail = [&] { ++fails; return 700; };
  if (once.run(9, 1, fail) != 700 || once.run(9, 1, fail) != 700 || fails != 2) return 5;
  if (once.run(9, 1, set_a) || a != 6) return 6;        // a failure is not remembered
  for (unsigned long long id = 100; id < 1000; ++id) once.run(id, 1, set_a);
  if (a != 906) return 7;
  once.run(999, 1, set_a);
  if (a != 906) return 8;
  int c = 0;
  std::vector<std::thread> ts;
  for (int i = 0; i < 8; ++i)
    ts.emplace_back([&] { for (int k = 0; k < 200; ++k) once.run(5000, 1, [&] { ++c; return 0; }); });
  for (auto& t : ts) t.join();
  return c == 1 ? 0 : 9;
}
"""


def test_settings_are_made_once_per_context(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_kernel_attributes_go_through_it():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "hier_avg_api.cu")).read())
    for call in ("ha::small_configure()", "ha::fp32_configure()", "ha::tc_configure()", "ha::head_configure()"):
        assert text.count(call) == 1, call
    body = text[text.index("int kernel_attributes("):]
    body = body[:body.index("\n}\n")]
    assert "current_context_id()" in body and body.count(".run(") == 1
    for call in ("small_configure", "fp32_configure", "tc_configure", "head_configure"):
        assert call in body
