"""Kernel attributes are set on every device that launches the kernel: they belong to the device
that is current, and a process may hold contexts on several. The helper is compiled for the host
here (one GPU cannot show it), and the sources are read for attributes set once per process."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_21236_gb300", "csrc")

MAIN = r"""
#include "per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  static attn::PerDevice p;
  std::atomic<int> calls[70] = {};
  std::atomic<int> wrong{0};
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&] {
      for (int d = 0; d < 64; ++d)
        if (p.get(d, [&] { ++calls[d]; std::this_thread::yield(); return 3 * d; }) != 3 * d) ++wrong;
    });
  for (auto& x : t) x.join();
  for (int d = 0; d < 64; ++d) if (calls[d] != 1) ++wrong;
  for (int i = 0; i < 2; ++i) if (p.get(64, [&] { ++calls[64]; return 7; }) != 7) ++wrong;
  if (calls[64] != 2) ++wrong;
  static attn::PerDevice q;
  try { q.get(1, []() -> int { throw 5; }); ++wrong; } catch (int) {}
  if (q.get(1, [] { return 0; }) != 0) ++wrong;
  if (q.get(1, [] { return 9; }) != 0) ++wrong;  // a value of 0 is remembered too
  std::printf("%d\n", wrong.load());
  return wrong.load() != 0;
}
"""


def test_evaluated_once_on_every_device(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, timeout=60).stdout.strip() == "0"


def _guards(text):
    """For every cudaFuncSetAttribute: the static variables of its function before it."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer("cudaFuncSetAttribute", text):
        function = text[text.rfind("\n}", 0, m.start()) + 1:m.start()]
        yield re.findall(r"\bstatic (\w+) \w+(?: = [^;]*)?;", function)


def test_no_attribute_is_set_once_per_process():
    """Every cudaFuncSetAttribute stands in a PerDevice evaluation, or unguarded."""
    guards = [(os.path.basename(p), g) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))
              for g in _guards(open(p).read())]
    assert guards
    assert [(f, g) for f, g in guards if set(g) - {"PerDevice"}] == []
    assert [g for g in _guards("static bool a = false;\nif (!a) cudaFuncSetAttribute(k);")] == [["bool"]]
