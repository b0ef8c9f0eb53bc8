"""Properties of the kernel sources that hold for the whole library (no GPU)."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_05194_gb300", "csrc")


def code(path):
    src = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)


def test_no_copy_or_commit_goes_to_several_ctas():
    """The library is loaded by every rank of a multi-GPU program: its tile loads and commits
    stay within one CTA."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        assert not re.search(r"multicast", code(path), re.I), os.path.basename(path)


def test_nothing_about_a_kernel_is_kept_per_process():
    """Launch attributes and occupancies belong to a device: a flag or a value kept in a plain
    static would leave a second device's kernels at the default shared-memory limit."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        assert not re.search(r"static (int|bool) \w+ = (-1|false);[^}]*cudaFuncSetAttribute", code(path)), path


ONCE = """
#include <assert.h>
#include <thread>
#include <vector>
#include "kite_once.h"
int main() {
  static kite::PerDevice p;
  int calls = 0;
  auto f = [&](int v) { return [&calls, v] { ++calls; return v; }; };
  assert(p.get(0, f(3)) == 3 && p.get(0, f(9)) == 3 && calls == 1);  // kept
  assert(p.get(1, f(0)) == 0 && p.get(1, f(9)) == 0 && calls == 2);  // another device, and zero
  assert(p.get(2, f(-1)) == -1 && p.get(2, f(5)) == 5 && p.get(2, f(9)) == 5 && calls == 4);  // failures are not
  assert(p.get(64, f(7)) == 7 && p.get(64, f(8)) == 8 && p.get(-1, f(6)) == 6);  // beyond the table: computed
  static kite::PerDevice q;
  std::vector<std::thread> ts;
  std::atomic<int> bad{0};
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&] { for (int d = 0; d < 64; ++d) if (q.get(d, [d] { return d + 1; }) != d + 1) ++bad; });
  for (auto& t : ts) t.join();
  assert(bad == 0);
}
"""


def test_values_are_kept_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(ONCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    subprocess.run([str(exe)], check=True)
