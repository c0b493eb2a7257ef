"""The renumbering kernel's shared memory, on the host: a launch is sized by the batch's largest tree while every CTA lays out its
own request's, so no smaller tree may need more.  (The layout header is plain C++.)"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_11744_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "dfs_layout.h"
int main() {
  int worst = 0;                                   // the most that any tree so far needs
  for (int n = 1; n <= 2048; ++n) {
    const dyspec::DfsLayout l(n);
    const dyspec::Splitters sp(2 * n);
    const bool all = n <= dyspec::kJumpAll;        // all elements jump, from the table's place on
    const int lists = l.jump + 8 * (all ? 2 * n : sp.count), tabled = l.table + (n + 1) * ((n + 31) / 32);
    if (!all && (l.next < l.table || l.at < l.next + 4 * n || l.jump < l.at + 8 * n)) { std::printf("n = %d: parts overlap\n", n); return 1; }
    if (l.bytes < lists || l.bytes < tabled) { std::printf("n = %d: %d bytes, %d and %d needed\n", n, l.bytes, lists, tabled); return 1; }
    if (l.bytes < worst) { std::printf("largest tree %d: %d bytes, %d needed by a smaller one\n", n, l.bytes, worst); return 1; }
    worst = l.bytes;
    int exist = 0;
    for (int e = 0; e < 2 * n; ++e) {              // a splitter's number gives its element back
      if (sp.element(sp.number(e)) != unsigned(e)) { std::printf("n = %d: element %d\n", n, e); return 1; }
      exist += sp.number(e) < sp.count;
    }
    if (exist > sp.exist) { std::printf("n = %d: %d splitters, %d expected\n", n, exist, sp.exist); return 1; }   // rounds of jumping
  }
  return worst <= 227 * 1024 ? 0 : 1;
}
"""


def test_no_request_of_a_batch_needs_more_than_the_largest(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
