"""The epoch a persistent kernel leaves for the next launch (csrc/epoch.h, as the kernels
call it), on the CPU: the exchanges of a launch, counted as its loops make them, stay
within the bound, and a launch whose wait gave up leaves an epoch behind everything any of
its blocks can have published (else the next launch takes stale words for its own)."""
import shutil
import subprocess

import pytest

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "epoch.h"
using namespace jko::epoch;
int main() {
  int bad = 0;
  for (unsigned pairs = 1; pairs <= 60; ++pairs) {
    unsigned ep = 0;                             // strips: an exchange a pair, and the end's
    for (unsigned p = 0; p < pairs; ++p) ep = 1 + p;
    const unsigned end = 2 + pairs;
    bad += ep > of_strip(pairs) || end > of_strip(pairs);
    for (unsigned D = 1; D <= 70; ++D) {         // the heat kernel's phases
      const unsigned H = 4;
      unsigned e = 0, published = 0;
      for (unsigned p = 0; p < pairs; ++p)
        for (int app = 0; app < 2; ++app) {
          ++e;
          published = e > published ? e : published;
          int ns = D % H == 0 ? H : D % H;
          for (int k = (int)D - 1; k >= 0; k -= ns, ns = H)
            if (k - ns >= 0) {
              published = e + 1 > published ? e + 1 : published;
              ++e;
            }
        }
      bad += published > of_heat(pairs, D, H);
    }
    unsigned a = 2;                              // the reverse pass
    for (unsigned k = 0; k < pairs; ++k) ++a;
    bad += ++a > of_adjoint(pairs);
  }
  // after a fault no epoch 1 .. most of the launch comes again; else they go on from the last
  for (unsigned first : {0u, 7u, 0xfffffff0u})
    for (unsigned most = 3; most < 40; ++most)
      for (unsigned last = 1; last <= most; ++last) {
        const unsigned next = after(first, first + last, most, true);
        for (unsigned e = 1; e <= most; ++e) bad += next + 1 == first + e;
        bad += after(first, first + last, most, false) != first + last;
      }
  std::printf("%d\n", bad);
}
"""


def test_a_launch_that_gave_up_leaves_a_later_epoch(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    import os
    import paper_1502_06216_gb300
    csrc = os.path.join(os.path.dirname(paper_1502_06216_gb300.__file__), "csrc")
    (tmp_path / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", csrc, str(tmp_path / "p.cpp"),
                    "-o", str(tmp_path / "p")], check=True)
    out = subprocess.run([str(tmp_path / "p")], check=True, capture_output=True, text=True)
    assert out.stdout.split() == ["0"]
