"""The change of lambda that stops the adjoint solve (csrc/adjoint_cell.h, as both of its
forms call it) is formed in FP64 from the working precision's values: an FP32 difference
would round each of them to 2^-24."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_1502_06216_gb300

PROGRAM = r"""
#include <cstdio>
#include "adjoint_cell.h"
int main() {
  float a, b;
  while (std::scanf("%a %a", &a, &b) == 2) std::printf("%a\n", jko::lambda_change(a, b));
}
"""


def test_change_of_lambda_keeps_the_bits_an_fp32_difference_drops(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    csrc = os.path.join(os.path.dirname(paper_1502_06216_gb300.__file__), "csrc")
    (tmp_path / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", csrc, str(tmp_path / "p.cpp"),
                    "-o", str(tmp_path / "p")], check=True)
    rng = np.random.default_rng(0)
    a = rng.uniform(-1, 1, 200).astype(np.float32)
    b = (a * rng.uniform(-1e-3, 1, 200)).astype(np.float32)
    text = "\n".join(f"{float(x).hex()} {float(y).hex()}" for x, y in zip(a, b))
    out = subprocess.run([str(tmp_path / "p")], input=text, check=True, capture_output=True, text=True)
    got = [float.fromhex(v) for v in out.stdout.split()]
    exact = [abs(float(x) - float(y)) for x, y in zip(a, b)]
    assert got == exact
    in_fp32 = [float(np.abs(x - y)) for x, y in zip(a, b)]
    assert sum(x != y for x, y in zip(in_fp32, exact)) > 50    # the inputs tell the two apart
