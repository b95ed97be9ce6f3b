"""The column pass's sum of a cluster's four FP32 partial results (sum4, sums.cuh),
compiled for the host: exact to 2^-46 of the largest, where a sum in FP32 is
off by 2^-24 -- partial results meet in FP64."""
import math
import os
import subprocess

import numpy as np

import paper_2609_01978_gb300 as fzp

CSRC = os.path.join(os.path.dirname(fzp.__file__), "csrc")
MAIN = r"""
#include <cstdio>
#include "sums.cuh"
int main() {
  float v[4];
  while (scanf("%a %a %a %a", v, v + 1, v + 2, v + 3) == 4) printf("%a\n", fzp::sum4(v));
}
"""


def test_sum_of_four(tmp_path):
    src = tmp_path / "main.cu"
    src.write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-std=c++17", "-O3", "-I", CSRC, "-o", exe, str(src)], check=True)
    rng = np.random.default_rng(3)
    v = (rng.standard_normal((4000, 4)) * 2.0 ** rng.integers(-12, 13, (4000, 4))).astype(np.float32)
    v[:50, 1:3] = -v[:50, [0]]  # cancelling pairs
    text = "\n".join(" ".join(float(x).hex() for x in row) for row in v)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    assert len(out) == len(v)
    worst = max(abs(float.fromhex(o) - math.fsum(map(float, row))) / float(np.abs(row).max()) for o, row in zip(out, v))
    assert worst <= 2.0 ** -46
