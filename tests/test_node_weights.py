"""The weights of P^T (longitudinal to transverse grid, transposed) in the
adjoint kernel with one thread per row: node_weights of csrc/sfd_df64.cuh,
compiled for the host, against exact fractions.

A double-float quotient carries 46 bits (rcp_df's bound 2^-46, an exact integer
product and a rounding 2^-47 of a sum below 1), so the weights are within
2^-44; a float's are 2^-25 off.  The kernel takes them from nowhere else."""

import os
import re
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_18505_gb300", "csrc")

# the device intrinsics the header's sums and products use
SHIM = """
#pragma once
#include <cmath>
#define __device__
#define __host__
#define __forceinline__ inline
static inline float __fadd_rn(float a, float b) { volatile float s = a + b; return s; }
static inline float __fsub_rn(float a, float b) { volatile float s = a - b; return s; }
static inline float __fmul_rn(float a, float b) { volatile float p = a * b; return p; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float __shfl_up_sync(unsigned, float v, int) { return v; }
static inline float __shfl_down_sync(unsigned, float v, int) { return v; }
static inline float __shfl_xor_sync(unsigned, float v, int) { return v; }
"""

PROGRAM = """
#include <cstdio>
#include "df64.h"
int main() {
  for (int n_t = 2; n_t <= 256; ++n_t) {
    const double d = 1.0 / n_t;
    const float h = static_cast<float>(d);
    const sfd::df64 inv(h, static_cast<float>(d - h));
    for (int rem = 0; rem < n_t; ++rem) {
      const sfd::dfl::NodeWeights w = sfd::dfl::node_weights(rem, n_t, inv);
      std::printf("%d %d %.17g %.17g\\n", n_t, rem, static_cast<double>(w.left.hi) + w.left.lo,
                  static_cast<double>(w.right.hi) + w.right.lo);
    }
  }
}
"""


def test_weights_carry_more_than_a_floats_bits(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    (tmp_path / "cuda_runtime.h").write_text(SHIM)
    header = open(os.path.join(CSRC, "sfd_df64.cuh")).read()
    # (the reciprocal is the only inline assembly; the program does not call it)
    (tmp_path / "df64.h").write_text(re.sub(r"  asm\(.*?\);\n", "  x0 = 1.f / b.hi;\n", header))
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = tmp_path / "weights"
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", str(tmp_path), str(tmp_path / "main.cpp"),
                    "-o", str(exe)], check=True)
    rows = np.array([r.split() for r in subprocess.run([str(exe)], capture_output=True, text=True,
                                                       check=True).stdout.splitlines()], float)
    n_t, rem, left, right = rows.T
    assert len(rows) == sum(range(2, 257))
    assert np.max(np.abs(left - (n_t - rem) / n_t)) <= 2.0 ** -44
    assert np.max(np.abs(right - rem / n_t)) <= 2.0 ** -44


def test_the_row_kernel_spreads_with_them():
    """Every product that P^T sums (arrays P0, P1 and Q0, Q1) is formed with them."""
    src = open(os.path.join(CSRC, "sfd_adjoint_rows.cu")).read()
    left = re.findall(r"put\([PQ]0 \+ i, (\S+) \* [fh]\);", src)
    right = re.findall(r"put\([PQ]1 \+ i, (\S+) \* [fh]\);", src)
    assert left == ["wt.left"] * 3 and right == ["wt.right"] * 3
