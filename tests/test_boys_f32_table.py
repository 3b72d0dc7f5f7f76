"""The FP32 tier's Boys table against the nodes that its kernel uses, on the host.

The harness compiles the table code and evaluates a seed the way the kernel does:
row k = round(20 T), x = fma(k, fl32(0.05), -T), a cubic in FP32.  T takes the
nodes, both sides of them and the largest distance from one.

Tolerance: the coefficient's and the last multiply-add's rounding, 2^-24 each, the
argument's below 2^-29, the truncation x^4 / 24 <= 1.7e-8, together 1.4e-7 of F_L.
A table made at other nodes is off by the node's offset times F_{L+1} / F_L, up to
9.5e-7 x 0.3."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2303_14280_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include "snk_internal.h"
int main() {
  snk::Setup s;
  snk::build_boys_tables(&s);
  double worst = 0.0;
  for (int k = 0; k < 600; ++k)
    for (int e = -4; e <= 4; ++e) {
      const float T = fmaf((float)k, snk::kBoysHF, 0.00624f * e);
      if (!(T >= 0.0f && T < snk::kBoysTMaxF)) continue;
      const float u = fmaf(T, 1.0f / snk::kBoysHF, 12582912.0f) - 12582912.0f;
      const float x = fmaf(u, snk::kBoysHF, -T);
      double F[snk::kBoysLMax + 1];
      snk::host_boys(snk::kBoysLMax, (double)T, F);
      for (int L = 0; L <= snk::kBoysLMax; ++L) {
        const float* r = &s.boys_f[((size_t)L * snk::kBoysRowsF + (int)u) * snk::kBoysColsF];
        const float f = fmaf(fmaf(fmaf(r[3], x, r[2]), x, r[1]), x, r[0]);
        const double rel = std::fabs((double)f - F[L]) / F[L];
        if (rel > worst) worst = rel;
      }
    }
  std::printf("%.3e\n", worst);
  return 0;
}
"""


def test_rows_belong_to_the_kernels_nodes(tmp_path):
    src, exe = tmp_path / "boys.cpp", tmp_path / "boys"
    src.write_text(SOURCE)
    cuda = next((d for d in ("/usr/local/cuda/include", "/usr/include")
                 if os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)
    if cuda is None:
        pytest.skip("no CUDA headers")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        "-I", cuda, str(src), os.path.join(CSRC, "host_setup.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0
    assert float(r.stdout) <= 1.4e-7, r.stdout
