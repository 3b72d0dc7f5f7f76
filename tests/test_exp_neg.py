"""e^{-x} of the collocation kernels, on the host, against long double.

Tolerance: the table holds 2^{-j/256} and its relative error, so what is left is the
rounding of the last addition, at most 2^-53, the polynomial's truncation, 4e-17, and
roundings 2^-9 times smaller: 1.6e-16 relative.  With the head alone its own rounding
comes on top, 2.4e-16."""
import host_cuda

SOURCE = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "exp_neg.cuh"
int main() {
  std::vector<double2> tab(snk::kExpTable);
  snk::exp_table_fill(tab.data());
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> u(0.0, 60.0), v(0.0, 1.0);
  double worst = 0.0;
  auto look = [&](double x) {
    const long double ref = expl(-(long double)x);
    const double rel = (double)fabsl(((long double)snk::exp_neg(x, tab.data()) - ref) / ref);
    if (rel > worst) worst = rel;
  };
  for (int n = 0; n < 1000000; ++n) look(u(g)), look(v(g));
  for (int k = 0; k < 22000; ++k)  // where the table row changes
    for (int e = -1; e <= 1; ++e) look(std::fmax(0.0, (k + 0.5 + 1e-12 * e) * 0.6931471805599453 / 256));
  look(0.0); look(5e-324); look(1e-300); look(699.0);
  std::printf("%.3e\n", worst);
}
"""


def test_error_is_one_rounding(tmp_path):
    assert float(host_cuda.run(tmp_path, SOURCE)) <= 1.6e-16
