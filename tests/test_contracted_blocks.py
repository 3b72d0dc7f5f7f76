"""The contracted integral code that builds run, entry by entry, against the recursion
for every primitive pair in long double, on the host.

For every class, 1 to 16 primitive pairs, centres 0 to 12 bohr apart and points on a
centre, near and far, both the FP64 form (prefactor in the coefficients) and the
double-FP32 form run the generated prim / build / hrr.

Tolerance per entry: the contracted form once more on absolute values, every
difference a sum, gives the sum of the absolute values of all terms; a chain of at
most 64 roundings of u each (2^-53, 2^-46 per operation in double-FP32), from seeds
exact to a rounding.  The primitive pairs' geometry is given exactly, as P - A =
-sigma AB in long double."""
import host_cuda

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "ds_arith.cuh"
typedef long double LD;
namespace snk {
using std::fma;
// sums of absolute values
struct Abs { LD v; Abs() : v(0) {} explicit Abs(LD x) : v(fabsl(x)) {} explicit Abs(int x) : v(x < 0 ? -x : x) {} };
inline Abs operator+(Abs a, Abs b) { return Abs(a.v + b.v); }
inline Abs operator-(Abs a, Abs b) { return Abs(a.v + b.v); }
inline Abs operator-(Abs a) { return a; }
inline Abs operator*(Abs a, Abs b) { return Abs(a.v * b.v); }
inline Abs& operator+=(Abs& a, Abs b) { a = a + b; return a; }
inline Abs fma(Abs a, Abs b, Abs c) { return Abs(a.v * b.v + c.v); }
}
#include "os_generated.cuh"
using namespace snk;

// F_n(T) by the ascending series
static void boys(int L, LD T, LD* F) {
  for (int n = 0; n <= L; ++n) {
    LD t = 1.0L / (2 * n + 1), s = t;
    for (int i = 1; i < 400; ++i) { t *= 2 * T / (2 * n + 2 * i + 1); s += t; if (t < 1e-22L * s) break; }
    F[n] = expl(-T) * s;
  }
}
static ds split(LD x) { const float h = (float)x; return ds_make(h, (float)(x - (LD)h)); }
static LD value(double x) { return x; }
static LD value(ds x) { return (LD)x.hi + (LD)x.lo; }
template <class R> R as(LD x);
template <> double as<double>(LD x) { return (double)x; }
template <> ds as<ds>(LD x) { return split(x); }
template <> Abs as<Abs>(LD x) { return Abs(x); }

template <int LA, int LB, class R>
static void contracted(int np, const LD* sg, const LD* kp, const LD* pf, const LD (*F)[5], const LD* AB, const LD* AC,
                       bool pref_in_c, R* xi) {
  using C = OsClass<LA, LB>;
  R M[C::NM], acc[C::NACC], S[C::L + 1];
  for (auto& m : M) m = as<R>(0.0L);
  for (int p = 0; p < np; ++p) {
    const LD f = pref_in_c ? 1.0L : pf[p], g = pref_in_c ? pf[p] : 1.0L;
    for (int n = 0; n <= C::L; ++n) S[n] = as<R>(f * F[p][n]);
    const LD s = sg[p], k = kp[p];
    OsCoef<R> c{as<R>(g), as<R>(g * s), as<R>(g * s * s), as<R>(g * s * s * s), as<R>(g * s * s * s * s), as<R>(g * k),
                as<R>(g * s * k), as<R>(g * s * s * k), as<R>(g * k * k)};
    C::prim(S, c, M);
  }
  C::build(M, as<R>(-AB[0]), as<R>(-AB[1]), as<R>(-AB[2]), as<R>(-AC[0]), as<R>(-AC[1]), as<R>(-AC[2]), acc);
  C::hrr(acc, as<R>(AB[0]), as<R>(AB[1]), as<R>(AB[2]), xi);
}

static double worst[2] = {0, 0};
template <int LA, int LB>
static void cls(std::mt19937_64& g) {
  using C = OsClass<LA, LB>;
  constexpr int N = C::NA * C::NB;
  std::uniform_real_distribution<double> u(0, 1);
  std::normal_distribution<double> z;
  for (int trial = 0; trial < 3000; ++trial) {
    const int np = 1 + trial % 16;
    const double apart[] = {0.0, 0.5, 1.5, 4.0, 12.0}, away[] = {0.0, 0.3, 2.0, 8.0};
    LD AB[3], AC[3], sg[16], kp[16], pf[16], F[16][5], ref[N], acc[C::NACC];
    for (int q = 0; q < 3; ++q) {
      AB[q] = (float)(z(g) * apart[trial % 5] / 1.7);  // floats: every type holds them exactly
      AC[q] = (float)(z(g) * away[trial % 4] / 1.7);
    }
    for (auto& a : acc) a = 0;
    for (int p = 0; p < np; ++p) {
      LD a = 0, b = 0, ab2 = 0, pc2 = 0, PA[3], PC[3], S[5];
      for (int q = 0; q < 3; ++q) ab2 += AB[q] * AB[q];
      // exponents from 0.1 to 30, e^{-a b |AB|^2 / (a + b)} not below e^-60 (1e-26)
      do {
        a = std::exp(std::log(0.1) + u(g) * std::log(300.0));
        b = std::exp(std::log(0.1) + u(g) * std::log(300.0));
        if (ab2 > 500) a = b = 0.1;
      } while (ab2 <= 500 && a * b / (a + b) * ab2 > 60);
      sg[p] = b / (a + b);
      kp[p] = 0.5L / (a + b);
      for (int q = 0; q < 3; ++q) { PA[q] = -sg[p] * AB[q]; PC[q] = AC[q] + PA[q]; pc2 += PC[q] * PC[q]; }
      pf[p] = (0.2L + u(g)) * expl(-a * b / (a + b) * ab2) / (a + b);
      boys(C::L, std::fmin((LD)60, (a + b) * pc2), F[p]);
      for (int n = 0; n <= C::L; ++n) S[n] = pf[p] * F[p][n];
      C::vrr(S, PA[0], PA[1], PA[2], PC[0], PC[1], PC[2], kp[p], 2 * kp[p], 3 * kp[p], acc);
    }
    C::hrr(acc, AB[0], AB[1], AB[2], ref);
    double x64[N];
    ds xds[N];
    Abs mag[N];
    contracted<LA, LB>(np, sg, kp, pf, F, AB, AC, true, x64);
    contracted<LA, LB>(np, sg, kp, pf, F, AB, AC, false, xds);
    contracted<LA, LB>(np, sg, kp, pf, F, AB, AC, false, mag);
    LD big = 0;
    for (int k = 0; k < N; ++k) big = fmaxl(big, fabsl(ref[k]));
    for (int k = 0; k < N; ++k) {
      const LD e[2] = {fabsl(value(x64[k]) - ref[k]), fabsl(value(xds[k]) - ref[k])};
      for (int f = 0; f < 2; ++f) {
        // below the smallest FP32 normal a double-FP32 value has no tail
        const LD tol = 64 * (f ? 0x1p-46L : 0x1p-53L) * mag[k].v + (f ? 1e-36L : 0);
        if (!(e[f] <= tol)) {
          std::printf("class %d %d form %d entry %d, %d primitive pairs: %.3Le > %.3Le\n", LA, LB, f, k, np, e[f], tol);
          std::exit(1);
        }
        if (mag[k].v > 0) worst[f] = std::fmax(worst[f], (double)(e[f] / mag[k].v));
      }
    }
  }
}
int main() {
  std::mt19937_64 g(5);
  cls<0, 0>(g); cls<1, 0>(g); cls<1, 1>(g); cls<2, 0>(g); cls<2, 1>(g); cls<2, 2>(g);
  std::printf("%.3e %.3e\n", worst[0], worst[1]);
}
"""


def test_contracted_blocks_match_the_recursion(tmp_path):
    fp64, ds = (float(v) for v in host_cuda.run(tmp_path, SOURCE).split())
    assert 0.0 < fp64 <= 64 * 2.0 ** -53 and 0.0 < ds <= 64 * 2.0 ** -46
