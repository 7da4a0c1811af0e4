// Host program of test_pointwise_algebra.py: the two passes of the pointwise
// Z4c right-hand side (csrc/z4c_pass.cuh) in double against long double, on
// random metrics stretched by a factor s along x with shear of relative size
// `shear`, matter and derivatives of relative size `grad`.  Prints, per
// quantity, the r.m.s. error over the r.m.s. value and the mean of the error
// relative to the value itself.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

namespace sacra {
inline long double z4c_rcp(long double v) { return 1 / v; }
inline long double z4c_sqrt(long double v) { return sqrtl(v); }
}  // namespace sacra
#include "z4c_pass.cuh"
using namespace sacra;

struct In {
  double U[30], D1[16][3], D2[11][6], PR[6];
};
constexpr int NO = 25 + zN + 1;   // right-hand sides, pass A's planes, the Ricci scalar

template <class T>
void cell(const In &in, T *out) {
  T scr[zN];
  auto U = [&](int f) { return T(in.U[f]); };
  auto D1 = [&](int a, int k) { return T(in.D1[a][k]); };
  z4c_pass_a<T>(U, D1, [&](int f, T v) { scr[f] = v; });
  for (int f = 0; f < zN; ++f) out[25 + f] = scr[f];
  const Z4cPar<T> p{T(0.02), T(1.25), 0};
  z4c_pass_b<T>(p, U, D1, [&](int a, int k) { return T(in.D2[a][k]); }, [&](int) { return T(0); },
                [&](int f) { return T(in.PR[f]); }, [&](int f) { return scr[f]; }, T(0.9),
                [&](int f, T v) { out[f] = v; }, [&](T v) { out[25 + zN] = v; });
}

int main(int argc, char **argv) {
  const double s = atof(argv[1]), shear = atof(argv[2]), grad = atof(argv[3]), offdiag = atof(argv[4]);
  const int n = 4000;
  std::mt19937_64 gen(7);
  std::uniform_real_distribution<double> uni(-1.0, 1.0);
  auto r = [&] { return uni(gen); };
  double e2[NO] = {}, v2[NO] = {}, rel[NO] = {};
  for (int t = 0; t < n; ++t) {
    In in;
    memset(&in, 0, sizeof in);
    const double d[3] = {s, 1 / std::sqrt(s), 1 / std::sqrt(s)};
    double gs[6];
    for (int i = 0; i < 3; ++i)
      for (int j = i; j < 3; ++j) {
        const int q = sq(i, j);
        gs[q] = std::sqrt(d[i] * d[j]);
        in.U[fHXX + q] = (i == j ? d[i] - 1.0 : 0.0) + shear * gs[q] * r();
        in.U[fAXX + q] = grad * gs[q] * r();
      }
    in.U[fW] = 0.9 + 0.05 * r();
    in.U[fAL] = 0.8 + 0.1 * r();
    in.U[fKH] = grad * r();
    in.U[fTH] = 0.1 * grad * r();
    for (int i = 0; i < 3; ++i) { in.U[fGX + i] = grad * r(); in.U[fBX + i] = 0.1 * r(); in.U[fBBX + i] = 0.1 * grad * r(); }
    for (int a = 0; a < 16; ++a)
      for (int k = 0; k < 3; ++k) in.D1[a][k] = grad * (a >= 1 && a <= 6 ? gs[a - 1] : 1.0) * r();
    for (int i = 0; i < 3; ++i)      // off-diagonal shift gradients of their own size
      for (int k = 0; k < 3; ++k)
        if (i != k) in.D1[13 + i][k] *= offdiag;
    for (int a = 0; a < 11; ++a)
      for (int q = 0; q < 6; ++q) in.D2[a][q] = grad * (a >= 1 && a <= 6 ? gs[a - 1] : 1.0) * r();
    in.PR[pRHO] = 1e-3 * (1 + 0.5 * r());
    in.PR[pP] = 1e-4 * (1 + 0.5 * r());
    in.PR[pEPS] = 0.1 * (1 + 0.5 * r());
    if (t & 1)
      for (int i = 0; i < 3; ++i) in.PR[pUX + i] = 0.1 * r();
    double a[NO];
    long double b[NO];
    cell<double>(in, a);
    cell<long double>(in, b);
    for (int f = 0; f < NO; ++f) {
      const double e = (double)((long double)a[f] - b[f]), v = (double)b[f];
      e2[f] += e * e;
      v2[f] += v * v;
      rel[f] += v == 0.0 ? 0.0 : std::fabs(e / v) / n;
    }
  }
  for (int f = 0; f < NO; ++f) printf("%.3e %.3e\n", v2[f] > 0 ? std::sqrt(e2[f] / v2[f]) : 0.0, rel[f]);
}
