// The degree-p reference element on the host: one-dimensional rules and bases, the order of the
// velocity dofs (ho_cells.cu and gauss_cells.cu form their tables from it).
#pragma once

#include <cmath>
#include <vector>

#include "ho_common.cuh"

namespace hmg {

// ---- reference tables, formed on the host ---------------------------------------------------
// n-point Gauss-Legendre rule on [0, 1]: Newton's method on the Legendre polynomial P_n from the
// initial guesses cos(pi (i + 3/4) / (n + 1/2)), weights 2 / ((1 - x^2) P_n'(x)^2) on [-1, 1],
// halved
static void gauss_legendre01(int n, double *x, double *w) {
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      // p1 = P_n(z), p0 = P_{n-1}(z) (n = 1: P_1 = z, P_0 = 1)
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    x[n - 1 - i] = 0.5 * (z + 1.0);   // ascending
    w[n - 1 - i] = 1.0 / ((1.0 - z * z) * dp * dp);
  }
}

// n = 2 .. 5 Gauss-Lobatto points on [0, 1]: the end points and the roots of P'_{n-1}
static void gauss_lobatto01(int n, double *x) {
  x[0] = 0.0;
  x[n - 1] = 1.0;
  if (n == 3) x[1] = 0.5;
  if (n == 4) {
    const double r = 1.0 / std::sqrt(5.0);
    x[1] = 0.5 * (1.0 - r);
    x[2] = 0.5 * (1.0 + r);
  }
  if (n == 5) {
    const double r = std::sqrt(3.0 / 7.0);
    x[1] = 0.5 * (1.0 - r);
    x[2] = 0.5;
    x[3] = 0.5 * (1.0 + r);
  }
}

static void lagrange1d(const double *nodes, int n, double x, double *val, double *der) {
  for (int i = 0; i < n; ++i) {
    double v = 1.0, d = 0.0;
    for (int j = 0; j < n; ++j)
      if (j != i) v *= (x - nodes[j]) / (nodes[i] - nodes[j]);
    for (int m = 0; m < n; ++m) {
      if (m == i) continue;
      double t = 1.0 / (nodes[i] - nodes[m]);
      for (int j = 0; j < n; ++j)
        if (j != i && j != m) t *= (x - nodes[j]) / (nodes[i] - nodes[j]);
      d += t;
    }
    val[i] = v;
    der[i] = d;
  }
}

// face f: the component normal to it, whether it is the far end (xi, eta or zeta = 1), the sign
// of the outward normal
static const int kFaceComp[6] = {1, 0, 1, 0, 2, 2};
static const int kFaceFar[6] = {0, 1, 1, 0, 0, 1};
static const double kFaceSign[6] = {-1.0, 1.0, 1.0, -1.0, -1.0, 1.0};

// a velocity dof: its component d, its node a along d (Gauss-Lobatto), its nodes (b, c) across d
// (Gauss-Legendre, the other two coordinates in increasing order), its sign
struct HoDof { int d, a, b, c; double sign; };

template <int P>
static std::vector<HoDof> ho_dofs() {
  using H = Ho<P>;
  std::vector<HoDof> v;
  for (int f = 0; f < 6; ++f)
    for (int s = 0; s < H::NT; ++s)
      for (int t = 0; t < H::NT; ++t) {
        const int b = (f == 2 || f == 3) ? P - s : s;   // e2, e3 traverse their edge backwards
        v.push_back({kFaceComp[f], kFaceFar[f] ? P + 1 : 0, b, t, kFaceSign[f]});
      }
  for (int d = 0; d < 3; ++d)
    for (int a = 1; a <= P; ++a)
      for (int b = 0; b < H::NT; ++b)
        for (int c = 0; c < H::NT; ++c) v.push_back({d, a, b, c, 1.0});
  return v;
}

}  // namespace hmg
