"""The arithmetic of the collision and of the FP64 lines, compiled for the host and compared with long
double: the collision in fixed point is no further from it than the FP64 collision is, for every
speed class (small populations included) and from small to full relaxation, and stays bounded on
populations that span many decades; the FP32 collision keeps the momentum on average; derivative and
filter of a line in fixed point are no further off than the same even-odd products in FP64."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_19171_gb300", "csrc")

COLLISION = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <random>
#include "selbm_moments.cuh"
using namespace slb;
using L = long double;

template <int LAT>
void exact(const double *g, double omega, double dt, const double *acc, bool forced, L *out) {
  constexpr VelTab V = LT<LAT>::v;
  const L w2[4] = {4.L / 9, 1.L / 9, 1.L / 36, 0}, w19[4] = {1.L / 3, 1.L / 18, 1.L / 36, 0}, w27[4] = {8.L / 27, 2.L / 27, 1.L / 54, 1.L / 216};
  const L *w = LAT == SELBM_D2Q9 ? w2 : LAT == SELBM_D3Q19 ? w19 : w27;
  L d = 0, u[3] = {0, 0, 0}, F[3] = {0, 0, 0}, uu = 0, uF = 0;
  for (int a = 0; a < V.Q; ++a) {
    d += g[a];
    for (int k = 0; k < 3; ++k) u[k] += (L)V.e[a][k] * g[a];
  }
  for (int k = 0; k < V.D; ++k) {
    u[k] /= 1 + d;
    uu += u[k] * u[k];
    if (forced) F[k] = (1 + d) * (L)acc[k];
    uF += u[k] * F[k];
  }
  for (int a = 0; a < V.Q; ++a) {
    L eu = 0, eF = 0;
    for (int k = 0; k < 3; ++k) { eu += V.e[a][k] * u[k]; eF += V.e[a][k] * F[k]; }
    const L t = w[speed_class(V, a)], S = t * (9 * eu * eF - 3 * uF);
    const L feq = t * (d + (1 + d) * (3 * eu + 4.5L * eu * eu - 1.5L * uu)) - 0.5L * dt * S;
    out[a] = (L)g[a] - (L)omega * ((L)g[a] - feq) + (L)dt * S;
  }
}

template <int LAT>
struct Node {
  static constexpr VelTab V = LT<LAT>::v;
  static constexpr int Q = V.Q;
  double fp64[Q], fixed[Q];
  L ex[27], top = 0;
  Node(const double *g, double omega, bool forced) {
    const double dt = 0.01, acc[3] = {1e-3, 2e-3, V.D == 3 ? 5e-4 : 0.0};
    exact<LAT>(g, omega, dt, acc, forced, ex);
    for (int a = 0; a < Q; ++a) { fp64[a] = g[a]; top = std::max(top, std::max(fabsl(ex[a]), fabsl((L)g[a]))); }
    bgk_collide<double, LAT>(fp64, 1.0, omega, dt, 0.5 * dt, acc, forced);
    collide_fixed<LAT>(make_collide_fix<LAT>(omega, dt), 1.0, omega, dt, 0.5 * dt, acc, forced, [&](int a) { return g[a]; },
                       [&](int a, double v) { fixed[a] = v; });
  }
};

template <int LAT>
int check() {
  constexpr VelTab V = LT<LAT>::v;
  std::mt19937_64 r(LAT);
  std::normal_distribution<double> N;
  std::uniform_real_distribution<double> R(0, 1);
  int bad = 0;
  const double states[5][3] = {{0.05, 1e-3, 1e-4}, {0.002, 1e-4, 1e-5}, {0.02, 0.0, 0.0}, {1e-4, 1e-3, 1e-5}, {1e-6, 1e-8, 1e-9}};
  const double omegas[6] = {1.99, 1.4, 0.9, 0.3, 0.05, 0.003};
  for (const auto &st : states)
    for (double omega : omegas)
      for (int forced = 0; forced < 2; ++forced) {
        L e[2][4] = {}, n = 0;
        for (int it = 0; it < 1500; ++it) {
          double g[27], u[3], uu = 0;
          const double d = st[1] * N(r);
          for (int k = 0; k < 3; ++k) { u[k] = k < V.D ? st[0] * N(r) * (it % 3 == 0 && k ? 1e-6 : 1) : 0; uu += u[k] * u[k]; }
          for (int a = 0; a < V.Q; ++a) {
            double eu = 0;
            for (int k = 0; k < 3; ++k) eu += V.e[a][k] * u[k];
            g[a] = V.t[a] * (d + (1 + d) * (3 * eu + 4.5 * eu * eu - 1.5 * uu)) + V.t[a] * st[2] * N(r);
          }
          const Node<LAT> node(g, omega, forced);
          for (int a = 0; a < V.Q; ++a) {
            const int c = speed_class(V, a);
            const L x = ((L)node.fp64[a] - node.ex[a]) / node.top, y = ((L)node.fixed[a] - node.ex[a]) / node.top;
            e[0][c] += x * x;
            e[1][c] += y * y;
          }
        }
        // a percent for the sample: where omega is small both forms are the rounding of one addition
        for (int c = 0; c < 4; ++c)
          if (e[1][c] > e[0][c] * 1.01L) {
            std::printf("lattice %d class %d U %g omega %g forced %d: fixed %Lg fp64 %Lg\n", LAT, c, st[0], omega, forced, sqrtl(e[1][c]), sqrtl(e[0][c]));
            ++bad;
          }
      }
  // any populations: 53 bits of the value itself, and of the largest one the rounding of rho, u and the products
  // (|j| <= 9, 1 / rho <= 4, 4.5 t <= 1/2: below 2^8 units)
  for (int it = 0; it < 20000; ++it) {
    double g[27];
    const double top = std::pow(10.0, -R(r) * (it % 5 ? 4 : 300)), span = it % 2 ? 14 : 2;
    for (int a = 0; a < V.Q; ++a) g[a] = R(r) < 0.1 ? 0.0 : 0.2 * (R(r) - 0.5) * top * std::pow(10.0, -span * R(r));
    const Node<LAT> node(g, 2.0 * R(r) + 1e-4, false);
    for (int a = 0; a < V.Q; ++a)
      if (!(fabsl((L)node.fixed[a] - node.ex[a]) <= ldexpl(fabsl(node.ex[a]) + 256 * node.top, -53) + 1e-300L)) {
        std::printf("lattice %d population %d: %g for %Lg, largest %Lg\n", LAT, a, node.fixed[a], node.ex[a], node.top);
        if (++bad > 20) return bad;
      }
  }
  return bad;
}

int main() { return check<SELBM_D2Q9>() + check<SELBM_D3Q19>() + check<SELBM_D3Q27>() ? 1 : 0; }
"""

MOMENTUM = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <random>
#include "selbm_moments.cuh"
using namespace slb;

// change of momentum in the direction of j by one FP32 collision, relative to |j|: its mean over n
// nodes of random size is zero up to the spread of the roundings (6 standard errors)
template <int LAT>
int check(double U, double omega) {
  constexpr VelTab V = LT<LAT>::v;
  std::mt19937_64 r(LAT);
  std::normal_distribution<double> N;
  double sum = 0, sq = 0;
  const int n = 60000;
  for (int it = 0; it < n; ++it) {
    float g[V.Q];
    const float acc[3] = {0, 0, 0};
    const double u[3] = {U * std::exp(N(r)) * (it & 1 ? 1 : -1), 0.1 * U * N(r), V.D == 3 ? 0.1 * U * N(r) : 0}, d = 1e-4 * N(r);
    const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    for (int a = 0; a < V.Q; ++a) {
      double eu = 0;
      for (int k = 0; k < 3; ++k) eu += V.e[a][k] * u[k];
      g[a] = (float)(V.t[a] * (d + (1 + d) * (3 * eu + 4.5 * eu * eu - 1.5 * uu)) + V.t[a] * 1e-5 * N(r));
    }
    double before = 0, after = 0;
    for (int a = 0; a < V.Q; ++a) before += V.e[a][0] * (double)g[a];
    bgk_collide<float, LAT>(g, 1.f, (float)omega, 0.01f, 0.005f, acc, false);
    for (int a = 0; a < V.Q; ++a) after += V.e[a][0] * (double)g[a];
    const double c = (after - before) / before;
    sum += c;
    sq += c * c;
  }
  const double mean = sum / n, err = std::sqrt(sq) / n;
  if (std::fabs(mean) <= 6 * err) return 0;
  std::printf("lattice %d U %g omega %g: mean %g, standard error %g\n", LAT, U, omega, mean, err);
  return 1;
}
template <int LAT>
int all() { return check<LAT>(0.04, 1.99) + check<LAT>(0.04, 0.7) + check<LAT>(0.003, 1.9); }
int main() { return all<SELBM_D2Q9>() + all<SELBM_D3Q19>() + all<SELBM_D3Q27>() ? 1 : 0; }
"""

LINES = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <random>
#include <vector>
#include "selbm_fixed_lines.cuh"
using namespace slb;
using L = long double;
struct Host { const double *D, *w, *Vm, *Vinv, *fixed_sigma; };

template <int n>
struct Basis {
  double xi[n], D[n * n], V[n * n], Vi[n * n], w[n] = {};
  static double leg(int k, double x) {
    double a = 1, b = x;
    if (k == 0) return 1;
    for (int i = 2; i <= k; ++i) { const double c = ((2 * i - 1) * x * b - (i - 1) * a) / i; a = b; b = c; }
    return b;
  }
  Basis() {
    const int N = n - 1;
    for (int i = 0; i < n; ++i) {
      double x = -std::cos(std::acos(-1.0) * i / N);
      if (i && i < N)
        for (int it = 0; it < 60; ++it) x -= (x * leg(N, x) - leg(N - 1, x)) / (n * leg(N, x));
      xi[i] = x;
    }
    for (int i = 0; i <= N / 2; ++i) { const double t = (xi[i] - xi[N - i]) / 2; xi[i] = t; xi[N - i] = -t; }
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        L p = 0;
        if (i == j) {
          for (int k = 0; k < n; ++k)
            if (k != j) p += 1.L / ((L)xi[j] - xi[k]);
        } else {
          p = 1.L / ((L)xi[j] - xi[i]);
          for (int m = 0; m < n; ++m)
            if (m != i && m != j) p *= ((L)xi[i] - xi[m]) / ((L)xi[j] - xi[m]);
        }
        D[i * n + j] = (double)p;
        V[i * n + j] = j < 2 ? (j ? xi[i] : 1.0) : leg(j, xi[i]) - leg(j - 2, xi[i]);
      }
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) D[(N - i) * n + N - j] = -D[i * n + j];
    if (n & 1) D[(N / 2) * n + N / 2] = 0;
    L a[n][2 * n];
    for (int i = 0; i < n; ++i)
      for (int k = 0; k < n; ++k) { a[i][k] = V[i * n + k]; a[i][n + k] = i == k; }
    for (int c = 0; c < n; ++c) {
      int p = c;
      for (int r = c; r < n; ++r) if (fabsl(a[r][c]) > fabsl(a[p][c])) p = r;
      for (int k = 0; k < 2 * n; ++k) std::swap(a[c][k], a[p][k]);
      const L d = a[c][c];
      for (int k = 0; k < 2 * n; ++k) a[c][k] /= d;
      for (int r = 0; r < n; ++r)
        if (r != c) { const L f = a[r][c]; for (int k = 0; k < 2 * n; ++k) a[r][k] -= f * a[c][k]; }
    }
    for (int i = 0; i < n; ++i)
      for (int k = 0; k < n; ++k) Vi[i * n + k] = (double)a[i][n + k];
  }
};

template <int n>
int derivative() {
  const Basis<n> b;
  const Host h{b.D, b.w, nullptr, nullptr, nullptr};
  const StageMats<double, n> m = make_stage_mats<double, n>(h);
  std::mt19937_64 r(2);
  std::normal_distribution<double> G;
  constexpr int N = n - 1, SHIFT = FixScale<n>::SHIFT;
  L e0 = 0, e1 = 0;
  for (int it = 0; it < 3000; ++it) {
    double v[n], top = 0;
    const double a = G(r), c = G(r), k = 1 + 2 * std::fabs(G(r));
    for (int j = 0; j < n; ++j) { v[j] = 0.5 * a + c * std::sin(k * b.xi[j] + a); top = std::max(top, std::fabs(v[j])); }
    int em = kMinExp;
    for (int j = 0; j < n; ++j) { v[j] /= top; em = std::max(em, exp_of(v[j])); }
    long long q[n], d[n];
    for (int j = 0; j < n; ++j) q[j] = to_fixed<SHIFT>(v[j], em);
    line_deriv<n>(m, q, d);
    for (int j = 0; j < n; ++j) {
      L ex = 0;
      for (int i = 0; i < n; ++i) ex += (L)b.D[j * n + i] * v[i];
      const int jj = 2 * j <= N ? j : N - j;
      double se = 0, so = 0;
      for (int i = 0; i < n / 2; ++i) {
        const double x = b.D[jj * n + i], y = b.D[jj * n + N - i];
        se = std::fma(2 * jj == N ? 0.0 : 0.5 * (x + y), v[i] + v[N - i], se);
        so = std::fma(0.5 * (x - y), v[i] - v[N - i], so);
      }
      if ((n & 1) && 2 * jj != N) se = std::fma(b.D[jj * n + N / 2], v[N / 2], se);
      const L x0 = (L)(2 * j <= N ? so + se : se - so) - ex;
      const L x1 = (L)from_fixed(d[j], 61 - m.cb + em - FixScale<n>::EXP0) - ex;
      e0 += x0 * x0;
      e1 += x1 * x1;
    }
  }
  if (e1 <= e0) return 0;
  std::printf("derivative n = %d: fixed %Lg fp64 %Lg\n", n, sqrtl(e1), sqrtl(e0));
  return 1;
}

// three passes over a tile; the result is the value plus the tile's change
template <int n>
int filter(double gamma) {
  const Basis<n> b;
  double sg[n];
  const double kc = std::max(1, n - 3);
  for (int k = 0; k < n; ++k) { const double r = (k - kc) / (n - 1 - kc); sg[k] = k > kc ? 1 - gamma * r * r : 1; }
  const Host h{nullptr, b.w, b.V, b.Vi, sg};
  const FilterMats<double, n> m = make_filter_mats<double, n>(h);
  const int shift = filter_gain_shift(m, m.ex);
  long long g[n];
  for (int k = 0; k < n; ++k) g[k] = filter_gain(sg[k] - 1, shift);
  std::mt19937_64 r(3);
  std::normal_distribution<double> G;
  L e0 = 0, e1 = 0;
  for (int it = 0; it < 3; ++it) {
    std::vector<double> v(n * n * n), a;
    for (double &x : v) x = G(r);
    a = v;
    std::vector<L> x(v.begin(), v.end());
    int em = kMinExp;
    for (double y : v) em = std::max(em, exp_of(y));
    std::vector<long long> t;
    for (double y : v) t.push_back(to_fixed<kFilterShift>(y, em));
    for (int ax = 0, st = 1; ax < 3; ++ax, st *= n)
      for (int l = 0; l < n * n; ++l) {
        const int base = ax == 0 ? l * n : ax == 1 ? (l % n) + (l / n) * n * n : l;
        long long q[n];
        double o[n];
        L y[n];
        for (int k = 0; k < n; ++k) { q[k] = t[base + k * st]; o[k] = a[base + k * st]; y[k] = x[base + k * st]; }
        line_filter<n>(m, g, shift, q);
        for (int k = 2; k < n; ++k) {
          double s = 0;
          L S = 0;
          for (int j = 0; j < n; ++j) { s = std::fma(b.Vi[k * n + j], a[base + j * st], s); S += (L)b.Vi[k * n + j] * x[base + j * st]; }
          s *= sg[k] - 1;
          S *= (L)sg[k] - 1;
          for (int j = 1; j < n - 1; ++j) { o[j] = std::fma(b.V[j * n + k], s, o[j]); y[j] += (L)b.V[j * n + k] * S; }
        }
        for (int k = 1; k < n - 1; ++k) { t[base + k * st] = q[k]; a[base + k * st] = o[k]; x[base + k * st] = y[k]; }
      }
    for (size_t i = 0; i < v.size(); ++i) {
      const double f = v[i] + from_fixed(t[i] - to_fixed<kFilterShift>(v[i], em), em - (1023 + 52 + kFilterShift));
      e0 += ((L)a[i] - x[i]) * ((L)a[i] - x[i]);
      e1 += ((L)f - x[i]) * ((L)f - x[i]);
    }
  }
  if (e1 <= e0) return 0;
  std::printf("filter n = %d gamma %g: fixed %Lg fp64 %Lg\n", n, gamma, sqrtl(e1), sqrtl(e0));
  return 1;
}

template <int n>
int all() {
  int bad = derivative<n>();
  if constexpr (n > 3)
    for (double gamma : {0.01, 0.1, 0.5, 1.0}) bad += filter<n>(gamma);
  if constexpr (n < 15) return bad + all<n + 1>();
  else return bad;
}
int main() { return all<3>() ? 1 : 0; }
"""


def run_host(tmp_path, source):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    shutil.copy(os.path.join(ROOT, "tests", "fixed_point_host.h"), tmp_path / "cuda_runtime.h")
    (tmp_path / "main.cpp").write_text(source)
    exe = str(tmp_path / "main")
    subprocess.run([gxx, "-std=c++17", "-O2", "-w", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_collision(tmp_path):
    run_host(tmp_path, COLLISION)


def test_fp32_momentum(tmp_path):
    run_host(tmp_path, MOMENTUM)


def test_lines(tmp_path):
    run_host(tmp_path, LINES)
