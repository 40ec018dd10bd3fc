"""The arithmetic of the collision, compiled for the host and compared with long
double: the collision in fixed point is no further from it than the FP64 collision is, for every
speed class (small populations included) and from small to full relaxation, and stays bounded on
populations that span many decades; the FP32 collision keeps the momentum on average."""
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
