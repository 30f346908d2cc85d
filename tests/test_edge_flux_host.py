"""The fixed-point edge flux (csrc/dg_edgeint.cuh) compiled for the host, against
long double: which states it takes, and the error of those it takes.  The header's
integer arithmetic is the device's; only the two float32 estimates differ (correctly
rounded here, one or two units off there).  The driver is compiled with traps on
undefined integer arithmetic.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_07944_gb300", "csrc")

DRIVER = r'''
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include "dg_edgeint.cuh"
using namespace dg;
typedef long double Q;

struct Face { double sx, sy, hk, g1; FaceFix f; long long G1; int eg; };
static Face face(double h, double th, double gamma) {
  Face a;
  a.g1 = gamma - 1.0;
  a.sx = h * std::cos(th);
  a.sy = h * std::sin(th);
  a.hk = h * h * gamma * a.g1;
  a.f = face_fix(a.sx, a.sy, a.hk);
  a.eg = exponent_of(a.g1);
  a.G1 = fx::fixed_of(a.g1, a.eg);
  return a;
}
static bool flux(const double *L, const double *R, const Face &a, double *o) {
  return edge_flux_fixed(L, R, a.f, a.sx, a.sy, a.G1, a.eg, o);
}
// p / (gamma - 1) of a state, and how much of its energy it is
static Q pressure(const double *s) { return (Q)s[3] - ((Q)s[1] * s[1] + (Q)s[2] * s[2]) / (2 * (Q)s[0]); }

// The largest error of the four results, in units of 2^-50 (1 + E/P on both sides)
// times the sums of the magnitudes they are formed from: ten float64 roundings
// (2^-53 each), fixed-point steps below 2^-55 of the wave speed, and the pressure,
// whose error is below 2^-53 E.
static double error(const double *L, const double *R, const Face &a, const double *o) {
  const double *S[2] = {L, R};
  Q w[2], P[2], A[2], la = 0, amp = 1;
  for (int s = 0; s < 2; ++s) {
    w[s] = ((Q)S[s][1] * a.sx + (Q)S[s][2] * a.sy) / S[s][0];
    P[s] = pressure(S[s]);
    A[s] = std::fabs(w[s]) + std::sqrt((Q)a.hk * P[s] / S[s][0]);
    la = std::fmax(la, A[s]);
    amp += S[s][3] / P[s];
  }
  const Q wa = w[0] + la, wb = w[1] - la, ps = (P[0] + P[1]) * (Q)a.g1, h = std::hypot((Q)a.sx, (Q)a.sy);
  const Q pm = ((Q)L[3] + R[3]) * a.g1;
  double worst = 0;
  for (int k = 0; k < 4; ++k) {
    Q x = (Q)L[k] * wa + (Q)R[k] * wb, mag = (std::fabs((Q)L[k]) + std::fabs((Q)R[k])) * la;
    if (k == 1 || k == 2) {
      x += ps * (k == 1 ? a.sx : a.sy);
      mag = (std::hypot((Q)L[1], (Q)L[2]) + std::hypot((Q)R[1], (Q)R[2])) * la + pm * h;
    }
    if (k == 3) {
      x += (Q)a.g1 * (P[0] * w[0] + P[1] * w[1]);
      mag += pm * (std::fabs(w[0]) + std::fabs(w[1]));
    }
    const Q e = std::fabs((Q)o[k] - x) / (mag * amp * 0x1p-50L);
    if (!(e <= worst)) worst = (double)e;                  // (a NaN stays)
  }
  return worst;
}

static std::mt19937_64 rng(11);
static double U(double a, double b) { return a + (b - a) * ((rng() >> 11) * 0x1p-53); }
static void state(double *s, double rho, double c, double mach, double p_over_e_sign, double gamma) {
  const double a = U(0, 6.283185307179586), p = rho * c * c / gamma, q = mach * c;
  s[0] = rho;
  s[1] = rho * q * std::cos(a);
  s[2] = rho * q * std::sin(a);
  s[3] = 0.5 * rho * q * q + p_over_e_sign * p / (gamma - 1.0);
}

// states of one side without pressure: none may be taken
static int refuse() {
  long taken = 0, n = 0;
  double o[4];
  for (double m : {1.5, 2.0, 4.5, 5.0, 5.5, 5.8, 7.5, 7.9, 8.5, 11.0, 20.0})
    for (int side = 0; side < 2; ++side) {
      const double bad[4] = {1.0, m, 0.0, 1.0}, good[4] = {1.0, 0.1, 0.2, 1.0};
      const Face a = face(0.1, 0.3, 1.4);
      ++n;
      if (flux(side ? good : bad, side ? bad : good, a, o)) { ++taken; std::printf("m %g side %d\n", m, side); }
    }
  for (int i = 0; i < 400000; ++i) {
    const double gamma = U(1.05, 2.0), rho = std::exp(U(-40, 40)), e = std::exp(U(-40, 40));
    double s[2][4];
    for (int k = 0; k < 2; ++k) {
      s[k][0] = rho * U(1, 2);
      s[k][3] = e * U(1, 2);
      const double m = std::sqrt(2.0 * s[k][0] * s[k][3]) * (k == i % 2 ? std::exp(U(1e-12, 3.5)) : U(0, 0.9)), t = U(0, 6.28);
      s[k][1] = m * std::cos(t);
      s[k][2] = m * std::sin(t);
    }
    if (pressure(s[i % 2]) > -0x1p-50 * s[i % 2][3]) continue;
    const Face a = face(std::exp(U(-6, 1)), U(0, 6.28), gamma);
    ++n;
    taken += flux(s[0], s[1], a, o);
  }
  std::printf("non-physical %ld taken %ld\n", n, taken);
  return taken != 0 || n < 300000;
}

// physical states: the share taken, and the error of those
static int accuracy() {
  double worst = 0;
  long taken = 0, n = 0;
  for (int i = 0; i < 600000; ++i) {
    const double gamma = i % 3 ? 1.4 : U(1.1, 3.0), unit = i % 4 ? 1.0 : std::exp(U(-150, 150));
    const double rho = unit * std::exp(U(-2, 2)), c = std::exp(U(-3, 3)), mach = i % 5 ? std::exp(U(-12, 1.5)) : 0.0;
    const double jump = i % 6 == 0 ? 1.0 : i % 6 == 1 ? 0.0 : 1e-3;
    double L[4], R[4], o[4];
    state(L, rho, c, mach, 1.0, gamma);
    if (jump == 0.0) std::memcpy(R, L, sizeof R);
    else state(R, rho * std::exp(jump * U(-1, 1)), c * std::exp(jump * U(-1, 1)), mach * (1 + jump * U(-1, 1)), 1.0, gamma);
    const Face a = face(std::exp(U(-8, 1)), i % 7 ? U(0, 6.28) : 1.5707963267948966 * (i / 7 % 4), gamma);
    ++n;
    if (!flux(L, R, a, o)) continue;
    ++taken;
    const double e = error(L, R, a, o);
    if (!(e <= worst)) worst = e;
  }
  std::printf("physical %ld taken %ld worst %g\n", n, taken, worst);
  return !(worst < 1.0) || taken < 9 * n / 10;
}

// the square root over its whole range, denser towards both ends, and a flux whose
// sound speeds lie at the upper end: gas at rest with rho = 1, P just below 2 and a
// face with hk just below 1/4
static int root() {
  double worst = 0;
  for (int i = 0; i < 2000000; ++i) {
    const long long span = (1ll << 62) - (1ll << 58), r = (long long)(rng() % (unsigned long long)span) >> (i % 61);
    const long long v = i & 1 ? (1ll << 62) - 1 - r : (1ll << 58) + r;
    const Q e = std::fabs((Q)fx::sqrt_fixed(v) / (std::sqrt((Q)v) * 0x1p30L) - 1) / 0x1p-55L;
    if (!(e <= worst)) worst = (double)e;
  }
  double flux_worst = 0;
  for (int i = 0; i < 30; ++i) {
    const double u[4] = {1.0, 0.0, 0.0, 2.0 - std::ldexp(1.0, i - 50)};
    const double h = std::sqrt(0.25 * (1.0 - std::ldexp(1.0, i - 50)) / (1.4 * 0.4));
    const Face a = face(h, 0.3, 1.4);
    double o[4];
    if (!flux(u, u, a, o)) return 1;
    const double e = error(u, u, a, o);
    if (!(e <= flux_worst)) flux_worst = e;
  }
  std::printf("root worst %g 2^-55, flux worst %g\n", worst, flux_worst);
  return !(worst < 1.0) || !(flux_worst < 1.0);
}

// exponents over the whole range that the fixed point may take: whatever is taken is
// accurate (an error far below the smallest normal number counts for nothing)
static int range() {
  double worst = 0;
  long taken = 0;
  for (int i = 0; i < 1500000; ++i) {
    const double rho = std::ldexp(U(1, 2), (int)U(-302, 302)), e = std::ldexp(U(1, 2), (int)U(-302, 302));
    const double f = i % 3 == 0 ? U(0, 0.9) : std::exp(U(-700, 0)), gamma = 1.0 + std::exp(U(-8, 1));
    double s[2][4], o[4];
    for (int k = 0; k < 2; ++k) {
      s[k][0] = rho * U(1, 2);
      s[k][3] = e * U(1, 2);
      const double m = std::sqrt(s[k][0]) * std::sqrt(s[k][3]) * f * U(0.5, 1), t = U(0, 6.28);
      s[k][1] = m * std::cos(t);
      s[k][2] = i % 5 ? m * std::sin(t) : 0.0;
    }
    const Face a = face(std::ldexp(1.0, (int)U(-290, 290)), U(0, 6.28), gamma);
    if (!flux(s[0], s[1], a, o)) continue;
    ++taken;
    bool tiny = true;                                       // results below 2^-960: float64's own range ends here
    for (int k = 0; k < 4; ++k) tiny &= std::fabs(o[k]) < 0x1p-960;
    const double x = error(s[0], s[1], a, o);
    if (!tiny && !(x <= worst)) worst = x;
  }
  std::printf("taken %ld worst %g\n", taken, worst);
  return !(worst < 1.0) || taken < 300000;
}

int main(int argc, char **argv) {
  if (!std::strcmp(argv[1], "range")) return range();
  if (!std::strcmp(argv[1], "root")) return root();
  if (!std::strcmp(argv[1], "refuse")) return refuse();
  if (!std::strcmp(argv[1], "accuracy")) return accuracy();
  return 2;
}
'''


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("edge_flux")
    src, exe = d / "driver.cpp", d / "driver"
    src.write_text(DRIVER)
    gxx = shutil.which("g++")
    assert gxx, "g++ is part of the toolchain"
    subprocess.check_call([gxx, "-std=c++17", "-O1", "-fsanitize=undefined", "-fsanitize-undefined-trap-on-error",
                           "-I", CSRC, "-o", str(exe), str(src)])
    return str(exe)


@pytest.mark.parametrize("what", ["refuse", "accuracy", "root", "range"])
def test_edge_flux_fixed(driver, what):
    r = subprocess.run([driver, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout)
