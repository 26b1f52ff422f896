"""The double-float pair terms of csrc/lj_device.cuh, compiled for the CPU and measured in long
double: shortcuts in them (products that are not renormalised) cost no precision against the
same terms with every operation renormalised."""
import os
import re
import shutil
import subprocess

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2510_25938_gb300", "csrc", "lj_device.cuh")
FUNCS = ["ff_two_sum", "df_fast_two_sum", "df_two_prod", "df_add", "df_sub", "df_mul_raw",
         "df_add_f", "df_mul", "df_sqr", "df_rcp", "df_norm2", "df_sqrt", "df_exp",
         "pair_term_morse_df", "pair_term_df"]

PRELUDE = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
struct ff { float hi, lo; };
struct PosDF { float xh, yh, zh, wh, xl, yl, zl, wl; };
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float rsqrtf(float a) { return 1.0f / sqrtf(a); }
static float rcp_approx(float a) { return 1.0f / a; }
static float __int_as_float(int i) { float f; memcpy(&f, &i, 4); return f; }
"""

MAIN = r"""
typedef long double L;
static ff split(double x) { ff r; r.hi = (float)x; r.lo = (float)(x - (double)r.hi); return r; }
// every operation renormalised
static void plain(int pot, const PosDF& a, const PosDF& b, ff v[3], ff& e) {
  const ff d[3] = {df_sub(ff{a.xh, a.xl}, ff{b.xh, b.xl}), df_sub(ff{a.yh, a.yl}, ff{b.yh, b.yl}),
                   df_sub(ff{a.zh, a.zl}, ff{b.zh, b.zl})};
  const ff r2 = df_norm2(d[0], d[1], d[2]);
  ff c;
  if (pot) {
    const ff rho{6.f, 0.f}, r = df_sqrt(r2), ex = df_exp(df_sub(rho, df_mul(rho, r)));
    e = df_mul(ex, df_add_f(ex, -2.f));
    c = df_mul(df_mul(ex, df_add_f(ex, -1.f)), df_rcp(r));
  } else {
    const ff s2 = df_rcp(r2), s6 = df_mul(df_sqr(s2), s2), t = df_add_f(s6, -1.f);
    e = df_mul(s6, t);
    c = df_mul(df_mul(s2, s6), df_add(s6, t));
  }
  for (int k = 0; k < 3; ++k) v[k] = df_mul(c, d[k]);
}
int main(int, char** arg) {
  const int pot = arg[1][0] == '1';
  const double half = atof(arg[2]), dist = atof(arg[3]);
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(-1, 1);
  double se[2] = {0, 0}, sv[2] = {0, 0};
  for (int n = 0; n < 100000;) {
    double a[3], d[3], r = 0;
    for (int k = 0; k < 3; ++k) { a[k] = half * U(g); d[k] = U(g); r += d[k] * d[k]; }
    r = sqrt(r);
    if (r > 1 || r < 0.1) continue;
    ++n;
    const double t = dist * (1 + 0.05 * U(g));
    ff A[3], B[3];
    L D[3], r2 = 0;
    for (int k = 0; k < 3; ++k) {
      A[k] = split(a[k]);
      B[k] = split(a[k] + d[k] / r * t);
      D[k] = ((L)A[k].hi + A[k].lo) - ((L)B[k].hi + B[k].lo);
      r2 += D[k] * D[k];
    }
    const PosDF p{A[0].hi, A[1].hi, A[2].hi, 0, A[0].lo, A[1].lo, A[2].lo, 0};
    const PosDF q{B[0].hi, B[1].hi, B[2].hi, 0, B[0].lo, B[1].lo, B[2].lo, 0};
    const L R = sqrtl(r2), m = expl(6 * (1 - R)), s6 = 1 / (r2 * r2 * r2);
    const L e = pot ? m * (m - 2) : s6 * (s6 - 1), c = pot ? m * (m - 1) / R : s6 * (2 * s6 - 1) / r2;
    for (int w = 0; w < 2; ++w) {
      ff v[3], x;
      if (w) plain(pot, p, q, v, x);
      else if (pot) pair_term_morse_df(p, q, ff{6.f, 0.f}, v[0], v[1], v[2], x);
      else pair_term_df(p, q, v[0], v[1], v[2], x);
      const L de = (L)x.hi + x.lo - e;
      se[w] += de * de;
      for (int k = 0; k < 3; ++k) {
        const L dv = (L)v[k].hi + v[k].lo - c * D[k];
        sv[w] += dv * dv;
      }
    }
  }
  printf("%.6f %.6f\n", sqrt(se[0] / se[1]), sqrt(sv[0] / sv[1]));
}
"""


def _function(src, name):
    m = re.search(r"__device__ __forceinline__ [^\n;]*\b%s\([^;{]*\)\s*\{" % name, src)
    end, depth = m.end(), 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[end], 0)
        end += 1
    return src[m.start():end].replace("__device__ __forceinline__", "static")


@pytest.fixture(scope="module")
def ratios(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    with open(SRC) as f:
        src = f.read()
    consts = re.search(r"constexpr double kLn2 .*?kF7l = [^\n]*\n", src, re.S).group(0)
    code = PRELUDE + consts + "\n".join(_function(src, f) for f in FUNCS) + MAIN
    folder = tmp_path_factory.mktemp("df")
    path = os.path.join(folder, "t.cpp")
    with open(path, "w") as f:
        f.write(code)
    exe = os.path.join(folder, "t")
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-w", "-include", "cstdlib", path,
                    "-o", exe], check=True)
    return lambda *a: [float(v) for v in subprocess.run(
        [exe] + [str(x) for x in a], check=True, capture_output=True, text=True).stdout.split()]


@pytest.mark.parametrize("pot", [0, 1])
@pytest.mark.parametrize("half", [1.0, 3.0, 6.0])     # half the extent of the cluster, in sigma
@pytest.mark.parametrize("dist", [0.95, 1.12, 2.5])
def test_pair_terms_are_as_exact_as_renormalised_ones(ratios, pot, half, dist):
    """Ratios of the root mean squares of 10^5 errors, the same inputs on both sides: 2% is
    beyond their sampling; differences that are not renormalised cost 14 to 80%."""
    energy, vector = ratios(pot, half, dist)
    assert energy <= 1.02 and vector <= 1.02
