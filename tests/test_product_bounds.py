"""No GPU needed: the error bound of the double-precision ring products, from the twiddle factors that the kernels use.

csrc/d2mhe_fft.cuh states the bound; a program compiled from that header evaluates its twiddle factors, its constants and its
double-double arithmetic on the host, and the sum over the stages is formed here.  An error below one half means that every
product is exact, whatever the residue polynomial."""
import math
import os
import subprocess

import numpy as np
import pytest

from common import make_oracle, small_moduli

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_04604_b200", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <complex>
#include <cstdio>
#include <vector>
#include "d2mhe_fft.cuh"
typedef long double ld;
typedef std::complex<ld> C;
const ld PI2 = 6.283185307179586476925286766559005768L, U = 1.0L / 9007199254740992.0L;
static C ex(ld num, ld den) { return std::polar(1.0L, PI2 * num / den); }
static cpx rounded(ld num, ld den) { return {(double)cosl(PI2 * num / den), (double)sinl(PI2 * num / den)}; }
static ld err(cpx a, C e) { return std::abs(C(a.r, a.i) - e) / U; }
template <int R, int SGN> void pass(const char* name, int logn, int count, ld order, int sign) {
  ld worst[4] = {};
  for (int k = 0; k < count; ++k) {
    const cpx t[2] = {rounded(sign * k, order), rounded(sign * 4 * k, order)};
    const TwDerived<R, SGN> tw(t);
    static_for<(R == 8 ? 3 : 4)>([&](auto s_) {
      constexpr int lg = decltype(s_)::value + 1, L = 1 << lg;
      static_for<(L >= 4 ? L / 4 : 1)>([&](auto m_) {
        constexpr int m = decltype(m_)::value;
        const C e = ex((ld)sign * k * (R / L), order) * ex(SGN * m, L);
        worst[lg - 1] = std::max(worst[lg - 1], err(tw.template get<lg, m>(), e));
      });
    });
  }
  for (int s = 0; s < (R == 8 ? 3 : 4); ++s) printf("%s %d %.4Lf\n", name, logn, worst[s]);
}
template <int R, int GR> void twists(int logn) {
  const ld m = 256.0L * R, order = GR == 1 ? 4 * m : 8 * m;
  ld worst = 0;
  for (int g = 0; g < GR; ++g)
    for (int r = 0; r < 256; ++r)
      static_for<R>([&](auto j_) {
        constexpr int j = decltype(j_)::value;
        const ld f = g ? 3.0L : -1.0L;
        worst = std::max(worst, err(fft_twist<R, GR, j>(rounded(f * r, order), g), ex(f * (r + 256 * j), order)));
      });
  printf("twist %d %.4Lf\n", logn, worst);
}
// the same by the table of digits, which the inverse transform of two groups takes
static void digits(int logn) {
  ld worst = 0;
  for (int g = 0; g < 2; ++g)
    for (int r = 0; r < 256; ++r)
      for (int j = 0; j < 16; ++j) {
        const ld f = g ? 3.0L : -1.0L, order = 8 * 4096.0L;
        worst = std::max(worst, err(cmul(rounded(f * r, order), fft_digit(g, j)), ex(f * (r + 256 * j), order)));
      }
  printf("digits %d %.4Lf\n", logn, worst);
  constexpr cpx last = fft_digit(1, 15);  // a constant expression, as the kernels' table needs it
  printf("digit 0 %.17g\n", last.r + last.i);
}
// a transform of random ternary coefficients in double-double arithmetic against long double sums
static void exact(unsigned m) {
  const unsigned order = 8 * m;
  std::vector<ddc> coarse, fine, z(m);
  for (unsigned k = 0; k < order / FFT_ROOT_FINE; ++k) coarse.push_back(dd_root_entry(order, k * FFT_ROOT_FINE));
  for (unsigned k = 0; k < FFT_ROOT_FINE; ++k) fine.push_back(dd_root_entry(order, k));
  std::vector<C> in(m);
  unsigned x = 12345;
  auto draw = [&] { x = x * 1664525u + 1013904223u; return (double)((int)((x >> 16) % 3u) - 1); };
  for (unsigned j = 0; j < m; ++j) {
    const double a = draw(), b = draw();
    in[j] = C(a, b);
    z[j] = dd_cmul(ddc{dd{a, 0.0}, dd{b, 0.0}}, dd_root(coarse.data(), fine.data(), order, 2 * j));
  }
  for (unsigned len = m / 2; len; len /= 2)
    for (unsigned b = 0; b < m / 2; ++b) {
      const unsigned j = b % len, lo = b / len * 2 * len + j, hi = lo + len;
      const ddc s = dd_cadd(z[lo], z[hi]);
      z[hi] = dd_cmul(dd_csub(z[lo], z[hi]), dd_root(coarse.data(), fine.data(), order, j * (4 * m / len)));
      z[lo] = s;
    }
  std::vector<C> table(order);
  for (unsigned k = 0; k < order; ++k) table[k] = ex(k, order);
  ld worst = 0;
  for (unsigned p = 0; p < m; p += 37) {
    unsigned k = 0;
    for (unsigned b = 1; b < m; b *= 2) k = 2 * k + (p / b & 1);
    C e = 0;
    for (unsigned j = 0; j < m; ++j) e += in[j] * table[(2ull * j + 8ull * j * k) % order];
    const C got((ld)z[p].r.h + z[p].r.l, (ld)z[p].i.h + z[p].i.l);
    worst = std::max(worst, std::abs(got - e) / std::sqrt((ld)m) / U);
  }
  printf("exact %u %.4Lf\n", m, worst);
}
int main() {
  ld c = 0;
  for (int m = 0; m <= 32; ++m) c = std::max(c, err(cpx{cos64(m), cos64(32 - m)}, ex(m, 128)));
  printf("const 0 %.4Lf\n", c);
  pass<16, 1>("fwd", 12, 8, 128, 1), pass<16, 1>("fwd", 12, 128, 2048, 1);
  pass<16, -1>("inv", 12, 16, 256, -1), pass<8, -1>("inv", 12, 256, 2048, -1);
  for (int logn = 13; logn <= 14; ++logn) {
    pass<16, 1>("fwd", logn, 16, 256, 1), pass<16, 1>("fwd", logn, 256, 4096, 1);
    pass<16, -1>("inv", logn, 16, 256, -1), pass<16, -1>("inv", logn, 256, 4096, -1);
  }
  twists<8, 1>(12), twists<16, 1>(13), twists<16, 2>(14), digits(14);
  exact(2048), exact(4096);
  for (int logn = 12; logn <= 14; ++logn) {
    printf("units %d %.6f\n", logn, fft_error_units(logn));
    for (int m = 16; m <= 30; ++m)
      printf("key%d %d %.9f\npk%d %d %.9f\nconv%d %d %.9f\n", m, logn, fft_error(logn, m), m, logn, fft_error_pk(logn, m), m, logn,
             fft_error_conv(logn, m));
  }
  printf("KEY 0 %.6f\nPK 0 %.6f\nMU 0 %.6f\nV 0 %d\n", FFT_KEY_MAX, FFT_PK_MAX, FFT_MU_NORM, FFT_CONV_V);
}
"""


@pytest.fixture(scope="module")
def values(tmp_path_factory):
    d = tmp_path_factory.mktemp("bound")
    (d / "b.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(d / "b.cc"), "-o", str(d / "b")], check=True)
    out = {}
    for line in subprocess.run([str(d / "b")], check=True, capture_output=True, text=True).stdout.splitlines():
        name, logn, v = line.split()
        out.setdefault((name, int(logn)), []).append(float(v))
    return out


def _butterfly():
    """Largest error of a butterfly in units of u and of the 2-norm of its outputs: the error of U is at most
    (1 + a) |U| + b |V|, that of V one |V| more."""
    worst = 0.0
    for t in np.linspace(0, np.pi, 4001):
        a, b = abs(3 + np.exp(1j * t)) / 4, abs(1 - np.exp(1j * t)) / 4
        worst = max(worst, np.linalg.norm([[1 + a, b], [1 + a, b + 1]], 2))
    return worst + 1e-5


@pytest.mark.parametrize("logn", [12, 13, 14])
def test_sum_over_the_stages(values, logn):
    B, const = _butterfly(), values["const", 0][0]
    assert B < 2.941
    plain = 2 * 1.0 + (1 if logn == 12 else 2) * (B + const)  # a pass without twiddles: w = 1, w = i, then constants
    derived = {k: sum(B + e for e in values[k, logn]) for k in ("fwd", "inv")}
    twist = values["twist", logn][0]
    join = 1 + const if logn == 14 else 0.0
    forward = join + (2 + twist) + plain + derived["fwd"]
    key = 1.2  # of a stored transform, in units of the bound on its points
    product = B + 2  # its first stage forms the products
    back = product + 1 + 2 * (B + const) + derived["inv"]
    back += (2 + values["digits", logn][0]) + (2 + const) if logn == 14 else twist  # the rounding of the last sums is counted with the results
    assert forward + key + back <= values["units", logn][0]
    # Conversion: both products and their sum in the first stage; columns: what |c s| and |c' s'| of a pair add
    a, m = np.array([[8, 4], [9, 5]]), np.array([[6, 2], [7, 3]])
    assert np.linalg.norm(a, 2) / math.sqrt(2) - product < 5 and np.linalg.norm(m, 2) / math.sqrt(2) - product < 3


def test_double_double_transforms_are_good_at_every_point(values):
    """The reference sums are long double (2^-64 of terms of size one, at random), so what is seen is theirs: far below
    the 0.2 units of max_k |S_k| < 8.5 sqrt(N) that the bound leaves for it."""
    assert values["exact", 2048][0] < 0.1 and values["exact", 4096][0] < 0.1


def test_bounds_of_every_admitted_size(values):
    """Parts of the sizes that the splits give, with the rounding of their results, stay below one half."""
    for logn in (12, 13, 14):
        for bits in range(32, 57):
            h = min((bits + 1) // 2, 40 - logn)
            if bits - h > 28:
                continue
            m, rounding = max(h, bits - h), 2.0 ** -min(8, 32 - (bits - h))
            units = values["units", logn][0]
            want = units * 8.5 * 2.0 ** (m - 1 + logn - 53)
            assert abs(values["key%d" % m, logn][0] - want) < 1e-6 and want + rounding < 0.5
            assert values["pk%d" % m, logn][0] + rounding < 0.5
            half = (bits + 1) // 2
            assert values["conv%d" % half, logn][0] + 2.0 ** -min(8, 32 - (bits - half)) < 0.5
            # low results: 40 bits for ternary factors, 44 in Conversion
            assert 2 ** (logn + h - 1) <= 2 ** 39 and values["V", 0][0] * 2 ** (logn + half - 1) < 2 ** 43
        for bits in range(17, 31):
            fits = max(values["key%d" % bits, logn][0] if bits >= 16 else 0, values["pk%d" % bits, logn][0]) + 2.0 ** -6 < 0.5
            assert fits == (logn + bits <= 43)


def test_probabilities_that_the_bounds_leave(values):
    directions, n = 32, 8192
    c2 = math.cos(math.pi / directions) ** 2
    key, pk, mu = values["KEY", 0][0], values["PK", 0][0], values["MU", 0][0]
    assert math.log2(directions * n) - 1.5 * key ** 2 * c2 / math.log(2) < -135
    assert math.log2(directions * n) - 12 * pk ** 2 * c2 / math.log(2) < -110
    # |mu|_2^2 of N = 4096 Gaussian coefficients, sigma 3.2 cut at 19: Chernoff
    x = np.arange(-19, 20)
    w = np.exp(-(x / 3.2) ** 2 / 2)
    w /= w.sum()
    assert min(4096 * math.log2(float((w * np.exp(lam * (x ** 2 - mu ** 2))).sum())) for lam in np.linspace(0.001, 0.045, 45)) < -300
    assert values["V", 0][0] >= 1 + mu


@pytest.mark.parametrize("log2_n", [12, 14])
def test_keys_stay_far_below_the_bound(values, log2_n):
    n = 1 << log2_n
    moduli = small_moduli(log2_n, 36, 1)
    for seed in range(4):
        s = make_oracle(log2_n, moduli, seed=seed).secret_share(3).astype(np.float64)
        z = (s[: n // 2] + 1j * s[n // 2:]) * np.exp(1j * np.pi * np.arange(n // 2) / n)
        assert np.abs(np.fft.ifft(z) * (n // 2)).max() < 4.5 * math.sqrt(n) < values["KEY", 0][0] * math.sqrt(n)
