"""The fixed-point digit arithmetic of the tensor-core contraction
(paper_2305_07181_gb300/csrc/digits.h), compiled for the host: whole sums over
the directions, digit by digit, with the accumulators rounded to float32 after
every 16 nodes, against exact rational sums, for every operator size, with
ordinary and wide data, zero rows and columns, and digits at the end of their
range (the accumulators' exactness: sums next to 2^24).

Bound, as the header of tc64.cuh states it, per direction with A, X the powers
of two above the largest entries and u = 2^-53:
  q (X sum|D| + A sum|x|) + (n_p w + c) A X + u/4 sum|D||x|, and u |result| once,
six digits q = 2^-60, w = 2^-59, c = 2^-55 (a rounding and an alignment of the
integer sum, each within 2^-56); seven q = 2^-63, w = c = 2^-60."""
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_07181_gb300", "csrc")

MAIN = r"""
#include "digits.h"
#include <cstdio>
#include <cstdlib>
#include <vector>
using namespace esplit::tc;
static double rd() { unsigned long long b; if (std::scanf("%llx", &b) != 1) std::exit(3); return __longlong_as_double((long long)b); }
static int expo(const std::vector<double>& v) {
  unsigned mx = 0;
  for (double x : v) { unsigned h = (unsigned)((unsigned long long)__double_as_longlong(x) >> 32) & 0x7FFFFFFFu; if (h > mx) mx = h; }
  return exp_of_max(mx);
}
// the digits of an operator row through the packed storage, of a column directly
template <int B> static void digits_of_row(const std::vector<double>& v, int E, std::vector<int>* d) {
  for (size_t n = 0; n < v.size(); n += 2) {
    unsigned p[2][4];
    pack_half<B>(fixed_fields<B>(v[n], E), p[0][0], p[0][1], p[0][2], p[0][3]);
    pack_half<B>(fixed_fields<B>(n + 1 < v.size() ? v[n + 1] : 0.0, E), p[1][0], p[1][1], p[1][2], p[1][3]);
    unsigned f[digits_of(B)];
    unpack_fields<B>(p[0][0] | p[1][0] << 16, p[0][1] | p[1][1] << 16, p[0][2] | p[1][2] << 16, p[0][3] | p[1][3] << 16, f);
    for (int k = 0; k < digits_of(B); ++k)
      for (size_t h = 0; h < 2 && n + h < v.size(); ++h)
        d[k].push_back((int)((f[k] >> (16 * h)) & ((1u << B) - 1)) - (1 << (B - 1)));
  }
}
template <int NP, int D> static void run() {
  constexpr int B = bits_for(NP), G = digits_of(B), T = B == 10 ? 6 : 7, UNIT = B == 10 ? (D == 3 ? 62 : 61) : 69;
  long long S = 0;
  int ES = 0;
  for (int i = 0; i < D; ++i) {
    std::vector<double> a(NP), x(NP);
    for (double& v : a) v = rd();
    for (double& v : x) v = rd();
    const int Ea = expo(a), Ex = expo(x);
    std::vector<int> da[G], dx[G];
    digits_of_row<B>(a, Ea, da);
    for (double v : x) {
      const unsigned long long f = fixed_fields<B>(v, Ex);
      for (int k = 0; k < G; ++k) dx[k].push_back((int)((f >> ((G - 1 - k) * B)) & ((1u << B) - 1)) - (1 << (B - 1)));
    }
    float t[T], b[T];
    for (int k = 0; k < T; ++k) t[k] = b[k] = 0.0f;
    for (int n0 = 0; n0 < NP; n0 += 16)
      for (int p = 0; p < (G + 1) / 2; ++p)
        for (int j = 0; j < G; ++j)
          if (j + 2 * p < T) {
            long long s = 0, s1 = 0;
            for (int n = n0; n < n0 + 16 && n < NP; ++n) {
              s += (long long)da[j][n] * dx[2 * p][n];
              s1 += (long long)da[j][n] * dx[2 * p + 1 < G ? 2 * p + 1 : 2 * p][n];
            }
            t[j + 2 * p] = (float)((double)t[j + 2 * p] + (double)s);
            b[j + 2 * p] = (float)((double)b[j + 2 * p] + (double)s1);
          }
    int fine;
    const long long J = level_sum<B, UNIT, NP, T>(t, b, fine);
    if (i == 0) { S = J; ES = Ea + Ex - fine; } else add_direction(S, ES, J, Ea + Ex - fine);
  }
  std::printf("%llx\n", (unsigned long long)__double_as_longlong(level_value<B, UNIT>(S, ES)));
}
int main() {
  int np, d;
  while (std::scanf("%d %d", &np, &d) == 2) {
    if (np == 12 && d == 2) run<12, 2>();
    else if (np == 18) run<18, 2>();
    else if (np == 27) run<27, 2>();
    else if (np == 12) run<12, 3>();
    else if (np == 25) run<25, 3>();
    else if (np == 58) run<58, 3>();
    else if (np == 78) run<78, 3>();
    else return 4;
  }
}
"""

SIZES = [(12, 2), (18, 2), (27, 2), (12, 3), (25, 3), (58, 3), (78, 3)]


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("digits")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "m.cpp"), "-o", str(d / "m")], check=True)
    return str(d / "m")


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _value(h):
    return struct.unpack("<d", struct.pack("<Q", int(h, 16)))[0]


def _sums(exe, cases):
    lines = []
    for n_p, d, dirs in cases:
        lines.append(f"{n_p} {d}")
        for a, x in dirs:
            lines += [f"{_bits(v):x}" for v in a] + [f"{_bits(v):x}" for v in x]
    out = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True, check=True).stdout.split()
    assert len(out) == len(cases)
    return [_value(h) for h in out]


def _two_above(v):
    m = max(abs(Fraction(x)) for x in v)
    if m == 0:
        return Fraction(0)
    h = ((_bits(float(m)) >> 32) + 0x1100) >> 20
    return Fraction(2) ** (h - 1022)


def _data(kind, rng, n):
    if kind == "ordinary":
        return [rng.uniform(-1.0, 1.0) for _ in range(n)]
    if kind == "near constant":
        return [rng.choice([-3.0, 3.0])] * n if rng.random() < 0.5 else [1.0 + 1e-6 * rng.random() for _ in range(n)]
    if kind == "wide":
        return [rng.choice([-1, 1]) * 10.0 ** rng.uniform(-6, 6) for _ in range(n)]
    if kind == "one large":
        v = [rng.uniform(-1.0, 1.0) for _ in range(n)]
        v[rng.randrange(n)] *= 1e6
        return v
    if kind == "tiny and huge":
        s = 10.0 ** rng.uniform(-250, 140)
        return [s * rng.uniform(-1.0, 1.0) for _ in range(n)]
    if kind == "holes":
        return [rng.uniform(-1.0, 1.0) if rng.random() < 0.3 else 0.0 for _ in range(n)]
    raise ValueError(kind)


def _extreme(bits, digits, sign):
    # every digit at the end of its range, as far as a float64 holds them
    half = 1 << (bits - 1)
    X = sum((half if k else half - 1) << (bits * (digits - 1 - k)) for k in range(digits))
    return sign * float(X) * 2.0 ** -(bits * digits - 1)


@pytest.mark.parametrize("n_p,d", SIZES)
def test_sums_within_the_stated_bound(exe, n_p, d):
    rng = random.Random(100 * n_p + d)
    kinds = ["ordinary", "near constant", "wide", "one large", "tiny and huge", "holes"]
    cases = []
    for k in range(180):
        ka, kx = kinds[k % 6], kinds[(k // 6) % 6]
        if ka == kx == "tiny and huge":
            ka = "ordinary"
        cases.append((n_p, d, [(_data(ka, rng, n_p), _data(kx, rng, n_p)) for _ in range(d)]))
    digits = 6 if n_p <= 32 else 7
    for sa in (1, -1):
        for sx in (1, -1):
            a, x = [_extreme(10 if n_p <= 32 else 9, digits, s) for s in (sa, sx)]
            cases.append((n_p, d, [([a] * n_p, [x] * n_p)] * d))
    cases.append((n_p, d, [([0.0] * n_p, _data("wide", rng, n_p))] * d))
    cases.append((n_p, d, [(_data("wide", rng, n_p), [0.0] * n_p)] * d))
    u = Fraction(1, 2 ** 53)
    q, w, c = (Fraction(1, 2 ** 60), Fraction(1, 2 ** 59), Fraction(1, 2 ** 55)) if n_p <= 32 else \
        (Fraction(1, 2 ** 63), Fraction(1, 2 ** 60), Fraction(1, 2 ** 60))
    for (_, _, dirs), got in zip(cases, _sums(exe, cases)):
        exact = bound = Fraction(0)
        for a, x in dirs:
            A, X = _two_above(a), _two_above(x)
            sa, sx = sum(abs(Fraction(v)) for v in a), sum(abs(Fraction(v)) for v in x)
            exact += sum(Fraction(p) * Fraction(r) for p, r in zip(a, x))
            sab = sum(abs(Fraction(p) * Fraction(r)) for p, r in zip(a, x))
            bound += q * (X * sa + A * sx) + (n_p * w + c) * A * X + u / 4 * sab
        bound += u * abs(exact)
        assert abs(Fraction(got) - exact) <= bound


@pytest.mark.parametrize("n_p,d", SIZES)
def test_non_finite_entries_give_nan(exe, n_p, d):
    rng = random.Random(n_p)
    cases = []
    for bad in (float("nan"), float("inf"), -float("inf")):
        for other in ("ordinary", "zero"):
            o = [0.0] * n_p if other == "zero" else _data("ordinary", rng, n_p)
            v = _data("ordinary", rng, n_p)
            v[rng.randrange(n_p)] = bad
            good = [(_data("ordinary", rng, n_p), _data("ordinary", rng, n_p)) for _ in range(d - 1)]
            cases += [(n_p, d, [(v, o)] + good), (n_p, d, good + [(o, v)])]
    assert all(r != r for r in _sums(exe, cases))


@pytest.mark.parametrize("n_p,d", SIZES)
def test_sums_at_the_end_of_the_float64_range(exe, n_p, d):
    """Finite sums up to the largest float64 come out finite, and infinite ones
    from there on; below the normal range they are zero."""
    top, zero = 1.7976931348623157e308, ([0.0] * n_p, [0.0] * n_p)
    cases = []
    for f in (0.49, 0.51, 0.75, 0.999, 1.0, 1.01):     # of 2^1024: biased exponents 2045, 2046, beyond
        for s in (1.0, -1.0):
            x = [0.0] * n_p
            x[0], x[n_p - 1] = s * f * (top / 2), s * f * (top / 2)
            cases.append((n_p, d, [([1.0] * n_p, x)] + [zero] * (d - 1)))
    for v in (2.0 ** -1022, 2.0 ** -1023, 2.0 ** -1060):
        cases.append((n_p, d, [([v * 2.0 ** 500] * n_p, [2.0 ** -500] + [0.0] * (n_p - 1))] + [zero] * (d - 1)))
    got = _sums(exe, cases)
    for (_, _, dirs), r in zip(cases, got):
        a, x = dirs[0]
        want = sum(Fraction(p) * Fraction(v) for p, v in zip(a, x))
        if abs(want) > Fraction(top):
            assert r == (float("inf") if want > 0 else -float("inf"))
        elif abs(want) < Fraction(1, 2 ** 1022):
            assert r == 0.0
        else:
            assert abs(Fraction(r) - want) <= abs(want) / 2 ** 50
