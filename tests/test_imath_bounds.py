"""Bounds of the functions of paper_2305_07181_gb300/csrc/imath.cuh, compiled for
the host, over random arguments of their whole domains, the ends of them, and
arguments found by searching millions (50-digit reference, exact integers).

Bounds of the series, relative, in units of 2^-53 (half an ulp of a result in
[1/2, 1) is one, of one in [1, 2) at most one): the rounding, and the float32
part's share of the sum times three float32 roundings --
  log1p_tail  1 + 2^53 2^-32 3 2^-24 = 1.4      expm1_tail  1 + 2^53 2^-31.3 3 2^-24 = 1.65
  atanhc      1 + 2^53 2^-36 3 2^-24 = 1.03     inv_atanhc  (below 1) the same
and a few units of 2^-62 from Horner's rule."""
import os
import random
import shutil
import struct
import subprocess

import pytest

mpmath = pytest.importorskip("mpmath")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_07181_gb300", "csrc")

MAIN = r"""
#include "imath.cuh"
#include <cstdio>
using namespace esplit::im;
int main() {
  char f;
  unsigned long long a;
  while (std::scanf(" %c %llx", &f, &a) == 2) {
    long long X = 0;
    const double x = __longlong_as_double((long long)a);
    if (f == 'L') { const bool ok = log_fixed62(x, X); std::printf("%d %lld\n", (int)ok, X); }
    if (f == 's') std::printf("1 %lld\n", small_to_fixed(x));
    if (f == 'u') std::printf("1 %lld\n", __double_as_longlong(unit62_to_double((long long)a)));
    if (f == 'p') std::printf("1 %lld\n", __double_as_longlong(log1p_tail(x)));
    if (f == 'm') std::printf("1 %lld\n", __double_as_longlong(expm1_tail(x)));
    if (f == 'a') std::printf("1 %lld\n", __double_as_longlong(atanhc(small_to_fixed(x))));
    if (f == 'i') std::printf("1 %lld\n", __double_as_longlong(inv_atanhc(small_to_fixed(x))));
    if (f == 'q') {
      unsigned long long c;
      if (std::scanf("%llx", &c) != 1) return 3;
      const bool ok = mul_q60((long long)a, (long long)c, X);
      std::printf("%d %lld\n", (int)ok, X);
    }
    if (f == 'l') { const bool ok = log_fixed(x, X); std::printf("%d %lld\n", (int)ok, X); }
  }
}
"""


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _double(b):
    return struct.unpack("<d", struct.pack("<q", b))[0]


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("imath")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "m.cpp"), "-o", str(d / "m")], check=True)
    mpmath.mp.dps = 50

    def call(f, xs):
        text = "\n".join(f"{f} " + (_bits(x).__format__("x") if isinstance(x, float) else
                                    " ".join(f"{v & (2 ** 64 - 1):x}" for v in (x if isinstance(x, tuple) else (x,))))
                         for x in xs)
        out = subprocess.run([str(d / "m")], input=text, capture_output=True, text=True, check=True).stdout.split()
        got = [(int(a), int(b)) for a, b in zip(out[::2], out[1::2])]
        assert len(got) == len(xs)
        return got

    return call


def test_log_fixed(run):
    rng = random.Random(2)
    xs = [float.fromhex(h) for h in ("0x1.eef4f3a5e200fp+73", "0x1.bfeb7a0ed002cp+76", "0x1.1fc6eeeca775bp+38")]
    xs += [2.0 ** rng.uniform(-90, 90) for _ in range(20000)] + [rng.uniform(0.5, 2.0) for _ in range(5000)]
    bound = mpmath.mpf(2) ** -mpmath.mpf("57.3")  # below the 2^-55.5 of a sum of separately rounded terms
    for x, (ok, X) in zip(xs, run("l", xs)):
        assert ok and abs(mpmath.mpf(X) / 2 ** 57 - mpmath.log(mpmath.mpf(x))) <= bound


def test_log_fixed62(run):
    rng = random.Random(3)
    xs = [0.25, 1.0, 1.0 - 2.0 ** -53, 1.0 + 2.0 ** -52, 4.0 - 2.0 ** -51, float.fromhex("0x1.01ffe335c78a5p+0")]
    xs += [2.0 ** rng.uniform(-2, 2) for _ in range(10000)] + [1.0 + rng.uniform(-1e-3, 1e-3) for _ in range(3000)]
    for x, (ok, X) in zip(xs, run("L", xs)):
        assert ok and abs(mpmath.mpf(X) / 2 ** 62 - mpmath.log(mpmath.mpf(x))) <= mpmath.mpf(2) ** -59
    outside = [0.25 - 2.0 ** -55, 4.0, 0.0, -1.0, float("inf"), float("nan")]
    assert not any(ok for ok, _ in run("L", outside))


def test_mul_q60(run):
    rng = random.Random(4)
    ab = [(rng.randrange(-2 ** 63, 2 ** 63), rng.randrange(-2 ** 63, 2 ** 63)) for _ in range(3000)]
    ab += [(rng.randrange(-2 ** 62, 2 ** 62), rng.randrange(-2 ** 61, 2 ** 61)) for _ in range(3000)]
    ab += [(s * 2 ** 62, t * 2 ** 60 + e) for s in (1, -1) for t in (1, -1) for e in (-1, 0, 1)]  # size 32
    for (a, b), (ok, out) in zip(ab, run("q", ab)):
        assert ok == (-2 ** 58 <= (a * b) >> 64 < 2 ** 58)   # |a b| / 2^60 below 32 in units of 2^-57
        if ok:
            assert out == (a * b) >> 60


def test_conversions(run):
    rng = random.Random(5)
    xs = [0.0, -0.0, 2.0 ** -4 - 2.0 ** -57, -(2.0 ** -4) + 2.0 ** -57, 2.0 ** -67, 5e-324]
    xs += [rng.choice([-1, 1]) * 2.0 ** rng.uniform(-70, -4) for _ in range(3000)]
    for x, (_, v) in zip(xs, run("s", xs)):
        assert v == int(mpmath.mpf(x) * 2 ** 66)              # toward zero
    ss = [1, 2 ** 62, 2 ** 63 - 1, 2 ** 54 - 1] + [rng.randrange(1, 2 ** 63) for _ in range(3000)]
    for s, (_, b) in zip(ss, run("u", ss)):
        cut = max(0, s.bit_length() - 53)                    # to the nearest, ties away from zero
        assert _double(b) == float(((s + ((1 << cut) >> 1)) >> cut) << cut) * 2.0 ** -62


@pytest.mark.parametrize("f,lo,hi,bound", [("p", -2.0 ** -5, 2.0 ** -5, 1.4), ("m", -2.0 ** -4, 2.0 ** -4, 1.65),
                                           ("a", 0.0, 1e-2, 1.05), ("i", 0.0, 1e-2, 1.05)])
def test_series(run, f, lo, hi, bound):
    rng = random.Random(6)
    end = lambda x: x * (1 - 2.0 ** -53)                     # the domains are open
    xs = [end(lo), end(hi), lo / 2, hi / 2, hi * 2.0 ** -20, lo * 2.0 ** -20]
    xs += [rng.uniform(end(lo), end(hi)) for _ in range(4000)] + [hi * 2.0 ** -rng.uniform(0, 60) for _ in range(2000)]
    mpmath.mp.dps = 60
    for x, (_, b) in zip(xs, run(f, xs)):
        z = mpmath.mpf(x)
        if abs(z) < mpmath.mpf(2) ** -40:   # first terms, the rest below 2^-80
            ref = {"p": 0.5 - z / 3, "m": 0.5 + z / 6, "a": 1 + z / 3, "i": 1 - z / 3}[f]
        elif f == "p":
            ref = (z - mpmath.log1p(z)) / z ** 2
        elif f == "m":
            ref = (mpmath.expm1(z) - z) / z ** 2
        else:
            r = mpmath.sqrt(z)
            ref = mpmath.atanh(r) / r
            ref = ref if f == "a" else 1 / ref
        assert abs(mpmath.mpf(_double(b)) - ref) <= bound * ref * mpmath.mpf(2) ** -53
