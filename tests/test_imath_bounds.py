"""Bounds stated in paper_2305_07181_gb300/csrc/imath.cuh for its logarithm,
compiled for the host, over random arguments of the whole domain and arguments
found by searching millions (50-digit reference)."""
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
    if (f == 'l') { const bool ok = log_fixed(x, X); std::printf("%d %lld\n", (int)ok, X); }
  }
}
"""


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


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
        text = "\n".join(f"{f} {_bits(x):x}" for x in xs)
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
