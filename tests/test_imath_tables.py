"""The integer-arithmetic log and exp of the nodal states
(paper_2305_07181_gb300/csrc/imath.cuh): the committed tables are the
generator's output, and the functions, compiled for the host from the same
header, stay within the bounds the header states over random arguments, at
the ends of the log's table intervals and at the ends of their domains
(50-digit reference)."""
import importlib.util
import os
import random
import shutil
import subprocess

import pytest

mpmath = pytest.importorskip("mpmath")

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2305_07181_gb300", "csrc")

MAIN = r"""
#include "imath.cuh"
#include <cstdio>
using namespace esplit::im;
int main() {
  char f;
  unsigned long long a;
  while (std::scanf(" %c %llx", &f, &a) == 2) {
    long long X = 0;
    double x = __longlong_as_double((long long)a);
    if (f == 'l') { const bool ok = log_fixed(x, X); std::printf("%d %lld\n", (int)ok, X); }
    if (f == 'e') { const double y = exp_fixed((long long)a); std::printf("1 %lld\n", __double_as_longlong(y)); }
    if (f == 'd') { const double y = to_double((long long)a); std::printf("1 %lld\n", __double_as_longlong(y)); }
    if (f == 'f') { const bool ok = from_double(x, X); std::printf("%d %lld\n", (int)ok, X); }
  }
}
"""


def test_header_is_the_generator_output():
    spec = importlib.util.spec_from_file_location("gen_imath_tables", os.path.join(CSRC, "gen_imath_tables.py"))
    gen = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(gen)
    with open(os.path.join(CSRC, "imath_tables.h")) as f:
        assert gen.render() == f.read()


def _bits(x):
    import struct
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _double(b):
    import struct
    return struct.unpack("<d", struct.pack("<q", b))[0]


def test_functions_within_their_bounds(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "m.cpp"
    src.write_text(MAIN)
    exe = str(tmp_path / "m")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    rng = random.Random(4)
    logs = [2.0 ** -90, 2.0 ** 90 * (1 - 2.0 ** -53), 1.0, 1.0 - 2.0 ** -53, 1.0 + 2.0 ** -52]
    for j in range(257):
        c = 1.0 + j / 256.0
        logs += [c, c * (1 - 2.0 ** -53), c * (1 + 2.0 ** -52)]
    logs += [2.0 ** rng.uniform(-89.9, 89.9) for _ in range(4000)] + [rng.uniform(0.5, 2.0) for _ in range(4000)]
    out_of = [0.0, -1.0, 2.0 ** 90, 2.0 ** -91, float("inf"), float("nan")]
    exps = [0, 1, -1, 2 ** 63 - 1, -2 ** 63] + [rng.randrange(-2 ** 63, 2 ** 63) for _ in range(4000)] \
        + [rng.randrange(-2 ** 58, 2 ** 58) for _ in range(4000)]
    conv = [0.0, -0.0, 1e-300, 63.999999, -63.999999] + [rng.uniform(-64, 64) for _ in range(1000)]
    lines = [f"l {_bits(x):x}" for x in logs + out_of] + [f"e {x & (2 ** 64 - 1):x}" for x in exps] \
        + [f"d {x & (2 ** 64 - 1):x}" for x in exps[5:]] + [f"f {_bits(x):x}" for x in conv + [64.0, float("nan")]]
    got = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True, check=True).stdout.split()
    got = [(int(a), int(b)) for a, b in zip(got[::2], got[1::2])]
    assert len(got) == len(lines)
    mpmath.mp.dps = 50
    unit = mpmath.mpf(2) ** -57
    for x, (ok, X) in zip(logs, got):
        assert ok and abs(X * unit - mpmath.log(mpmath.mpf(x))) <= mpmath.mpf(2) ** -mpmath.mpf("55.5")
    at = len(logs)
    assert not any(ok for ok, _ in got[at:at + len(out_of)])
    at += len(out_of)
    for x, (_, b) in zip(exps, got[at:at + len(exps)]):
        y = mpmath.exp(x * unit)
        # half an ulp of rounding and 2^-56 of the series and its tables
        assert abs(mpmath.mpf(_double(b)) - y) <= y * mpmath.mpf(2) ** -53 * mpmath.mpf("1.2")
    at += len(exps)
    for x, (_, b) in zip(exps[5:], got[at:at + len(exps) - 5]):
        cut = max(0, abs(x).bit_length() - 53)  # to the nearest 53-bit integer, ties away from zero
        near = ((abs(x) + ((1 << cut) >> 1)) >> cut) << cut
        assert _double(b) == (-near if x < 0 else near) * 2.0 ** -57
    at += len(exps) - 5
    for x, (ok, X) in zip(conv, got[at:at + len(conv)]):
        assert ok and abs(X * unit - mpmath.mpf(x)) <= unit / 2
    assert not any(ok for ok, _ in got[at + len(conv):])
