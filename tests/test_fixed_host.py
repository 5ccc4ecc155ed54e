"""cls_fixed.h, the FP64 walk's 96-bit fixed point, compiled for the host and checked against
Python's integers."""
from __future__ import annotations

import math
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1708_00765_gb300", "csrc")
FIXED_NONE = 4000

PROGRAM = r"""
#define CLS_TABLE_SPACE
#include "cls_fixed.h"
#include <cstdio>
#include <cstdlib>
using namespace cls;
static void put(const Fix96 &q) { std::printf("%u %u %u\n", q.w0, q.w1, q.w2); }
int main() {
    char op, a[64], b[64];
    while (std::scanf(" %c", &op) == 1) {
        if (op == 'f') {  // value, F
            int F;
            if (std::scanf("%63s %d", a, &F) != 2) return 1;
            put(fixed96(std::strtod(a, nullptr), F));
        } else if (op == 'm' || op == 's' || op == 'a' || op == 'd') {  // fraction, a - b, a + b, to double
            unsigned long long f;
            Fix96 q, p;
            if (std::scanf("%llu %u %u %u %u %u %u", &f, &q.w0, &q.w1, &q.w2, &p.w0, &p.w1, &p.w2) != 7) return 1;
            if (op == 'd') std::printf("%a\n", fix96_to_double(q));
            else put(op == 'm' ? fraction96(f, q) : op == 's' ? sub96(q, p) : add96(q, p));
        } else {  // fraction bits of (dx, sigma0, sigma1, lambda0, lambda1)
            double v[5];
            for (double &x : v) {
                if (std::scanf("%63s", b) != 1) return 1;
                x = std::strtod(b, nullptr);
            }
            const double sg[2] = {v[1], v[2]}, la[2] = {v[3], v[4]};
            std::printf("%d\n", fixed_bits(v[0], sg, la));
        }
    }
}
"""


@pytest.fixture(scope="module")
def fixed(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("fixed")
    src, exe = d / "t.cc", d / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(lines):
        return subprocess.run([str(exe)], input="\n".join(lines), capture_output=True, text=True,
                              check=True).stdout.strip().split("\n")
    return run


def words(q):
    return f"{q & 0xffffffff} {(q >> 32) & 0xffffffff} {q >> 64}"


def value(line):
    w = list(map(int, line.split()))
    return w[0] | w[1] << 32 | w[2] << 64


def test_conversion_is_the_floor_at_every_scale(fixed):
    rnd = random.Random(1)
    cases = [(0.0, 64), (5e-324, 64), (1.0, 64), (math.nextafter(2.0**26, 0), 64), (2.0**-64, 64), (2.0**-65, 64)]
    for F in (64, 65, 77, 90, 91, 128, 400):
        for _ in range(400):
            cases.append((rnd.uniform(1, 2) * 2.0 ** (89 - F - rnd.randint(0, 100)), F))
    got = fixed([f"f {v.hex()} {F}" for v, F in cases])
    for (v, F), line in zip(cases, got):
        n, d = v.as_integer_ratio()
        assert value(line) == (n << F) // d, (v, F)


def test_fractions_sums_and_doubles(fixed):
    rnd = random.Random(2)
    rows = []
    for _ in range(2000):
        f = rnd.choice((rnd.getrandbits(64), rnd.getrandbits(rnd.randint(1, 64)), 2**64 - 1, 0, 2**32 - 1))
        q = rnd.choice((rnd.getrandbits(rnd.randint(1, 90)), 2**90 - 1, 2**64 - 1))
        p = rnd.getrandbits(96)
        rows.append((f, q, p))
    for op in "msad":
        got = fixed([f"{op} {f} {words(q)} {words(p)}" for f, q, p in rows])
        for (f, q, p), line in zip(rows, got):
            if op == "m":
                assert 0 <= (f * q >> 64) - value(line) <= 3
            elif op == "s":
                assert value(line) == (q - p) % 2**96
            elif op == "a":
                assert value(line) == (q + p) % 2**96
            else:
                v = float.fromhex(line)
                assert abs(int(v) - q) <= (0 if q < 2**53 else math.ulp(v))


def test_fraction_bits_follow_the_mean_flight(fixed):
    """The unit is below 2^-55 of the flights that make up the sums, and 2^34 of them still fit."""
    rnd = random.Random(3)
    rows = [(rnd.choice((1.0, 0.05, 1e-3)) * 10.0 ** rnd.randint(0, 30), 10.0 ** rnd.uniform(-3, 3), 10.0 ** rnd.uniform(-3, 3),
             10.0 ** rnd.uniform(-3, 3), 10.0 ** rnd.uniform(-3, 3)) for _ in range(500)]
    got = fixed(["b " + " ".join(x.hex() for x in r) for r in rows])
    for (dx, s0, s1, l0, l1), line in zip(rows, got):
        F, t = int(line), (1 / (s0 + 1 / l0), 1 / (s1 + 1 / l1))
        flight = min(max(t[0], t[1] / (1 + s0 * l0)), max(t[1], t[0] / (1 + s1 * l1)))
        assert F >= 64 and dx * 2.0**-F <= 2.0**-55 * flight
        assert F == 64 or dx * 2.0 ** (90 - F) >= 2.0**33 * flight
    # flights that no unit above the subnormal doubles can hold, and a bin width whose reciprocal overflows
    for r in ((1e300, 1e300, 1e300, 1.0, 1.0), (1e-310, 1.0, 1.0, 1.0, 1.0), (1.0, 0.0, 0.0, 5e-324, 5e-324)):
        assert fixed(["b " + " ".join(x.hex() for x in r)]) == [str(FIXED_NONE)], r
