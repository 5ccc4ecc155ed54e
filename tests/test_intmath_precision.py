"""The errors of the FP64 walk's elementary functions before and at their last
rounding, on the arguments where they peak.

Tolerances, in units of the last place kept before the rounding:
  * -ln(1 - u): the only roundings that reach the sum are r^2's (half a unit of
    2^-63, times |P| = 1/2) and the last one.  The smallest results of the table
    path, from 2^-9 on, have an ulp of 2^-61, so the error is at most 0.5 + 0.25/4
    ulp, and 0.57 with the truncated terms of the series.
  * sin, cos: two floored products of opposite sign (within one unit of 2^-62
    together), 1 - cos(delta) (its coefficient within half a unit of 2^-36, times
    delta^4 < 2^-25.4: 0.8 units; floors 0.5) and sin(delta) (Q68): below 3 units.
  * 1/a: y's two floors and one rounded factor, and the neglected square of 1 - m y
    (below one unit): 2 units of 2^-62, so 0.5 + 2/512 ulp.
  * sqrt: 1 - v y^2 within half a unit of 2^-58, so 2 units of 2^-61, the
    neglected 3/8 (1 - v y^2)^2 and the floor of v y: 4 units of 1/256 ulp together.
"""
from __future__ import annotations

import os
import random
import shutil
import subprocess
from decimal import Decimal, getcontext

import pytest

from tests.test_intmath_host import dec_pi, dec_sin_cos

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1708_00765_gb300", "csrc")

PROGRAM = r"""
#define CLS_TABLE_SPACE
#include "cls_intmath.h"
#include <cstdio>
#include <cstring>
typedef unsigned __int128 u128;
static unsigned long long rng = 88172645463325252ull;
static unsigned long long next() {
    rng ^= rng << 13;
    rng ^= rng >> 7;
    rng ^= rng << 17;
    return rng * 0x2545F4914F6CDD1Dull;
}
static unsigned long long mantissa(double v, int *e) {  // v = m 2^e, m of 53 bits
    unsigned long long b;
    std::memcpy(&b, &v, 8);
    *e = (int)(b >> 52) - 1075;
    return (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
}
int main(int argc, char **argv) {
    if (argc > 1) {  // worst errors of 1/a and sqrt, in ulps, from exact products
        double wr = 0, wq = 0;
        for (long i = 0; i < 3000000; ++i) {
            const int low = (int)(next() % 52);
            const double a = 1.0 + (double)((i & 1) ? next() >> 12 : (1ull << 52) - 1 - ((next() >> 12) >> low)) * 0x1p-52;
            int ea, ev;
            const unsigned long long A = mantissa(a, &ea), V = mantissa(cls::recip_int(a), &ev);
            // V A 2^(ea + ev) - 1 in units of A 2^ev
            const u128 p = (u128)V * A, one = (u128)1 << (-ea - ev);
            const double er = (double)(p > one ? p - one : one - p) / (double)A;
            wr = er > wr ? er : wr;
            // sqrt(4 u (1 - u)), u = k 2^-53, = sqrt(X) 2^-53
            const unsigned long long k = (next() >> 11) | 1, n = (1ull << 53) - k;
            const u128 X = (u128)k * n * 4;
            int eq;
            unsigned long long Q = mantissa(cls::sqrt_int(cls::U128{(uint64_t)X, (uint64_t)(X >> 64)}, 106), &eq);
            eq += 53;  // sqrt(X) = Q 2^eq, eq <= 0
            const u128 q2 = (u128)Q * Q;
            if (-2 * eq > 127 - 106 && (X >> (127 + 2 * eq)) != 0) continue;  // X 2^(-2 eq) beyond 128 bits
            const u128 x = X << (-2 * eq);
            const double e = (double)(q2 > x ? q2 - x : x - q2) / (2.0 * (double)Q);
            wq = e > wq ? e : wq;
        }
        std::printf("%.6f %.6f\n", wr, wq);
        return 0;
    }
    cls::IntLogTables tab{cls::cls_log_n_init, cls::cls_log_t_init};
    unsigned long long k;
    while (std::scanf("%llu", &k) == 1) {
        int64_t s, c;
        cls::sincos_2pi_q62(k, cls::cls_sincos_q62_init, &s, &c);
        std::printf("%a %lld %lld\n", cls::exp_variate(k, tab), (long long)s, (long long)c);
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("precision")
    src, exe = d / "t.cc", d / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(ks):
        out = subprocess.run([str(exe)], input="\n".join(map(str, ks)), capture_output=True, text=True,
                             check=True).stdout.split("\n")
        return [line.split() for line in out[:len(ks)]]

    run.exe = str(exe)
    return run


def test_exp_variate_error_at_its_smallest_table_results(program):
    import math
    getcontext().prec = 40
    rnd = random.Random(21)
    ks = [2**44 + rnd.getrandbits(43) for _ in range(20000)]
    two53 = Decimal(2) ** 53
    worst = 0.0
    for k, (v, _, _) in zip(ks, program(ks)):
        v = float.fromhex(v)
        ref = -((two53 - k) / two53).ln()
        worst = max(worst, float(abs(Decimal(v) - ref) / Decimal(math.ulp(v))))
    assert worst <= 0.57, worst


def test_sincos_error_before_the_rounding(program):
    getcontext().prec = 40
    rnd = random.Random(22)
    # next to the midpoints between the tabulated angles, where delta is largest
    ks = [j * 2**45 + 2**44 - 1 - rnd.getrandbits(40) for j in range(256) for _ in range(20)]
    ks += [rnd.getrandbits(53) for _ in range(2000)]
    two_pi, scale = 2 * dec_pi(), Decimal(2) ** 62
    worst = 0.0
    for k, (_, s, c) in zip(ks, program(ks)):
        a = two_pi * k / Decimal(2) ** 53
        rs, rc = dec_sin_cos(a - two_pi if a > dec_pi() else a)
        worst = max(worst, float(abs(int(s) - rs * scale)), float(abs(int(c) - rc * scale)))
    assert worst <= 3.0, worst


def test_reciprocal_and_square_root_errors(program):
    out = subprocess.run([program.exe, "worst"], capture_output=True, text=True, check=True).stdout.split()
    recip, root = map(float, out)
    assert recip <= 0.5 + 2 / 512, recip
    assert root <= 0.5 + 4 / 256, root
