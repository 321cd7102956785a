"""The FP64 functions by integer arithmetic (csrc/fixed.cuh), compiled for the host, against
decimal arithmetic of 60 digits.

Bounds: combine_f64 and round_f64 round once (half an ulp, ties to even: equal to the nearest
double); fixed64 rounds to the nearest integer.  sigmoid_neg's error before its rounding is
below 2^-58 relative, so half an ulp and 2^-58 / 2^-53 = 1/32 of one in all."""

import decimal
import os
import random
import shutil
import subprocess
from decimal import Decimal
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <cinttypes>
#include "fixed.cuh"
using namespace kglm;
static const unsigned long long tab[64] = {KGLM_EXP2_TABLE};
int main() {
    char op;
    while (std::scanf(" %c", &op) == 1) {
        if (op == 's') {
            double t, e;
            if (std::scanf("%la", &t) != 1) return 1;
            const double q = sigmoid_neg(t, tab, &e);
            std::printf("%a %a %a\n", q, e, 1.0 / (1.0 + std::exp(t)));
        } else if (op == 'c') {
            int64_t H, L;
            int x;
            if (std::scanf("%" SCNd64 " %" SCNd64 " %d", &H, &L, &x) != 3) return 1;
            std::printf("%a\n", combine_f64(H, L, x));
        } else {
            double v;
            int e;
            if (std::scanf("%la %d", &v, &e) != 2) return 1;
            std::printf("%" PRId64 " %" PRId64 "\n", fixed64<64>(v, e), fixed64<48>(v, e));
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("fixed")
    (d / "t.cu").write_text(PROGRAM)
    subprocess.run([NVCC, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I",
                    os.path.join(ROOT, "paper_2605_22188_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(d / "t.cu"), "-o", str(d / "t")], check=True, capture_output=True)

    def go(lines):
        out = subprocess.run([str(d / "t")], input="\n".join(lines) + "\n", check=True, capture_output=True, text=True)
        return [line.split() for line in out.stdout.splitlines()]
    return go


def _ulps(got, want):
    """|got - want| in units of got's last place (want: Decimal)."""
    f = Decimal(got)
    u = Decimal(2) ** (max(-1074, _exponent(got) - 52))
    return abs(f - want) / u


def _exponent(v):
    import math
    return math.frexp(v)[1] - 1 if v else -1074


def test_sigmoid(run):
    rng = random.Random(1)
    args = [0.0, -0.0, 5e-324, 2.0 ** -60, -2.0 ** -60, 708.0, -708.0, 0.5, -0.5]
    args += [rng.uniform(-708, 708) for _ in range(2000)] + [rng.uniform(-40, 40) for _ in range(2000)]
    args += [rng.choice([-1, 1]) * 2.0 ** rng.uniform(-60, 9) for _ in range(2000)]
    # around the table's entries and the middles between them, where N changes
    args += [(j + h + rng.uniform(-1e-9, 1e-9)) * 0.010830424696249145 for j in range(-300, 300) for h in (0.0, 0.5)]
    worst = [0, 0, 0]
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        ctx.Emin, ctx.Emax = -9999, 9999
        for t, (q, e, lib) in zip(args, run(["s %s" % float(t).hex() for t in args])):
            et = Decimal(t).exp()
            want = 1 / (1 + et)
            for i, (got, ref) in enumerate(((q, want), (e, et), (lib, want))):
                worst[i] = max(worst[i], _ulps(float.fromhex(got), ref))
    print("worst ulp: sigmoid %.4f, exponential %.4f; exp, addition and division in FP64 %.2f" % tuple(worst))
    assert worst[0] <= 0.5 + 1 / 32 and worst[1] <= 0.5 + 1 / 32


def test_combine_rounds_once(run):
    rng = random.Random(2)
    cases = [(0, 0, 5), (1, 0, -72), (-1, 0, -72), (0, -1, 0), (1 << 61, -(1 << 62), -72), (-(1 << 61), 1 << 62, 40)]
    for _ in range(5000):
        H = rng.getrandbits(rng.randint(1, 62)) * rng.choice([-1, 1])
        L = rng.getrandbits(rng.randint(1, 62)) * rng.choice([-1, 1])
        cases.append((H, L, rng.choice([-72, rng.randint(-400, 400)])))
    for _ in range(3000):                                    # halfway between two doubles, and one off it
        m, s = rng.getrandbits(53) | (1 << 52), rng.randint(1, 40)
        v = (m << s) + (1 << (s - 1)) + rng.choice([-1, 0, 1])
        lo = v & 0xffffffff
        cases.append((v >> 32, lo, rng.randint(-200, 200)))
    for _ in range(1000):                                    # subnormal and overflowing results
        cases.append((rng.getrandbits(60), rng.getrandbits(60) - (1 << 59), rng.choice([rng.randint(-1200, -1060),
                                                                                    rng.randint(920, 1000)])))
    for (H, L, x), (got,) in zip(cases, run(["c %d %d %d" % c for c in cases])):
        v = Fraction(H * 2 ** 32 + L) * Fraction(2) ** x
        try:
            want = float(v)                                  # correctly rounded
        except OverflowError:
            want = float("inf") if v > 0 else float("-inf")
        assert float.fromhex(got) == want, (H, L, x, got, want.hex())


def test_fixed_point_rounds_to_nearest(run):
    rng = random.Random(3)
    cases = [(0.0, 3), (5e-324, -1000), (1.0 - 2.0 ** -53, 1), (-(1.0 - 2.0 ** -53), 1)]
    for _ in range(5000):
        e = rng.randint(-300, 300)
        cases.append((rng.choice([-1, 1]) * rng.uniform(0.5, 1) * 2.0 ** (e - 1 - rng.randint(0, 70)), e))
    for (v, e), got in zip(cases, run(["f %s %d" % (float(v).hex(), e) for v, e in cases])):
        for bits, z in zip((64, 48), map(int, got)):
            exact = Fraction(v) * Fraction(2) ** (bits - e)
            assert abs(z - exact) <= Fraction(1, 2), (v, e, bits, z)
