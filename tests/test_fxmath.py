"""The FP64 path's integer elementary functions (csrc/fxmath.cuh), compiled for
the host, against many-digit arithmetic.

Bounds: each function rounds once to double (half an ulp) and carries a
relative error below 2^-56 (an eighth of an ulp) before that; the logarithm's
absolute error is below 2^-55. The bond order's arguments are rounded doubles:
(beta zeta) and 1/(2n) with half an ulp each, which the exponents n and
log(1 + u)/(2n) carry into the result.
"""
import os
import random
import subprocess

import pytest

mpmath = pytest.importorskip("mpmath")
mp, mpf = mpmath.mp, mpmath.mpf

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_02904_gb300", "csrc")

HARNESS = r"""
#include "fxmath.cuh"
#include <cstdio>
#include <cstdlib>
#include <cstring>
int main(int argc, char** argv) {
  namespace fx = tgb::fx;
  fx::host_jitter() = (float)atof(argv[1]);  // error of the float approximations
  char fn[16];
  double a, b, c, d;
  while (scanf("%15s %la", fn, &a) == 2) {
    double x = 0, y = 0;
    int ok = 1;
    if (!strcmp(fn, "bond")) {
      if (scanf("%la %la %la", &b, &c, &d) != 3) return 1;
      ok = fx::bond(a, b, c, d, &x, &y);
    } else if (!strcmp(fn, "sincospi")) fx::sincospi(a, &x, &y);
    else if (!strcmp(fn, "exp")) x = fx::exp(a);
    else if (!strcmp(fn, "log")) x = fx::log(a);
    else if (!strcmp(fn, "rcp")) x = fx::rcp(a);
    else x = fx::rsqrt(a);
    printf("%d %a %a\n", ok, x, y);
  }
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "t.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)

    def go(calls, jitter):
        text = "".join(f"{c[0]} {' '.join(float(v).hex() for v in c[1:])}\n" for c in calls)
        out = subprocess.run([str(d / "t"), str(jitter)], input=text, capture_output=True, text=True, check=True).stdout
        return [(int(a), float.fromhex(b), float.fromhex(c)) for a, b, c in (r.split() for r in out.splitlines())]

    return go


def ulps(got, want):
    """|got - want| in units of the last place of want as a double."""
    return float(abs(mpf(got) - want) / mpf(2) ** (mpmath.frexp(want)[1] - 53)) if want else (0.0 if got == 0 else 1e9)


@pytest.mark.parametrize("jitter", [0.0, 1.1e-7, -1.1e-7])  # the hardware's approximations are good to 2^-23
def test_functions_against_many_digits(evaluate, jitter):
    mp.dps = 50
    r = random.Random(7)
    edge = [1.0, 2.0, 4.0, 0.5, 0.25, 1.9999999999999998, 3.9999999999999996, 0.9999999999999999]
    calls = [(f, v) for f in ("rcp", "rsqrt", "log", "exp") for v in edge]
    calls += [("sincospi", v) for v in (0.5, 0.25, 0.24999999999999997, 0.49999999999999994, 0.0, 1e-12)]
    for _ in range(3000):
        calls += [("exp", r.choice([r.uniform(-31.9, 31.9), r.uniform(-1, 1) * 10 ** r.uniform(-20, 0)])),
                  ("log", r.choice([10 ** r.uniform(-18, 18), 1 + r.uniform(-0.05, 0.05)])),
                  ("rcp", r.choice([1, -1]) * 10 ** r.uniform(-30, 30)), ("rsqrt", 10 ** r.uniform(-30, 30)),
                  ("sincospi", min(0.5, r.choice([r.uniform(0, 0.5), 10 ** r.uniform(-9, -0.3)])))]
    for c, (ok, x, y) in zip(calls, evaluate(calls, jitter)):
        v = mpf(c[1])
        if c[0] == "exp":
            # the exponent argument x log2(e) carries 2^-57 absolute
            assert ulps(x, mpmath.exp(v)) <= 0.5 + 0.125, c
        elif c[0] == "log":
            want = mpmath.log(v)
            assert abs(mpf(x) - want) <= mpf(2) ** -55 + abs(want) * mpf(2) ** -53, c
        elif c[0] == "rcp":
            assert ulps(x, 1 / v) <= 0.625, c
        elif c[0] == "rsqrt":
            assert ulps(x, 1 / mpmath.sqrt(v)) <= 0.625, c
        elif c[1] >= 1e-9:
            assert ulps(x, mpmath.sin(mp.pi * v)) <= 0.625, c
            assert c[1] == 0.5 and abs(y) < 1e-15 or ulps(y, mpmath.cos(mp.pi * v)) <= 0.625, c


def test_bond_order_against_many_digits(evaluate):
    mp.dps = 50
    r = random.Random(8)
    calls = []
    for _ in range(3000):
        n = r.choice([0.78734, 0.72751, 1.0, r.uniform(0.3, 4.0), 22.956])
        calls.append(("bond", 10 ** r.uniform(-12, 8), 10 ** r.uniform(-7, 0), n, -1 / (2 * n)))
    calls += [("bond", 1e-300, 1e-7, 0.8, -0.625), ("bond", 1e30, 1.0, 22.0, -1 / 44), ("bond", 5e-324, 1.0, 1.0, -0.5),
              ("bond", 1.0, 0.0, 1.0, -0.5)]
    taken = 0
    for c, (ok, b, db) in zip(calls, evaluate(calls, 0.0)):
        if not ok:
            continue  # outside the formats: the caller's FP64 formulas
        taken += 1
        z, be, n = mpf(c[1]), mpf(c[2]), mpf(c[3])
        u = (be * z) ** n
        want = (1 + u) ** (-1 / (2 * n))
        dwant = -want * u / (2 * (1 + u) * z)
        e = abs(float(mpmath.log(want)))
        # half an ulp of 1/(2n) in the exponent, of beta zeta (n u/(2n(1+u)) <= 1/2 of it), 2^(en - 55) of n log, one rounding
        assert ulps(b, want) <= 1.0 + 2 * e + 0.5, c
        # d log u = n d log(beta zeta) in db
        assert ulps(db, dwant) <= 2.0 + 2 * e + 2 * float(n) + 0.5, c
    assert taken > 2000
    assert [v[0] for v in evaluate(calls, 0.0)][-4:] == [0, 0, 0, 0]
