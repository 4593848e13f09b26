"""What the integer functions' callers and loads rely on beyond their values
(csrc/fxmath.cuh), compiled for the host."""
import math
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_02904_gb300", "csrc")


def run(tmp_path, body, text=""):
    (tmp_path / "t.cpp").write_text(body)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")], check=True)
    return subprocess.run([str(tmp_path / "t")], input=text, capture_output=True, text=True, check=True).stdout


def test_logarithm_table_is_declared_for_its_16_byte_loads(tmp_path):
    # the declaration's alignment, not where a linker happened to put the table
    out = run(tmp_path, '#include "fxmath.cuh"\n#include <cstdio>\nint main() { printf("%zu", __alignof__(tgb::fx::kLog2)); }')
    assert int(out) % 16 == 0


FUNCTIONS = r"""
#include "fxmath.cuh"
#include <cstdio>
#include <cstdlib>
#include <cstring>
int main(int argc, char** argv) {
  namespace fx = tgb::fx;
  fx::host_jitter() = (float)atof(HOST_JITTER);
  char fn[16];
  double a;
  while (scanf("%15s %la", fn, &a) == 2) printf("%a\n", CALL);
}
"""


def evaluate(tmp_path, call, values, jitter=0.0):
    body = FUNCTIONS.replace("HOST_JITTER", f'"{jitter}"').replace("CALL", call)
    out = run(tmp_path, body, "".join(f"f {float(v).hex()}\n" for v in values))
    return [float.fromhex(r) for r in out.split()]


@pytest.mark.parametrize("jitter", [6e-7, -6e-7])
def test_reciprocals_up_to_the_stated_error_of_their_first_approximation(tmp_path, jitter):
    # 6e-7 and the cut argument's 2^-23 and a float rounding: 0.86 x 2^-20
    mpmath = pytest.importorskip("mpmath")
    mpmath.mp.dps = 50
    r = random.Random(21)
    v = [10 ** r.uniform(-30, 30) for _ in range(4000)] + [1.0, 2.0, 4.0, 3.9999999999999996, 1.9999999999999998]
    for call, want in (("fx::rcp(a)", lambda t: 1 / t), ("fx::rsqrt(a)", lambda t: 1 / mpmath.sqrt(t))):
        for a, got in zip(v, evaluate(tmp_path, call, v, jitter)):
            w = want(mpmath.mpf(a))
            assert abs(mpmath.mpf(got) - w) <= 0.625 * mpmath.mpf(2) ** (mpmath.frexp(w)[1] - 53), (call, a)


def test_reciprocal_and_square_root_are_correctly_rounded(tmp_path):
    # the adjoint's double divisions and square roots, against the host's IEEE ones
    r = random.Random(22)
    v = [math.ldexp(1 + r.getrandbits(52) * 2.0 ** -52, r.randrange(-1022, 1024)) for _ in range(60000)]
    v += [math.ldexp(m, e) for e in (-1022, -1, 0, 1, 2, 500, 1020, 1021, 1022, 1023)
          for m in (1.0, 1 + 2.0 ** -52, 2 - 2.0 ** -52, 1.5, 1 + 2.0 ** -26, 1.9999999)]
    v += [5e-324, 2.0 ** -1023, math.inf, 0.0]
    v += [float(k * k) for k in range(1, 2000)] + [3.0 * 2.0 ** -1024]
    for jitter in (0.0, 1.1e-7, -1.1e-7):
        w = v + [-a for a in v]
        for a, got in zip(w, evaluate(tmp_path, "fx::rcp(a)", w, jitter)):
            assert got == (1.0 / a if a else math.copysign(math.inf, a)), a
        for a, got in zip(v, evaluate(tmp_path, "fx::sqrt(a)", v, jitter)):
            assert got == math.sqrt(a), a


def test_logarithm_is_good_to_an_ulp_near_one_too(tmp_path):
    # an ulp is what CUDA's log states; away from 1 the fixed-point logarithm's 2^-55
    # is a quarter of an ulp of log(2), and the product and the rounding add 0.7
    mpmath = pytest.importorskip("mpmath")
    mpmath.mp.dps = 50
    r = random.Random(23)
    v = [1 + s * 2.0 ** r.uniform(-50, -1.01) for _ in range(3000) for s in (1, -1)]
    v += [r.uniform(0.4, 2.6) for _ in range(3000)] + [0.5, 2.0, 0.49999999999999994, 1.9999999999999998, 4.0, 1.0]
    for a, got in zip(v, evaluate(tmp_path, "fx::log(a)", v)):
        w = mpmath.log(mpmath.mpf(a))
        assert got == 0 if not w else abs(mpmath.mpf(got) - w) <= mpmath.mpf(2) ** (mpmath.frexp(w)[1] - 53), a
