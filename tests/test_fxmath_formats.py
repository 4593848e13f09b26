"""What the integer functions' callers and loads rely on beyond their values
(csrc/fxmath.cuh), compiled for the host."""
import math
import os
import random
import shutil
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


PAIR = r"""
#include "tersoff_fx.cuh"
#include "params_fx.cu"
#include <cstdio>
using namespace tgb;
int main() {
  double A, B, l1, l2, beta, n, c, d, h, r, zeta;
  while (scanf("%la %la %la %la %la %la %la %la %la %la %la", &A, &B, &l1, &l2, &beta, &n, &c, &d, &h, &r, &zeta) == 11) {
    Ctx x;
    x.ns = 1;
    x.rmax_cut = 3.0;
    x.h_rec64.assign(RSTRIDE, 0.0);
    double* o = x.h_rec64.data();
    o[K_A] = A, o[K_B] = B, o[K_LAM1] = l1, o[K_LAM2] = l2, o[K_BETA] = beta, o[K_N] = n;
    o[K_GAMMA] = 1.0, o[K_H] = h, o[K_D2] = d * d, o[K_GC2D2] = c * c / (d * d), o[K_G2C2] = 2 * c * c;
    make_fx_records(&x);
    if (!x.fx_ok) return 1;
    const fx::Mant m = fx::unpack(r);
    double fr = 0, bfa = 0, dz = 0;
    const int ok = fx::pair64(x.h_fx[0], m.m, m.e, zeta, &fr, &bfa, &dz);
    printf("%d %a %a %a\n", ok, fr, bfa, dz);
  }
}
"""


@pytest.mark.parametrize("element", ["Si", "C"])
def test_pair_term_takes_every_zeta_of_real_neighbourhoods(tmp_path, element):
    """Below n = 1 too the integer formats hold the whole range (n log2(beta zeta) is
    -21 to 0 here); the caller's FP64 formulas are for what is outside of them.

    Bounds: logarithms carry 2^-55, products with n, 1/(2n) and lambda r 2^-57 each;
    2^x turns them into relative errors (times ln 2), and one rounding adds 2^-53."""
    mpmath = pytest.importorskip("mpmath")
    mp, mpf = mpmath.mp, mpmath.mpf
    mp.dps = 50
    rec = {"Si": (1830.8, 471.18, 2.4799, 1.7322, 1.1e-6, 0.78734, 1.0039e5, 16.217, -0.59825),
           "C": (1393.6, 346.74, 3.4879, 2.2119, 1.5724e-7, 0.72751, 3.8049e4, 4.3484, -0.57058)}[element]
    rnd = random.Random(24)
    calls = [rec + (rnd.uniform(1.2, 3.0), 10 ** rnd.uniform(-2, 6)) for _ in range(3000)]
    inc = ["-I", os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include"), "-I", cuda_include()]
    (tmp_path / "t.cpp").write_text(PAIR)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, *inc, "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")], check=True)
    text = "".join(" ".join(float(v).hex() for v in c) + "\n" for c in calls)
    out = subprocess.run([str(tmp_path / "t")], input=text, capture_output=True, text=True, check=True).stdout
    u53 = mpf(2) ** -53
    rows = out.splitlines()
    assert len(rows) == len(calls)
    for c, row in zip(calls, rows):
        ok, fr, bfa, dz = (float.fromhex(v) if "x" in v else float(v) for v in row.split())
        A, B, l1, l2, beta, n, _, _, _, r, zeta = (mpf(v) for v in c)
        assert ok, c
        u = (beta * zeta) ** n
        b = (1 + u) ** (-1 / (2 * n))
        want = A * mpmath.exp(-l1 * r), -b * B * mpmath.exp(-l2 * r)
        assert abs(mpf(fr) / want[0] - 1) <= 1.5 * u53
        assert abs(mpf(bfa) / want[1] - 1) <= 2 * u53
        assert abs(mpf(dz) / (-want[1] * u / (4 * (1 + u) * zeta)) - 1) <= 3 * u53


def cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(d, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    return d


BOND = r"""
#include "tersoff_fx.cuh"
#include <cstdio>
int main() {
  long long x, y, z;
  int q;
  while (scanf("%lld %lld %lld %d", &x, &y, &z, &q) == 4) {
    const auto b = tgb::fx::bond64(BOND_CALL);
    printf("%a %lld %lld %lld\n", tgb::fx::pack_in(b.r), (long long)b.ux, (long long)b.uy, (long long)b.uz);
  }
}
"""


def test_bond_lengths_keep_their_bits_for_close_pairs(tmp_path):
    """Lengths from 1e-6 A up and every scale of positions: the square to 2^-57, its
    root to 2^-56 (fxmath) and a rounding to double; unit vectors to 2^-56 of 1."""
    mpmath = pytest.importorskip("mpmath")
    mp, mpf = mpmath.mp, mpmath.mpf
    mp.dps = 50
    rnd = random.Random(25)
    calls = []
    for _ in range(4000):
        q = rnd.choice([30, 44, 52, 57])
        r = 10 ** rnd.uniform(-6 if q > 44 else -2, 0.6)
        d = [rnd.gauss(0, 1) * rnd.choice([1, 1, 1e-3, 0]) for _ in range(3)]
        n = math.sqrt(sum(v * v for v in d)) or 1.0
        v = [int(r * c / n * 2.0 ** q) for c in d]
        if any(v):
            calls.append((*v, q))
    calls += [(1, 0, 0, 52), (0, -1, 0, 52), (1, 1, 1, 52), ((1 << 62) - 1, 0, 0, 60), (1 << 61, -(1 << 61), 1 << 61, 60)]
    inc = ["-I", os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include"), "-I", cuda_include()]
    (tmp_path / "t.cpp").write_text(BOND.replace("BOND_CALL", "x, y, z, q"))
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, *inc, "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")], check=True)
    out = subprocess.run([str(tmp_path / "t")], input="".join("%d %d %d %d\n" % c for c in calls), capture_output=True,
                         text=True, check=True).stdout.splitlines()
    assert len(out) == len(calls)
    for c, row in zip(calls, out):
        r, *u = row.split()
        n = mpmath.sqrt(mpf(c[0]) ** 2 + mpf(c[1]) ** 2 + mpf(c[2]) ** 2)
        assert abs(mpf(float.fromhex(r)) * mpf(2) ** c[3] / n - 1) <= mpf(2) ** -53 + mpf(2) ** -55, c
        for a, b in zip(c[:3], u):
            assert abs(mpf(int(b)) / mpf(2) ** 62 - a / n) <= mpf(2) ** -56, c
