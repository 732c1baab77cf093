"""The fixed-point arithmetic of the float64 sweeps (gp_fix.cuh) on the host, against exact integers.

gp_fix.cuh is compiled into a small program by the host compiler; Python's integers are the reference.
Tolerances: a table component is stored in units of 2^-62 (2^-60 allows four of them); a
product by a table factor rounds four half products to one unit each: 4 units a component.
"""
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "gp_fix.cuh"
// lines "c s x y" (doubles by their bits, integers): the stored factors and (x + i y)(c + i s)
int main() {
  unsigned long long bc, bs;
  long long x, y;
  while (std::scanf("%llu %llu %lld %lld", &bc, &bs, &x, &y) == 4) {
    double c, s;
    std::memcpy(&c, &bc, 8);
    std::memcpy(&s, &bs, 8);
    const gp::ufix2 w{gp::fix_factor(c), gp::fix_factor(s)};
    const gp::cfix z = gp::ftwmul(gp::cfix{x, y}, w);
    std::printf("%llu %llu %lld %lld\n", w.c, w.s, z.x, z.y);
  }
}
"""


@pytest.fixture(scope="module")
def host_program(tmp_path_factory):
    """A function that compiles a C++ source that includes gp_fix.cuh and returns the program's path."""
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")

    def build(source):
        d = tmp_path_factory.mktemp("fix")
        (d / "fix.cpp").write_text(source)
        subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2003_03590_gb300", "csrc"), "-I", cuda,
                        str(d / "fix.cpp"), "-o", str(d / "fix")], check=True)
        return str(d / "fix")
    return build


@pytest.fixture(scope="module")
def multiply(host_program):
    prog = host_program(SOURCE)

    def run(c, s, x, y):
        bits = [struct.unpack("<Q", struct.pack("<d", v))[0] for v in np.concatenate([c, s])]
        m = len(c)
        text = "".join(f"{bits[i]} {bits[m + i]} {x[i]} {y[i]}\n" for i in range(m))
        out = subprocess.run([prog], input=text, capture_output=True, text=True, check=True).stdout.split()
        return [tuple(int(v) for v in out[4 * i:4 * i + 4]) for i in range(m)]
    return run


def pair_table(n, alpha, s):
    """E[k1] E[k2] of the kinetic factors, formed in float64 as the library's tables are."""
    k = np.where(np.arange(n) < (n + 1) // 2, np.arange(n), np.arange(n) - n).astype(float)
    ph = np.fmod(alpha * k * k * s, 2 * np.pi)
    re, im = np.cos(ph), -np.sin(ph)
    return (np.multiply.outer(re, re) - np.multiply.outer(im, im)).ravel(), \
        (np.multiply.outer(re, im) + np.multiply.outer(im, re)).ravel()


def check(multiply, c, s):
    r = np.random.default_rng(1)
    x, y = (r.integers(-2 ** 61, 2 ** 61, len(c)).tolist() for _ in range(2))
    for i, (uc, us, zx, zy) in enumerate(multiply(c, s, x, y)):
        ec, es = (min(max(float(v), -1.0), 1.0) for v in (c[i], s[i]))
        assert abs(Fraction(uc, 2 ** 63) - 1 - Fraction(ec)) <= Fraction(1, 2 ** 60), (c[i], uc)
        assert abs(Fraction(us, 2 ** 63) - 1 - Fraction(es)) <= Fraction(1, 2 ** 60), (s[i], us)
        fc, fs = Fraction(uc, 2 ** 63) - 1, Fraction(us, 2 ** 63) - 1
        assert abs(zx - (x[i] * fc - y[i] * fs)) <= 4 and abs(zy - (y[i] * fc + x[i] * fs)) <= 4


@pytest.mark.parametrize("n,alpha,s", [(16, 0.05, np.pi), (256, 0.05206503443154336, 0.0068034478138743991),
                                       (64, 0.05, 2.4166097335306098), (32, 0.5, 2 * np.pi / 40), (32, 0.5, np.pi / 40),
                                       (64, 0.5, 2 * np.pi / 10), (64, 0.5, np.pi / 10), (128, 0.5, 2 * np.pi / 20)])
def test_kinetic_factors_near_a_quarter_turn(multiply, n, alpha, s):
    """Time steps at which factors are 1, i, -1, -i up to rounding: every entry keeps its value."""
    c, r = pair_table(n, alpha, s)
    near = np.maximum(np.abs(c), np.abs(r)) >= 1.0 - 2.0 ** -50
    assert near.any()
    sel = np.flatnonzero(near)[:2000]
    check(multiply, c[sel], r[sel])


def test_components_at_and_beyond_one(multiply):
    ulp = 2.0 ** -53
    v = np.array([1.0, 1 + 2 * ulp, 1 + 4 * ulp, 1 - ulp, 1 - 2 * ulp, 0.0, 2.0 ** -30, 0.7071067811865476])
    c = np.concatenate([v, -v, np.zeros(16)])
    s = np.concatenate([np.zeros(16), v, -v])
    check(multiply, c, s)


def test_flow_coefficients_that_are_not_finite(host_program):
    """nl_fix ends for every double (the sweeps then write NaN)."""
    run = host_program(r"""
#include <cstdio>
#include <limits>
#include "gp_fix.cuh"
int main() {
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  for (double v : {inf, -inf, nan, 0.0, 5e-324, 1.7e308, -1.7e308})
    std::printf("%d ", gp::nl_fix(v, 1.0).m >> 63 == 1 ? 1 : 0);
}
""")
    out = subprocess.run([run], capture_output=True, text=True, check=True, timeout=20).stdout
    assert out.split() == ["0", "0", "0", "0", "1", "1", "1"]


CONVERT = r"""
#include <cstdio>
#include "gp_fix.cuh"
// "t bits s": to_fix; "f v s": from_fix
int main() {
  char k;
  unsigned long long u;
  int s;
  while (std::scanf(" %c %llu %d", &k, &u, &s) == 3)
    std::printf("%lld\n", k == 't' ? gp::to_fix(u, s) : (long long)gp::from_fix((long long)u, s));
}
"""


def test_conversions_round_to_nearest_even(host_program):
    """float64 to fixed point and back: the nearest number, ties to even, over the float64 range."""
    prog = host_program(CONVERT)
    r = np.random.default_rng(2)
    lines, want = [], []
    for _ in range(3000):
        d = float(r.standard_normal() * 2.0 ** r.integers(-1000, 960))
        e = int(np.frexp(d)[1])
        s = int(61 - e - r.integers(0, 70))                  # |d| 2^s < 2^62, down to less than a unit
        lines.append(f"t {struct.unpack('<Q', struct.pack('<d', d))[0]} {s}")
        want.append(round(Fraction(d) * Fraction(2) ** s))
        v = int(r.integers(-2 ** 62, 2 ** 62)) >> int(r.integers(0, 62))
        s = int(r.integers(-900, 900))
        lines.append(f"f {v % 2 ** 64} {s}")
        want.append(struct.unpack("<q", struct.pack("<d", float(Fraction(v) * Fraction(2) ** -s)))[0])
    # ties: 53 bits and a half
    for k in range(64):
        v = ((2 ** 52 + k) << 11) + 2 ** 10
        lines.append(f"f {v - 2 ** 62 if v >= 2 ** 63 else v} 0")
        want.append(struct.unpack("<q", struct.pack("<d", float(v - 2 ** 62 if v >= 2 ** 63 else v)))[0])
    out = subprocess.run([prog], input="\n".join(lines), capture_output=True, text=True, check=True).stdout.split()
    assert [int(x) for x in out] == want


FLOW = r"""
#include <cmath>
#include <cstdio>
#include "gp_fix.cuh"
static unsigned long long factor(long double v) {   // (v + 1) 2^63, even
  const long double u = (v + 1.0L) * 4611686018427387904.0L;
  return u >= 9223372036854775807.0L ? ~1ull : (unsigned long long)std::nearbyintl(u) << 1;
}
// "coef shift x y s": exp(-i coef (|psi|^2 - shift)) psi for psi = (x + i y) 2^-s, in units of 2^-s
int main() {
  gp::ufix2 dir[256];
  const long double pi = 3.14159265358979323846264338327950288L;
  for (int k = 0; k < 256; ++k) dir[k] = gp::ufix2{factor(cosl(2 * pi * k / 256)), factor(sinl(2 * pi * k / 256))};
  double coef, shift;
  long long x, y;
  int s;
  while (std::scanf("%lf %lf %lld %lld %d", &coef, &shift, &x, &y, &s) == 5) {
    const gp::NlFix f = gp::nl_fix(coef, shift);
    const gp::cfix z = gp::fnonlinear(gp::cfix{x, y}, 2 * s + f.q - 126, f.m, f.tc, f.neg, dir);
    std::printf("%lld %lld\n", z.x, z.y);
  }
}
"""


def test_nonlinear_flow_against_extended_precision(host_program):
    """N(s) at one point, |psi|^2 from 1e-12 to 100 and |coef| |psi|^2 up to 20.

    At the kernels' scale the larger component has 62 bits, |psi|^2 then 61 and two truncations: the phase is good to
    2^-59 |coef| |psi|^2 (float64: 2^-53); the directions, the products and the series add a few 2^-61, 1e-17 in all.
    Needs a long double of 64 bits or more.
    """
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("long double is double here")
    prog = host_program(FLOW)
    r = np.random.default_rng(3)
    ext = np.longdouble
    cases = []
    for _ in range(2000):
        amp = 10.0 ** r.uniform(-6, 1)
        ph = r.uniform(0, 2 * np.pi)
        re, im = amp * np.cos(ph), amp * np.sin(ph)
        s = int(62 - np.frexp(max(abs(re), abs(im)))[1])
        x, y = int(re * 2.0 ** s), int(im * 2.0 ** s)
        coef = float(r.uniform(-20, 20) / max(amp * amp, 1.0))
        cases.append((coef, float(r.integers(0, 2)), x, y, s))
    text = "".join(f"{c!r} {h!r} {x} {y} {s}\n" for c, h, x, y, s in cases)
    out = subprocess.run([prog], input=text, capture_output=True, text=True, check=True).stdout.split()
    for i, (c, h, x, y, s) in enumerate(cases):
        u = ext(2) ** ext(-s)
        X, Y = ext(x) * u, ext(y) * u
        ph = ext(c) * (X * X + Y * Y - ext(h))
        cs, sn = np.cos(ph), np.sin(ph)
        err = np.hypot(ext(int(out[2 * i])) * u - (X * cs + Y * sn), ext(int(out[2 * i + 1])) * u - (Y * cs - X * sn))
        bound = (ext(2) ** -59 * abs(c) * (X * X + Y * Y) + 1e-17) * np.hypot(X, Y)
        assert err <= bound, (cases[i], float(err / np.hypot(X, Y)))
