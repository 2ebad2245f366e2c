"""exp, log2, log and reciprocal of csrc/fxmath.cuh, compiled for the host, against exact decimal
arithmetic.

Bounds, in units of the result's last place: rounding costs 1/2; the fixed-point evaluation adds
2^-58 relative for exp2, exp and 1/x (below 0.04), and for the logarithms 2^-53 of the Q52 result
(1/2 at results just above 1), once more through ln 2 where the mantissa is renormalised.
"""
import os
import struct
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

from tests.conftest import ROOT

HOST = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#define FX_HOST
#define FX_FN static inline
#define FX_SLOW static
#define FX_TAB static const
typedef unsigned long long fx_u64;
typedef long long fx_i64;
FX_FN fx_u64 fx_mulhi(fx_u64 a, fx_u64 b) { return (fx_u64)(((unsigned __int128)a * b) >> 64); }
FX_FN fx_i64 fx_mulhi_s(fx_i64 a, fx_i64 b) { return (fx_i64)(((__int128)a * b) >> 64); }
FX_FN unsigned fx_mulhi32(unsigned a, unsigned b) { return (unsigned)(((fx_u64)a * b) >> 32); }
FX_FN int fx_mulhi32_s(int a, int b) { return (int)(((fx_i64)a * b) >> 32); }
FX_FN int fx_clz(fx_u64 a) { return a ? __builtin_clzll(a) : 64; }
FX_FN double fx_as_double(fx_u64 a) { double d; memcpy(&d, &a, 8); return d; }
FX_FN fx_u64 fx_bits(double a) { fx_u64 d; memcpy(&d, &a, 8); return d; }
FX_FN float fx_rcp_seed(float f) { return 1.0f / f * (1.0f + 1.2e-7f); }  // off by the seed's allowance
FX_FN unsigned fx_bits_f(float a) { unsigned d; memcpy(&d, &a, 4); return d; }
FX_FN float fx_as_float(unsigned a) { float d; memcpy(&d, &a, 4); return d; }
#include "fxmath.cuh"
int main() {
  char f; double x;
  while (scanf(" %c %la", &f, &x) == 2) {
    double y = f == 'e' ? fx_exp(x) : f == 'l' ? fx_log(x) : f == 'r' ? fx_rcp(x) : f == '2' ? fx_log2_d(x)
               : f == 'q' ? (double)fx_log2(x) : fx_exp2(fx_from_double(x, 52));
    printf("%a\n", y);
  }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(HOST)
    exe = str(d / "fx")
    subprocess.check_call(["g++", "-O1", "-std=gnu++17", "-w", "-I",
                           os.path.join(ROOT, "paper_2205_05681_gb300", "csrc"), str(d / "fx.cpp"), "-o", exe])

    def run(f, xs):
        out = subprocess.run([exe], input="".join("%s %s\n" % (f, float(x).hex()) for x in xs),
                             capture_output=True, text=True, check=True).stdout
        return [float.fromhex(v) for v in out.split()]

    return run


def _inputs(f):
    rng = np.random.default_rng(5)
    if f == "e":
        x = np.concatenate([rng.uniform(-700, 700, 300), rng.uniform(-1, 1, 300), [0.0, 1.0, -1.0, 511.0, -600.0]])
    elif f == "p":
        x = np.concatenate([rng.uniform(-1020, 1020, 300), np.arange(-64, 65) / 64.0])
        x = np.round(x * 2.0 ** 40) / 2.0 ** 40  # exact in Q52
    else:
        edge = np.array([1 + i / 64.0 for i in range(64)])  # the tables' interval edges
        x = np.concatenate([np.exp(rng.uniform(-600, 600, 300)), rng.uniform(0.3, 3.0, 300), edge,
                            np.nextafter(edge, 0.0), np.nextafter(edge, 9.0)])
    return x


@pytest.mark.parametrize("f,bound", [("e", 0.54), ("p", 0.54), ("r", 0.54), ("l", 1.25), ("2", 1.05)])
def test_against_decimal(fx, f, bound):
    getcontext().prec = 50
    ln2 = Decimal(2).ln()
    xs = _inputs(f)
    if f in "l2":
        xs = xs[np.abs(np.log(xs)) > 0.1]  # the callers' logarithms: relative to the result there
    for x, y in zip(xs, fx(f, xs)):
        d = Decimal(float(x))
        ref = {"e": lambda: d.exp(), "p": lambda: (d * ln2).exp(), "r": lambda: 1 / d, "l": lambda: d.ln(),
               "2": lambda: d.ln() / ln2}[f]()
        ulp = Decimal(float(np.spacing(abs(float(ref)))))
        assert abs(Decimal(y) - ref) <= Decimal(bound) * ulp, (f, x, y)


def test_edges(fx):
    assert fx("e", [800.0, -800.0, -745.0]) == [float("inf"), 0.0, 5e-324]
    assert fx("p", [1023.5, 1024.5, -1074.0, -1500.0])[1:] == [float("inf"), 5e-324, 0.0]
    assert fx("r", [1.0, -2.0, 2.0 ** 1023, 4e-320]) == [1.0, -0.5, 2.0 ** -1023, float("inf")]
    # a logarithm of 1 is off by the fixed-point unit at most
    assert abs(fx("2", [1.0])[0]) <= 2.0 ** -59
    assert abs(struct.unpack("d", struct.pack("d", fx("q", [2.0 ** 100])[0]))[0] - 100 * 2.0 ** 52) <= 1
