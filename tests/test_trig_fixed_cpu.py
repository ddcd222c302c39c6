"""The FP64 sine and cosine of csrc/trig_fixed.cuh compiled for the host, against
mpmath at 140 bits.

Bar: 1.52 ulp of the result. The reduced angle r carries one rounding (half an ulp
of r; the third term of pi/2 moves the result by far less), the polynomials and the
final operation 0.51 ulp; where the result lies in the binade below r's, half an ulp
of r is a whole one of the result.
"""
import ctypes
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1609_04493_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
#define __noinline__
using std::fma;
static unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((uint64_t)a * b) >> 32); }
static long long bits(double x) { long long l; memcpy(&l, &x, 8); return l; }
static int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static int __double2loint(double x) { return (int)bits(x); }
static double __longlong_as_double(long long l) { double x; memcpy(&x, &l, 8); return x; }
static double __hiloint2double(int h, int l)
{
    return __longlong_as_double((long long)(((uint64_t)(unsigned)h << 32) | (unsigned)l));
}
static int __clzll(long long x) { return __builtin_clzll((unsigned long long)x); }
static void sincos(double x, double *s, double *c) { *s = std::sin(x); *c = std::cos(x); }
"""


@pytest.fixture(scope="module")
def sincos(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    fixed = open(os.path.join(CSRC, "trig_fixed.cuh")).read()
    consts = re.findall(r"^constexpr double kDf\w+ = .*$", open(os.path.join(CSRC, "df_trig.cuh")).read(), re.M)
    assert len(consts) == 3
    body = "\n".join(l for l in fixed.splitlines() if not re.match(r"#(include|pragma)", l))
    d = tmp_path_factory.mktemp("trig")
    src, so = str(d / "t.cpp"), str(d / "t.so")
    with open(src, "w") as fh:
        fh.write(SHIM.replace("static void sincos", "static void library_sincos") +
                 "#define sincos library_sincos\nnamespace rdyn {\n" + "\n".join(consts) + "\n}\n" + body +
                 '\nextern "C" void run(const double *x, double *s, double *c, int n)\n'
                 "{ for (int i = 0; i < n; ++i) rdyn::sincos_fixed(x[i], s + i, c + i); }\n")
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    p = ctypes.POINTER(ctypes.c_double)

    def run(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        s, c = np.empty_like(x), np.empty_like(x)
        lib.run(*(a.ctypes.data_as(p) for a in (x, s, c)), ctypes.c_int(x.size))
        return s, c

    return run


def ulps(x, got, f, mp):
    e = np.empty(len(x))
    for i in range(len(x)):
        want = f(mp.mpf(float(x[i])))
        if want == 0:
            e[i] = 0.0 if got[i] == 0 else np.inf
        else:
            ulp = mp.mpf(2) ** (mp.frexp(abs(want))[1] - 53)
            e[i] = float(abs(mp.mpf(float(got[i])) - want) / ulp)
    return e


def angles():
    rng = np.random.default_rng(11)
    half = rng.integers(-1000, 1000, 3000) * (np.pi / 2)
    return {
        "one turn": rng.uniform(-np.pi, np.pi, 20000),
        "to 2^30": rng.uniform(-1, 1, 20000) * 2.0 ** rng.uniform(0, 30, 20000),
        "beside multiples of pi/2": np.concatenate([half, half + rng.standard_normal(3000) * 2.0 ** -rng.integers(1, 60, 3000)]),
        "small": np.concatenate([2.0 ** -np.arange(0.0, 1074.0, 3), -1.7 * 2.0 ** -np.arange(0.0, 1000.0, 7)]),
    }


@pytest.mark.parametrize("which", list(angles()))
def test_within_the_stated_error(sincos, which):
    mp = pytest.importorskip("mpmath").mp.clone()
    mp.prec = 140
    x = angles()[which]
    s, c = sincos(x)
    es, ec = ulps(x, s, mp.sin, mp), ulps(x, c, mp.cos, mp)
    print(f"{which}: sine {es.max():.2f}, cosine {ec.max():.2f}, mean {es.mean():.2f}, {ec.mean():.2f}")
    assert es.max() <= 1.52 and ec.max() <= 1.52


def test_zero(sincos):
    s, c = sincos([0.0, -0.0])
    assert np.all(s == 0.0) and np.all(c == 1.0)
