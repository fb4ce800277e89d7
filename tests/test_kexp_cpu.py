"""The exponential of the FP64 engine's kernel values (csrc/kexp.cuh), whose arithmetic is
integer throughout, compiled for the host and compared with long double exp: no GPU needed."""
import os
import subprocess

import numpy as np
import pytest

from paper_2510_26574_gb300.build import CSRC, nvcc

SRC = r"""
#include <cstdio>
#include <cstring>
#include <vector>
static unsigned long long __umul64hi(unsigned long long a, unsigned long long b) { return (unsigned __int128)a * b >> 64; }
static long long __mul64hi(long long a, long long b) { return (__int128)a * b >> 64; }
static long long __double_as_longlong(double d) { long long x; memcpy(&x, &d, 8); return x; }
#include "kexp.cuh"
int main() {
    unsigned long long tbl[1024];
    for (int j = 0; j < 1024; ++j) tbl[j] = (unsigned long long)llroundl(ldexpl(exp2l(j / 1024.0L), 62));
    double v[2];
    while (fread(v, 8, 2, stdin) == 2) {
        const unsigned long long b = kevd::kexp_bits(v[0], kevd::kexp_scale(v[1]), tbl);
        fwrite(&b, 8, 1, stdout);
    }
}
"""


@pytest.fixture(scope="module")
def kexp(tmp_path_factory):
    d = tmp_path_factory.mktemp("kexp")
    (d / "kexp.cpp").write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-w", "-I", CSRC, "-I", inc, str(d / "kexp.cpp"), "-o", str(d / "kexp")],
                   check=True)

    def run(d2, s):
        pairs = np.stack(np.broadcast_arrays(np.asarray(d2, np.float64), np.asarray(s, np.float64)), -1)
        out = subprocess.run([str(d / "kexp")], input=np.ascontiguousarray(pairs).tobytes(), stdout=subprocess.PIPE,
                             check=True)
        return np.frombuffer(out.stdout, np.float64)
    return run


# Scales 1 / eps: 1, ordinary, and so far out that t's exponents meet in other places (the last
# two are subnormal or next to it).  Below t = 128 the bound is 1 ulp (0.76 of the method, and the
# long double product), above 2 ulp (1.5 of the method).
@pytest.mark.parametrize("s", [1.0, 1 / 0.37, 3.0e5, 1 / 3e150, 1e200, 2.5e-308, 3e-310])
def test_engine_exponential_relative(kexp, s):
    rng = np.random.Generator(np.random.PCG64(3))
    step = np.log(2.0) / 1024
    t = np.concatenate([707.9 * rng.random(20000), rng.random(20000), 10.0 ** (-20 * rng.random(2000)),
                        step * np.arange(4000), step * (np.arange(4000) + 0.5) * (1 + 1e-15),      # table points, halves
                        2.0 ** np.arange(-60, 9), np.nextafter(2.0 ** np.arange(-60, 10), 0), [707.0, 43.7, 44.0]])
    with np.errstate(over="ignore"):
        d2 = t / s
    d2 = d2[np.isfinite(d2)]
    p = np.longdouble(d2) * np.longdouble(s)
    keep = p < 707.99
    d2, p = d2[keep], p[keep]
    ref = np.exp(-p)
    ulp = np.ldexp(np.longdouble(1), np.frexp(ref)[1] - 53)
    err = np.abs(np.longdouble(kexp(d2, s)) - ref) / ulp
    assert err[p < 128].max() < 1.0 and err.max() < 2.0, (float(err[p < 128].max()), float(err.max()))


def test_engine_exponential_ends(kexp):
    inf = np.inf
    d2 = [0.0, -0.0, -1e-9, -inf, 5e-324, 707.9, 708.0, 709.0, 1e300, inf, np.nan]
    out = kexp(d2, 1.0)
    assert out[:5].tolist() == [1.0] * 5 and out[5] > 0 and out[6:].tolist() == [0.0] * 5
    assert kexp([1.0, 1e-300], inf).tolist() == [0.0, 0.0]
    assert kexp([0.0], 1e308)[0] == 1.0 and abs(kexp([5e-324], 1e308)[0] - (1.0 - 5e-324 * 1e308)) <= 2.0 ** -53
