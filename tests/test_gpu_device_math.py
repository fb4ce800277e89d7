"""Device functions that no entry point exposes by themselves, compiled into a small library
and compared with exact references (-m gpu): the root and quotient of Algorithm 3
(csrc/rej_root.cuh) and the assembly of a digit product's sums (csrc/oz_mma.cuh)."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2510_26574_gb300.build import ARCH, CSRC, FLAGS, nvcc

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda_runtime.h>
#include <stdint.h>
#include "rej_root.cuh"
#include "oz_mma.cuh"
__global__ void k_root(const double* h, const double* c, double* s, double* y, double* q, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    kevd::rej_root(h[i], s[i], y[i]);
    q[i] = kevd::rej_quot(c[i], s[i], y[i]);
}
__global__ void k_value(const long long* T, const float* M, const int* sc, double* v, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) v[i] = kevd::oz_value(T[i], M[i], sc[i]);
}
extern "C" int run_root(const double* h, const double* c, double* s, double* y, double* q, int n) {
    k_root<<<(n + 255) / 256, 256>>>(h, c, s, y, q, n);
    return cudaDeviceSynchronize();
}
extern "C" int run_value(const long long* T, const float* M, const int* sc, double* v, int n) {
    k_value<<<(n + 255) / 256, 256>>>(T, M, sc, v, n);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    d = tmp_path_factory.mktemp("math")
    (d / "m.cu").write_text(SRC)
    subprocess.run([nvcc(), *ARCH, *FLAGS, "-I", CSRC, "-shared", "-o", str(d / "m.so"), str(d / "m.cu")], check=True)
    torch.zeros(1, device="cuda")
    return ctypes.CDLL(str(d / "m.so"))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


# h over the range that takes them (above 2^-900) with exponents of both parities and neighbours of powers of
# four, where a root is next to a power of two; |c| as an entry of the column, up to 1 and down to 2^-400.
# Both end in one rounding of a value whose own error is the square of a rounding (2^-104): the
# rounded root or quotient, or its neighbour where the exact one is that close to a tie; the
# reciprocal root is one step from 2^-22 (cubed) with three roundings.
def test_reject_root_and_quotient(L):
    g = torch.Generator().manual_seed(7)
    n = 1 << 20
    e = torch.randint(-899, 2, (n,), generator=g).double()
    h = torch.ldexp(1 + torch.rand(n, generator=g, dtype=torch.float64), e)
    p4 = torch.ldexp(torch.ones(400, dtype=torch.float64), -2 * torch.arange(400).double())
    h[:800] = torch.cat([torch.nextafter(p4, torch.zeros(1).double()), p4])
    h[800:200000] = torch.rand(199200, generator=g, dtype=torch.float64)
    c = torch.ldexp(torch.rand(n, generator=g, dtype=torch.float64) - 0.5, -torch.randint(0, 400, (n,), generator=g).double())
    c[:100000] = h[:100000]
    h, c = h.cuda(), c.cuda()
    s, y, q = (torch.empty_like(h) for _ in range(3))
    assert L.run_root(_p(h), _p(c), _p(s), _p(y), _p(q), n) == 0
    root = torch.sqrt(h)

    def ulps(a, b):
        return (a.view(torch.int64) - b.view(torch.int64)).abs().max().item()
    assert ulps(s, root) <= 1
    assert ((s != root).double().mean().item()) < 1e-3
    assert ulps(q, c / s) <= 1
    assert (((q != c / s).double().mean().item())) < 1e-3
    assert ((y * root - 1).abs().max().item()) <= 4 * 2.0 ** -53


# (T 2^-32 + M) 2^sc with T up to 2^62, M up to 2^-5 (normal, zero and far below T's last bit),
# cancelling sums, T = 0, and scales that leave the normal range: one rounding (two where the
# result is subnormal) of a sum on the grid of 2^-61 of T, at the finest 2^-66, to which M is cut.
def test_digit_sum_value(L):
    rng = np.random.Generator(np.random.PCG64(1))
    n = 20000
    T = (rng.integers(-2**62 + 1, 2**62, n) >> rng.integers(0, 62, n)).astype(np.int64)
    M = ((rng.random(n) - 0.5) * 2.0 ** -rng.integers(4, 60, n)).astype(np.float32)
    T[:500] = 0
    M[500:1000] = 0
    T[1000:2000] = rng.integers(-2**27, 2**27, 1000)            # |T 2^-32| of the size of M: they cancel
    M[1000:2000] = (-T[1000:2000] * 2.0**-32 * (1 + rng.choice([0, 2.0**-20, -2.0**-9], 1000))).astype(np.float32)
    sc = rng.integers(-60, 30, n).astype(np.int32)
    sc[2000:3000] = rng.choice([-1100, -1050, -1030, -1000, 990, 1000], 1000)
    T[2000:3000] >>= 20
    t = [torch.from_numpy(a).cuda() for a in (T, M, sc)]
    v = torch.empty(n, dtype=torch.float64, device="cuda")
    assert L.run_value(*map(_p, t), _p(v), n) == 0
    v = v.cpu().numpy()
    for i in range(n):
        big = max(abs(Fraction(int(T[i]), 2**32)), abs(Fraction(float(M[i]))))
        exact = (Fraction(int(T[i]), 2**32) + Fraction(float(M[i]))) * Fraction(2) ** int(sc[i])
        half = Fraction(51 if abs(v[i]) >= 2.0 ** -1022 else 101, 100) * Fraction(float(np.spacing(abs(v[i]))))
        grid = max(big * Fraction(1, 2**61), Fraction(1, 2**66)) * Fraction(2) ** int(sc[i])
        assert abs(Fraction(float(v[i])) - exact) <= half + grid, (i, T[i], M[i], sc[i], v[i])
