"""The fixed-point transform (csrc/fixfft.cuh, compiled for the host) against long
double, beside the FP64 transform it takes the place of: every length class
(radix 8 or 4 first, with and without the radix-3 pass) on flat and decaying
inputs, and the Chebyshev derivative of grid values, which multiplies the
errors of the coefficients by up to K^2 and adds up any that share a sign.  Bar:
the error of numpy's FP64 transform of the same values."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_07092_gb300", "csrc")

SOURCE = r"""
#include <climits>
#include <cmath>
#include <cstdlib>
#include <vector>
#include "fixfft.cuh"
using namespace pz;
// forward transform of L = (three ? 3 : 1) << lg points x (re, im), |x| < 1, in units
// of 2^-FX_BITS; the result as integers, scaled by 2^-S (returned).  RND: as the radial
// kernels run it
template <bool RND>
static int run(int lg, int three, const double* x, long long* out) {
    const int L = (three ? 3 : 1) << lg;
    std::vector<fxw> tw(L);
    std::vector<fxc> a(L), b(L);
    auto split = [](long double c, int& hi, int& lo) {
        const long long v = llroundl(c * 4611686018427387904.0L);
        lo = (int)(unsigned)(unsigned long long)v;
        hi = (int)((v - lo) >> 32);
        if (lo == INT_MIN) ++lo;
    };
    unsigned l1 = 0;
    for (int j = 0; j < L; ++j) {
        const long double w = 2.0L * 3.141592653589793238462643383279502884L * j / L;
        split(cosl(w), tw[j].x1, tw[j].x0);
        split(-sinl(w), tw[j].y1, tw[j].y0);
        fx64* q[2] = {&a[j].x, &a[j].y};
        for (int p = 0; p < 2; ++p) {
            int h, l;
            *q[p] = llrint(ldexp(x[2 * j + p], FX_BITS));
            fx_words(*q[p], h, l);
            l1 += (unsigned)abs(h) / (1u << 11) + 1u;
        }
    }
    int S, p = 1;
    const unsigned back = fx_schedule(lg, three, 43 + 32 - __builtin_clz(l1), S);
    for (int n = (lg & 1) ? L >> 3 : L >> 2, t = 0; t < n; ++t)
        (lg & 1) ? fx_first8<RND>(a.data(), b.data(), n, t) : fx_first4(a.data(), b.data(), n, t);
    a.swap(b);
    for (int q = (lg & 1) ? 3 : 2; q < lg; q += 2, ++p, a.swap(b))
        for (int t = 0; t < L >> 2; ++t)
            fx_pass4<RND>(a.data(), b.data(), L >> 2, q, tw.data(), L >> (q + 2), (back >> p) & 1, p == 1, t);
    if (three) {
        for (int t = 0; t < 1 << lg; ++t)
            fx_pass3(a.data(), b.data(), 1 << lg, tw.data(), 1, (back >> p) & 1, p == 1, t);
        a.swap(b);
    }
    for (int j = 0; j < L; ++j) out[2 * j] = a[j].x, out[2 * j + 1] = a[j].y;
    return S;
}
extern "C" int transform(int rnd, int lg, int three, const double* x, long long* out) {
    return rnd ? run<true>(lg, three, x, out) : run<false>(lg, three, x, out);
}
"""


@pytest.fixture(scope="module")
def fixed(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, lib = d / "fx.cpp", d / "fx.so"
    src.write_text(SOURCE)
    nvcc = os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")
    cuda = os.path.dirname(os.path.dirname(nvcc))
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-I" + os.path.join(cuda, "include"),
                    str(src), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).transform

    def transform(x, even=False):
        """of a complex vector, normalised by the power of two above its largest part, as
        the azimuthal kernels run it; of an even one, whose parts stay apart, each part
        by its own, as the radial kernels do"""
        L = len(x)
        three = L % 3 == 0
        lg = (L // 3 if three else L).bit_length() - 1
        parts = np.stack([x.real, x.imag], 1)
        e = np.frexp(np.abs(parts).max(0))[1]
        if not even:
            e[:] = e.max()
        v = np.ascontiguousarray(np.ldexp(parts, -e))
        out = np.zeros((L, 2), np.int64)
        S = fn(int(even), lg, int(three), v.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p))
        y = np.ldexp(out.astype(np.longdouble), S - 60 + e)
        return y[:, 0] + 1j * y[:, 1]
    return transform


def exact(x):
    return np.fft.fft(x.astype(np.clongdouble))


def norm(x):
    return float(np.sqrt((np.abs(x) ** 2).sum()))


@pytest.mark.parametrize("L", [16, 32, 64, 128, 256, 512, 1024, 2048, 4096, 8192, 12, 24, 48, 96, 192, 384, 768, 1536,
                               3072, 6144])
@pytest.mark.parametrize("decay", [0, 2])
def test_transform(fixed, L, decay):
    rng = np.random.default_rng(L)
    x = (rng.uniform(-1, 1, L) + 1j * rng.uniform(-1, 1, L)) / (1.0 + np.arange(L)) ** decay
    ref = exact(x)
    assert norm(fixed(x) - ref) <= norm(np.fft.fft(x) - ref)


@pytest.mark.parametrize("K", [16, 64, 256, 512, 1024, 2048])
def test_derivative_of_grid_values(fixed, K):
    rng = np.random.default_rng(K)
    ld = np.longdouble
    n = min(K - 1, 40)
    c = np.zeros((2, K + 1), ld)
    c[:, :n] = rng.uniform(-1, 1, (2, n)) / (1 + np.arange(n)) ** 2

    def grid(c):  # sum_n c_n cos(pi n k / K), each row
        v = c.copy()
        v[:, [0, K]] *= 2
        return np.stack([exact(np.concatenate([r, r[-2:0:-1]]))[:K + 1].real / 2 for r in v])

    def derivative(C):  # on the grid, from the transform C of the even extension
        c = C / K
        c[:, [0, K]] /= 2
        t = 2 * np.arange(K + 1).astype(ld) * c
        s, d = np.zeros_like(c), np.zeros_like(c)
        for q in (0, 1):
            s[:, q::2] = np.cumsum(t[:, q::2][:, ::-1], 1)[:, ::-1]
        d[:, :-1] = s[:, 1:]
        d[:, 0] /= 2
        return grid(d)

    f = grid(c).astype(float)
    z = np.concatenate([f, f[:, -2:0:-1]], 1)
    z = z[0] + 1j * z[1]
    parts = lambda y: np.stack([y.real, y.imag])[:, :K + 1].astype(ld)  # noqa: E731
    ref = derivative(parts(exact(z)))
    err = [norm(derivative(parts(y)) - ref) for y in (fixed(z, even=True), np.fft.fft(z))]
    assert err[0] <= err[1], [e / norm(ref) for e in err]
