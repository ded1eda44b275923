"""The degrees of the near field's power series (csrc/g3_series.cuh), compiled for the host.

Seven points of pairs of neighbouring panels at |z| just below each degree's limit, the
series evaluated with more digits than the precision it serves: the degrees of float32
in float64, those of float64 in extended precision.  What is left of the difference to
the points summed one by one is the series' end, at most |z|^(N+1) / (N+1)! of p(0)
for the single layer and the double layer.

The float32 exponential beside it, against float64: its reduction carries the products'
roundings, so that its error does not grow with the phase.
"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from inputs import meshes

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <algorithm>
#include <cmath>
#define __host__
#define __device__
#define __forceinline__ inline
using std::min; using std::max; using std::fma;
#define __expf(x) std::exp(x)
namespace g3 { template <class T> struct Cx { T x, y; }; enum { G3_SLP = 0, G3_DLP = 1 }; }
#include "g3_series.cuh"
using namespace g3;
template <int KER, class D, int N, class T> static double run(int n, const double* r, const double* a, T x, T y) {
    double worst = 0;
    for (int e = 0; e < n; ++e) {
        constexpr int M = N + SERIES_MORE<KER>;
        T rr[7], aa[7], c[M + 1], rc, R;
        for (int q = 0; q < 7; ++q) { rr[q] = r[7 * e + q]; aa[q] = a[7 * e + q]; }
        series_setup<KER, M, T>(rr, aa, c, rc, R);
        const T zx = -x * R, zy = -y * R;
        const Cx<T> w = series_sum<M>(c, zx, zy, zx * zx + zy * zy);
        T px = 0, py = 0;   // sum_q a_q (1 + s r_q) exp(-s (r_q - r_c))
        for (int q = 0; q < 7; ++q) {
            const T m = aa[q] * std::exp(-x * (rr[q] - rc)), t = y * (rr[q] - rc);
            T fx = 1, fy = 0;
            if (KER) { fx += x * rr[q]; fy = y * rr[q]; }
            px += m * (fx * std::cos(t) + fy * std::sin(t));
            py += m * (fy * std::cos(t) - fx * std::sin(t));
        }
        worst = std::max(worst, (double)(std::hypot(w.x - px, w.y - py) / std::hypot(px, py)));
    }
    return worst;
}
template <int KER, class D, class T> static double levels(int l, int n, const double* r, const double* a, T x, T y) {
    using S = NearSeries<D>;
    return l == 0 ? run<KER, D, S::N0, T>(n, r, a, x, y) : l == 1 ? run<KER, D, S::N1, T>(n, r, a, x, y) : run<KER, D, S::N2, T>(n, r, a, x, y);
}
extern "C" double cexp_worst(int n, const float* sre, const float* sim, const float* r) {
    double worst = 0;
    for (int e = 0; e < n; ++e) {
        const Cx<float> v = cexp_acc(sre[e], sim[e], r[e]);
        const double m = std::exp(-(double)sre[e] * r[e]), t = (double)sim[e] * r[e];
        worst = std::max(worst, std::max(std::abs(v.x - m * std::cos(t)), std::abs(v.y + m * std::sin(t))) / m);
    }
    return worst;
}
extern "C" double worst(int ker, int f64, int l, int n, const double* r, const double* a, double x, double y) {
    if (f64) return ker ? levels<G3_DLP, double, long double>(l, n, r, a, x, y) : levels<G3_SLP, double, long double>(l, n, r, a, x, y);
    return ker ? levels<G3_DLP, float, double>(l, n, r, a, x, y) : levels<G3_SLP, float, double>(l, n, r, a, x, y);
}
"""
Z = {0: (0.5, 1.25, 2.25), 1: (0.5, 1.25, 2.0)}
N = {0: (8, 12, 16), 1: (14, 20, 24)}


@pytest.fixture(scope="module")
def series(tmp_path_factory):
    d = tmp_path_factory.mktemp("series")
    (d / "s.cpp").write_text(SRC)
    so = str(d / "s.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-Wno-unknown-pragmas", "-I",
                    os.path.join(ROOT, "paper_2312_11219_gb300", "csrc"), "-o", so, str(d / "s.cpp")], check=True)
    lib = ctypes.CDLL(so)
    lib.worst.restype = lib.cexp_worst.restype = ctypes.c_double
    return lib


@pytest.fixture(scope="module")
def pairs():
    """Distances and double-layer / single-layer amplitudes of near pairs on a sphere."""
    v, t = meshes.icosphere(2)
    P = v[t]
    c = P.sum(1) / 3
    q = math.sqrt(15.0)
    a1, b1, a2, b2 = (6 - q) / 21, (9 + 2 * q) / 21, (6 + q) / 21, (9 - 2 * q) / 21
    L = np.array([[1 / 3] * 3, [a1, a1, b1], [a1, b1, a1], [b1, a1, a1], [a2, a2, b2], [a2, b2, a2], [b2, a2, a2]])
    w = np.array([9 / 40] + [(155 - q) / 1200] * 3 + [(155 + q) / 1200] * 3)
    y = np.einsum("qa,eak->eqk", L, P)
    n = np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
    r = np.linalg.norm(c[:, None, None] - y[None], axis=3)
    near = (np.linalg.norm(c[:, None] - c[None], axis=2) < 0.9) & ~np.eye(len(t), dtype=bool)
    r = np.ascontiguousarray(r[near])
    pd = ((c[:, None] - P[None, :, 0]) * n[None]).sum(2)[near]
    R = 0.5 * (r.max(1) - r.min(1))
    keep = R > 0.95 * R.max()
    r, pd, R = r[keep], pd[keep], R[keep]
    amp = {0: w / r, 1: w * pd[:, None] / r ** 3}
    return r, {k: np.ascontiguousarray(x) for k, x in amp.items()}, R.max()


@pytest.mark.parametrize("level", [0, 1, 2])
@pytest.mark.parametrize("f64", [0, 1])
@pytest.mark.parametrize("ker", [0, 1])
def test_series_end(series, pairs, ker, f64, level):
    r, amp, Rmax = pairs
    P = ctypes.POINTER(ctypes.c_double)
    z, n = Z[f64][level], N[f64][level]
    bound = z ** (n + 1) / math.factorial(n + 1)
    # |p| >= exp(-|z|) |p(0)| for amplitudes of one sign and real s, and for these pairs
    eps = 2.0 ** (-63 if f64 else -52)
    for phase in (0.0, 0.7, 1.5):
        s = 0.9999 * z / Rmax * np.exp(1j * phase)
        w = series.worst(ker, f64, level, r.shape[0], r.ctypes.data_as(P), amp[ker].ctypes.data_as(P),
                   ctypes.c_double(s.real), ctypes.c_double(s.imag))
        assert w <= math.exp(z) * bound + 64 * eps * math.exp(2 * z)


@pytest.mark.parametrize("decay", [0.0, 1.0, 80.0])
@pytest.mark.parametrize("phase", [0.5, 30.0, 2300.0])
def test_exponential(series, decay, phase):
    rng = np.random.default_rng(int(phase))
    n = 200000
    r = rng.uniform(0.3, 3.0, n).astype(np.float32)
    sre = (decay * rng.uniform(0, 1, n) / r).astype(np.float32)
    sim = (phase * rng.uniform(-1, 1, n) / r).astype(np.float32)
    P = ctypes.POINTER(ctypes.c_float)
    w = series.cexp_worst(n, sre.ctypes.data_as(P), sim.ctypes.data_as(P), r.ctypes.data_as(P))
    # the exponential, the reduced arguments, the polynomial and the product: five roundings
    assert w <= 5 * 2.0 ** -24
