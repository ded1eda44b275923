#pragma once
// The power series of the near field's regular entries, and its exponential.  Needs Cx
// (g3_device.cuh) and the kernel kinds; compiles for the host, too.

namespace g3 {

// A regular entry at all its frequencies from one power series.  With r_c the middle of
// the points' distances and R their half range (d_q = (r_q - r_c) / R, |d_q| <= 1),
//   sum_q a_q exp(-s r_q) = exp(-s r_c) p(-s R),  p(z) = sum_n m_n z^n,  m_n = sum_q a_q d_q^n / n!,
// and with a_q (1 + s r_q) in place of a_q the coefficients (1 - n) m_n - (r_c / R) m_{n-1}.
// The coefficients are real and are formed once per entry, so that a frequency takes
// one exponential, one sine and cosine, and two multiply-adds per term
// (b_n = c_n + 2 Re z b_{n+1} - |z|^2 b_{n+2}) instead of an exponential, a sine and a
// cosine per point.  The degree goes by |z| of the warp's entries: N = 8, 12 or 16 in
// float32 up to |z| = 0.5, 1.25, 2.25, N = 14, 20 or 24 in float64 up to 0.5, 1.25, 2;
// beyond, point by point.  The first term left out is at most |z|^(N+1) / (N+1)! of
// p(0): 5.4e-9 in float32, 2.4e-17 in float64.  The double layer takes one degree more:
// its coefficient N + 1 holds (r_c / R) m_N, and without it the bound, against its factor
// 1 + s r_c, would be |z|^N / N! (9.7e-8 and 7e-16).  The terms grow to
// at most exp(|z|), but the phase s r_c is formed once, with the rounding of its product
// carried along, where the points' phases were rounded to |s r| 2^-24 each.
template <class T>
struct NearSeries;
template <>
struct NearSeries<float> {
    static constexpr int N0 = 8, N1 = 12, N2 = 16;
    static constexpr float Z0 = 0.5f, Z1 = 1.25f, Z2 = 2.25f;
};
template <>
struct NearSeries<double> {
    static constexpr int N0 = 14, N1 = 20, N2 = 24;
    static constexpr double Z0 = 0.5, Z1 = 1.25, Z2 = 2.0;
};

template <int KER>
constexpr int SERIES_MORE = KER == G3_DLP ? 1 : 0;   // degrees beyond N

// coefficients c[0 .. N] from NP points; returns r_c and R
template <int KER, int N, class T, int NP>
__host__ __device__ __forceinline__ void series_setup(const T (&r)[NP], const T (&a)[NP], T* c, T& rc, T& R) {
    T lo = r[0], hi = r[0];
#pragma unroll
    for (int q = 1; q < NP; ++q) {
        lo = min(lo, r[q]);
        hi = max(hi, r[q]);
    }
    rc = (T)0.5 * (lo + hi);
    R = max((T)0.5 * (hi - lo), rc * (T)0x1p-10);   // (points at one distance: any unit does)
    const T iR = (T)1 / R;
#pragma unroll
    for (int n = 0; n <= N; ++n) c[n] = 0;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const T d = (r[q] - rc) * iR;
        T t = a[q];
        c[0] += t;
#pragma unroll
        for (int n = 1; n <= N; ++n) {
            t *= d;
            c[n] += t;
        }
    }
    double f = 1.0;   // 1 / n!, folded at compile time
#pragma unroll
    for (int n = 2; n <= N; ++n) {
        f /= n;
        c[n] *= (T)f;
    }
    if constexpr (KER == G3_DLP) {
        const T g = rc * iR;
#pragma unroll
        for (int n = N; n >= 1; --n) c[n] = (T)(1 - n) * c[n] - g * c[n - 1];
    }
}
template <int N, class T>
__host__ __device__ __forceinline__ Cx<T> series_sum(const T* c, T x, T y, T z2) {
    const T x2 = x + x;
    T b1 = c[N], b2 = 0;
#pragma unroll
    for (int n = N - 1; n >= 1; --n) {
        const T b = fma(x2, b1, fma(-z2, b2, c[n]));
        b2 = b1;
        b1 = b;
    }
    return {fma(x, b1, fma(-z2, b2, c[0])), y * b1};
}

// exp(-(sre + i sim) r) with the products' rounding errors carried along.  float32:
// argument reduction with constants in two parts (Cody and Waite, Software Manual for the
// Elementary Functions, 1980): log 2 = 2839 / 2^12 + a rest, whose first part times an
// integer of at most 12 bits is exact, and pi / 2 = 201 / 2^7 + a rest, exact up to 16
// bits; |s| r_c stays below 2304 here (|s| R <= 2.25, R >= r_c / 1024).  That leaves at
// most log(2) / 2 and pi / 4, for the exponential function and for Taylor polynomials of
// degree 9 and 10 (2e-9).  Each part is within 5 x 2^-24 of the result.
__device__ __forceinline__ Cx<float> cexp_acc(float sre, float sim, float r) {
    const float u0 = -sre * r, u = fmaxf(u0, -200.0f);
    const float ul = u0 >= -200.0f ? fmaf(-sre, r, -u0) : 0.0f;
    const float m = rintf(u * 1.44269504f);
    float f = fmaf(-m, 2839.0f / 4096.0f, u);
    f = fmaf(-m, 3.19461849453e-5f, f) + ul;
    const float e = __expf(f) * exp2f(m);
    const float t = sim * r, tl = fmaf(sim, r, -t);
    const float n = rintf(t * 0.636619772f);
    float h = fmaf(-n, 201.0f / 128.0f, t);
    h = fmaf(-n, 4.83826794897e-4f, h) + tl;
    const float h2 = h * h;
    float sn = fmaf(h2, 1.0f / 362880.0f, -1.0f / 5040.0f);
    sn = fmaf(h2, sn, 1.0f / 120.0f);
    sn = fmaf(h2, sn, -1.0f / 6.0f);
    sn = fmaf(h * h2, sn, h);
    float cs = fmaf(h2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
    cs = fmaf(h2, cs, -1.0f / 720.0f);
    cs = fmaf(h2, cs, 1.0f / 24.0f);
    cs = fmaf(h2, cs, -0.5f);
    cs = fmaf(h2, cs, 1.0f);
    const int k = (int)n;
    const float c1 = (k & 1) ? sn : cs, s1 = (k & 1) ? cs : sn;   // cos, sin of n quarter turns + h
    const float c = ((k + 1) & 2) ? -c1 : c1, s = (k & 2) ? -s1 : s1;
    return {e * c, -e * s};
}
__device__ __forceinline__ Cx<double> cexp_acc(double sre, double sim, double r) {
    const double u = -sre * r, ul = fma(-sre, r, -u);
    double e = exp(u);
    if (e > 0.0 && e < 1e300) e = fma(e, ul, e);
    const double t = sim * r, tl = fma(sim, r, -t);
    double sn, cs;
    sincos(t, &sn, &cs);
    return {e * fma(-sn, tl, cs), -e * fma(cs, tl, sn)};
}

}  // namespace g3
