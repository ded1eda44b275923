// Frequencies, device geometry, diagnostic entries and near-field assembly.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "g3_device.cuh"
#include "g3_series.cuh"

namespace g3 {

// ============================================================================
// Frequencies (float64)
// ============================================================================

// Multistep CQ with the BDF2 generating function: s_k = delta(zeta_k) / dt,
// delta(z) = (1 - z) + (1 - z)^2 / 2, zeta_k = lam exp(2 pi i k / K),
// computed for the unique half k = 0..Ku-1.
__global__ void k_freqs_bdf2(int K, int Ku, double lam, double dt, double2* sd, float2* sf) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Ku) return;
    double sn, cs;
    sincospi(2.0 * (double)k / (double)K, &sn, &cs);
    double omr = 1.0 - lam * cs, omi = -lam * sn;             // 1 - zeta
    double sqr = omr * omr - omi * omi, sqi = 2.0 * omr * omi;  // (1 - zeta)^2
    double dr = omr + 0.5 * sqr, di = omi + 0.5 * sqi;
    sd[k] = make_double2(dr / dt, di / dt);
    sf[k] = make_float2((float)(dr / dt), (float)(di / dt));
}

// Complete elliptic integral of the first kind, parameter m: K = pi / (2 AGM(1, sqrt(1 - m))).
__device__ double ellipk_agm(double m) {
    double a = 1.0, b = sqrt(1.0 - m);
    for (int it = 0; it < 40 && fabs(a - b) > 1e-16 * a; ++it) {
        double an = 0.5 * (a + b);
        b = sqrt(a * b);
        a = an;
    }
    return 3.141592653589793 / (2.0 * a);
}

// Jacobi sn, cn, dn of a real argument by the arithmetic-geometric mean and
// descending Landen recursion (Abramowitz & Stegun 16.4).
__device__ void jacobi_real(double u, double m, double* sn, double* cn, double* dn) {
    double a[24], c[24];
    a[0] = 1.0;
    double b = sqrt(1.0 - m);
    c[0] = sqrt(m);
    int N = 0;
    while (N < 22 && fabs(c[N]) > 1e-16) {
        double an = 0.5 * (a[N] + b);
        double cn1 = 0.5 * (a[N] - b);
        b = sqrt(a[N] * b);
        ++N;
        a[N] = an;
        c[N] = cn1;
    }
    double phi = ldexp(1.0, N) * a[N] * u;
    double phi_next = phi;
    for (int n = N; n >= 1; --n) {
        phi_next = phi;
        phi = 0.5 * (phi + asin(c[n] * sin(phi) / a[n]));
    }
    *sn = sin(phi);
    *cn = cos(phi);
    *dn = (N == 0) ? 1.0 : cos(phi) / cos(phi_next - phi);
}

// gCQ contour (Appendix A) with q = dt_max / dt_min:
//   s_l = gamma(sigma_l), omega_l = -4 K gamma'(sigma_l) / (2 pi i NQ),
// sn/cn/dn at complex sigma from the addition formula with Jacobi's
// imaginary transformation (A&S 16.21.1-3).
__global__ void k_freqs_gcq(int NQ, double dt_min, double dt_max, double2* s_out, double2* w_out) {
    int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= NQ) return;
    double q = dt_max / dt_min;
    double r = sqrt(2.0 * q - 1.0);
    double k = (q - r) / (q + r);
    double m = k * k;
    double Kk = ellipk_agm(m), Kp = ellipk_agm(1.0 - m);
    double x = -Kk + ((double)(l + 1) - 0.5) * 4.0 * Kk / (double)NQ;
    double y = 0.5 * Kp;
    double s, c, d, s1, c1, d1;
    jacobi_real(x, m, &s, &c, &d);
    jacobi_real(y, 1.0 - m, &s1, &c1, &d1);
    double den = c1 * c1 + m * s * s * s1 * s1;
    Cx<double> sn{s * d1 / den, c * d * s1 * c1 / den};
    Cx<double> cn{c * c1 / den, -s * d * s1 * d1 / den};
    Cx<double> dn{d * c1 * d1 / den, -m * s * c * s1 / den};
    double pref = 1.0 / (dt_min * (q - 1.0));
    double ik = 1.0 / k;
    Cx<double> num{ik + sn.x, sn.y}, dnm{ik - sn.x, -sn.y};
    Cx<double> ratio = cdiv(num, dnm);
    double2 sl = make_double2(pref * (r * ratio.x - 1.0), pref * r * ratio.y);
    Cx<double> cd = cmul(cn, dn);
    Cx<double> d2 = cmul(dnm, dnm);
    Cx<double> gp = cdiv(cd, d2);
    double fac = pref * r * 2.0 / k;
    gp.x *= fac;
    gp.y *= fac;
    // omega = -4K gp / (2 pi i NQ) = (4K / (2 pi NQ)) * i * gp
    double wfac = 4.0 * Kk / (2.0 * 3.141592653589793 * (double)NQ);
    s_out[l] = sl;
    w_out[l] = make_double2(-wfac * gp.y, wfac * gp.x);
}

g3_status launch_freqs_bdf2(g3_ctx* ctx, int K, int Ku, double lam, double dt, double* d_sd, float* d_sf) {
    k_freqs_bdf2<<<(Ku + 127) / 128, 128, 0, ctx->stream>>>(K, Ku, lam, dt, (double2*)d_sd, (float2*)d_sf);
    ctx->count("k_freqs_bdf2");
    G3_CUDA(cudaGetLastError());
    return G3_OK;
}

g3_status launch_freqs_gcq(g3_ctx* ctx, int NQ, double dt_min, double dt_max, double* d_s, double* d_w) {
    k_freqs_gcq<<<(NQ + 127) / 128, 128, 0, ctx->stream>>>(NQ, dt_min, dt_max, (double2*)d_s, (double2*)d_w);
    ctx->count("k_freqs_gcq");
    G3_CUDA(cudaGetLastError());
    return G3_OK;
}

// ============================================================================
// Geometry in cluster order
// ============================================================================

// One thread per cluster position p (element e = perm[p]): centroid
// ((v0 + v1) + v2) / 3, unit normal and area from the cross product, the
// 7-point degree-5 rule (Radon; constants from their closed forms) and the
// 4-point degree-3 conical-product rule (2-point Gauss-Jacobi in u with
// weight (1 - u), 2-point Gauss-Legendre in v), as offsets from the centroid.
__global__ void k_geometry(int ne, const double* __restrict__ verts, const int* __restrict__ tris,
                           const int* __restrict__ perm, GeomF gf, GeomD gd, float* chw, float* clw, float* qw,
                           float* ww, float* nw, float* q4w, float* w4w, double* cdw, double* qdw, double* wdw,
                           double* ndw, double* vdw, double* q4dw, double* w4dw) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= ne) return;
    const int E = ne;
    int e = perm[p];
    double v[3][3];
    for (int a = 0; a < 3; ++a)
        for (int k = 0; k < 3; ++k) v[a][k] = verts[3 * (size_t)tris[3 * e + a] + k];
    double c[3];
    for (int k = 0; k < 3; ++k) c[k] = ((v[0][k] + v[1][k]) + v[2][k]) / 3.0;
    double u[3], w[3];
    for (int k = 0; k < 3; ++k) {
        u[k] = v[1][k] - v[0][k];
        w[k] = v[2][k] - v[0][k];
    }
    double cr[3] = {u[1] * w[2] - u[2] * w[1], u[2] * w[0] - u[0] * w[2], u[0] * w[1] - u[1] * w[0]};
    double n2 = sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]);
    double area = 0.5 * n2;
    for (int k = 0; k < 3; ++k) {
        float hi = (float)c[k];
        chw[k * E + p] = hi;
        clw[k * E + p] = (float)(c[k] - (double)hi);
        cdw[k * E + p] = c[k];
        double nk = cr[k] / n2;
        nw[k * E + p] = (float)nk;
        ndw[k * E + p] = nk;
        for (int a = 0; a < 3; ++a) vdw[(a * 3 + k) * E + p] = v[a][k];
    }
    // 7-point rule
    const double r15 = sqrt(15.0);
    const double a1 = (6.0 - r15) / 21.0, b1 = (9.0 + 2.0 * r15) / 21.0;
    const double a2 = (6.0 + r15) / 21.0, b2 = (9.0 - 2.0 * r15) / 21.0;
    const double w1 = (155.0 - r15) / 1200.0, w2 = (155.0 + r15) / 1200.0;
    const double t3 = 1.0 / 3.0;
    const double L[7][3] = {{t3, t3, t3}, {a1, a1, b1}, {a1, b1, a1}, {b1, a1, a1},
                            {a2, a2, b2}, {a2, b2, a2}, {b2, a2, a2}};
    const double W[7] = {9.0 / 40.0, w1, w1, w1, w2, w2, w2};
    for (int q = 0; q < 7; ++q) {
        for (int k = 0; k < 3; ++k) {
            double y = L[q][0] * v[0][k] + L[q][1] * v[1][k] + L[q][2] * v[2][k];
            double off = y - c[k];
            qw[(q * 3 + k) * E + p] = (float)off;
            qdw[(q * 3 + k) * E + p] = off;
        }
        ww[q * E + p] = (float)(W[q] * area);
        wdw[q * E + p] = W[q] * area;
    }
    // 4-point conical product rule
    const double r6 = sqrt(6.0);
    const double uu[2] = {(4.0 - r6) / 10.0, (4.0 + r6) / 10.0};
    const double wu[2] = {(9.0 + r6) / 36.0, (9.0 - r6) / 36.0};
    const double vv[2] = {0.5 - 0.5 / sqrt(3.0), 0.5 + 0.5 / sqrt(3.0)};
    for (int ia = 0; ia < 2; ++ia)
        for (int ib = 0; ib < 2; ++ib) {
            int q = ia * 2 + ib;
            double l1 = uu[ia], l2 = vv[ib] * (1.0 - uu[ia]), l0 = 1.0 - l1 - l2;
            for (int k = 0; k < 3; ++k) {
                double y = l0 * v[0][k] + l1 * v[1][k] + l2 * v[2][k];
                q4w[(q * 3 + k) * E + p] = (float)(y - c[k]);
                q4dw[(q * 3 + k) * E + p] = y - c[k];
            }
            double wq = 2.0 * wu[ia] * 0.5 * area;
            w4w[q * E + p] = (float)wq;
            w4dw[q * E + p] = wq;
        }
}

g3_status launch_geometry(g3_ctx* ctx, g3_tree* t) {
    const int E = t->ne;
    // float arrays: ch 3, cl 3, q 21, w 7, n 3, q4 12, w4 4 = 53 per element
    const size_t nf = 53;
    // double arrays: c 3, q 21, w 7, n 3, v 9, q4 12, w4 4 = 59 per element
    const size_t nd = 59;
    G3_CUDA(t->d_geom_f.alloc(nf * E * sizeof(float)));
    G3_CUDA(t->d_geom_d.alloc(nd * E * sizeof(double) + 48 * sizeof(double)));
    float* F = t->d_geom_f.as<float>();
    double* D = t->d_geom_d.as<double>();
    GeomF gf{};
    gf.E = E;
    gf.ch = F;
    gf.cl = F + 3 * (size_t)E;
    gf.q = F + 6 * (size_t)E;
    gf.w = F + 27 * (size_t)E;
    gf.n = F + 34 * (size_t)E;
    gf.q4 = F + 37 * (size_t)E;
    gf.w4 = F + 49 * (size_t)E;
    GeomD gd{};
    gd.E = E;
    gd.c = D;
    gd.q = D + 3 * (size_t)E;
    gd.w = D + 24 * (size_t)E;
    gd.n = D + 31 * (size_t)E;
    gd.v = D + 34 * (size_t)E;
    gd.q4 = D + 43 * (size_t)E;
    gd.w4 = D + 55 * (size_t)E;
    gd.gl = D + 59 * (size_t)E;
    G3_CUDA(cudaMemcpyAsync((void*)gd.gl, ctx->gl.p, 48 * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream));
    DevBuf dv, dt;
    G3_CUDA(dv.alloc(t->verts.size() * sizeof(double)));
    G3_CUDA(dt.alloc(t->tris.size() * sizeof(int)));
    G3_CUDA(cudaMemcpyAsync(dv.p, t->verts.data(), t->verts.size() * sizeof(double), cudaMemcpyHostToDevice,
                            ctx->stream));
    G3_CUDA(cudaMemcpyAsync(dt.p, t->tris.data(), t->tris.size() * sizeof(int), cudaMemcpyHostToDevice, ctx->stream));
    k_geometry<<<(E + 127) / 128, 128, 0, ctx->stream>>>(
        E, dv.as<double>(), dt.as<int>(), t->d_perm.as<int>(), gf, gd, (float*)gf.ch, (float*)gf.cl, (float*)gf.q,
        (float*)gf.w, (float*)gf.n, (float*)gf.q4, (float*)gf.w4, (double*)gd.c, (double*)gd.q, (double*)gd.w,
        (double*)gd.n, (double*)gd.v, (double*)gd.q4, (double*)gd.w4);
    ctx->count("k_geometry");
    G3_CUDA(cudaGetLastError());
    G3_CUDA(cudaStreamSynchronize(ctx->stream));  // dv, dt are released on return
    t->gf = gf;
    t->gd = gd;
    return G3_OK;
}

// n-point Gauss-Legendre nodes and weights on [0, 1] (Newton iteration on the
// Legendre recurrence)
static void gauss_legendre01(int n, double* x01, double* w01) {
    for (int i = 0; i < n; ++i) {
        double x = std::cos(M_PI * (i + 0.75) / (n + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (x * p1 - p0) / (x * x - 1.0);
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) break;
        }
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= n; ++k) {
            double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = n * (x * p1 - p0) / (x * x - 1.0);
        x01[i] = 0.5 * (x + 1.0);
        w01[i] = 1.0 / ((1.0 - x * x) * dp * dp);  // (2 / ((1 - x^2) P'^2)) / 2
    }
}

// 24-point Gauss-Legendre nodes and weights on [-1, 1] (Newton iteration on
// the Legendre recurrence), uploaded once per context.
g3_status gl_table(g3_ctx* ctx) {
    const int n = 24;
    std::vector<double> tab(2 * n);
    for (int i = 0; i < n; ++i) {
        double x = std::cos(M_PI * (i + 0.75) / (n + 0.5));
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            double dp = n * (x * p1 - p0) / (x * x - 1.0);
            double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) {
                tab[i] = x;
                tab[n + i] = 2.0 / ((1.0 - x * x) * dp * dp);
                break;
            }
        }
        // recompute the weight at the converged node
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= n; ++k) {
            double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        double dp = n * (x * p1 - p0) / (x * x - 1.0);
        tab[i] = x;
        tab[n + i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
    G3_CUDA(ctx->gl.alloc(2 * n * sizeof(double)));
    G3_CUDA(upload(ctx->stream, ctx->gl.p, tab.data(), 2 * n * sizeof(double)));
    G3_CUDA(cudaStreamSynchronize(ctx->stream));  // (the context may change its stream)
    return G3_OK;
}

// ============================================================================
// Diagnostic entries
// ============================================================================

// Gauss-Legendre rule of the Sauter-Schwab quadrature (n = SS_N per coordinate)
constexpr int SS_N = 6;
struct SsRule {
    double x[SS_N], w[SS_N];
};

template <int KER, class T>
__global__ void k_entries(GeomF gf, GeomD gd, const int* __restrict__ tv, SsRule gr, const double2* __restrict__ sd,
                          const int* __restrict__ rows, const int* __restrict__ cols, int n,
                          const int* __restrict__ ku, const int* __restrict__ conj, int nk, double2* out) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)n * nk) return;
    int pr = (int)(idx / nk), m = (int)(idx % nk);
    int i = rows[pr], j = cols[pr];
    double2 s = sd[ku[m]];
    Cx<T> v;
    if constexpr (KER == G3_GAL_P1D || KER == G3_GAL_P1KP) {
        v = p1_entry<KER, T>(gf, gd, i, j, (T)s.x, (T)s.y);  // regular pairs (checked on the host)
    } else if constexpr (KER == G3_GAL_SLP) {
        int8_t px[3], py[3];
        const int cas = ss_classify(tv + 3 * (size_t)i, tv + 3 * (size_t)j, i == j, px, py);
        if (cas == 0) {
            v = gal_regular<T>(gf, gd, i, j, (T)s.x, (T)s.y);
        } else {  // Sauter-Schwab, one thread (diagnostic path)
            SsPanels P;
            ss_panels(gd, i, j, px, py, P);
            Cx<T> acc{0, 0};
            const int nr = ss_regions(cas);
            for (int q = 0; q < SS_N * SS_N * SS_N * SS_N * nr; ++q) {
                const int mreg = q / (SS_N * SS_N * SS_N * SS_N);
                int rem = q % (SS_N * SS_N * SS_N * SS_N);
                double g4[4], gw = 1.0;
                for (int a = 3; a >= 0; --a) {
                    g4[a] = gr.x[rem % SS_N];
                    gw *= gr.w[rem % SS_N];
                    rem /= SS_N;
                }
                double r, w;
                ss_point(P, cas, mreg, g4, gw, r, w);
                const T mm = (T)w * kexp(-(T)s.x * (T)r);
                T sn, cs;
                ksincos((T)s.y * (T)r, &sn, &cs);
                acc.x += mm * cs;
                acc.y -= mm * sn;
            }
            v = acc;
        }
    } else if (i == j && KER == G3_SLP) {  // self entries: float64 with the float64 frequency
        Cx<double> d = slp_self_f64(gd, i, s.x, s.y);
        v = Cx<T>{(T)d.x, (T)d.y};
    } else {
        v = colloc_entry<KER, T>(gf, gd, i, j, (T)s.x, (T)s.y);
    }
    double im = conj[m] ? -(double)v.y : (double)v.y;
    out[idx] = make_double2((double)v.x, im);
}

g3_status launch_entries(g3_ctx* ctx, const g3_tree* t, const g3_freqs* f, int kernel, int scheme, int prec,
                         const int* d_rows, const int* d_cols, int n, const int* d_ku, const int* d_conj, int nk,
                         double* d_out) {
    if (!t->p1 && scheme == G3_GALERKIN4x4 && kernel != G3_SLP)
        return fail(G3_EUNSUPPORTED, "g3_entries: the Galerkin scheme is implemented for G3_SLP");
    long long tot = (long long)n * nk;
    int blocks = (int)((tot + 127) / 128);
    if (tot == 0) return G3_OK;
    const double2* sd = f->d_sd.as<double2>();
    double2* out = (double2*)d_out;
    SsRule gr;
    gauss_legendre01(SS_N, gr.x, gr.w);
    const int* tv = t->d_tv.as<int>();
#define G3_ENT(K, T) \
    k_entries<K, T><<<blocks, 128, 0, ctx->stream>>>(t->gf, t->gd, tv, gr, sd, d_rows, d_cols, n, d_ku, d_conj, nk, out)
    if (t->p1 && kernel == G3_GAL_P1D && prec == G3_MIXED) G3_ENT(G3_GAL_P1D, float);
    else if (t->p1 && kernel == G3_GAL_P1D) G3_ENT(G3_GAL_P1D, double);
    else if (t->p1 && prec == G3_MIXED) G3_ENT(G3_GAL_P1KP, float);
    else if (t->p1) G3_ENT(G3_GAL_P1KP, double);
    else if (scheme == G3_GALERKIN4x4 && prec == G3_MIXED) G3_ENT(G3_GAL_SLP, float);
    else if (scheme == G3_GALERKIN4x4) G3_ENT(G3_GAL_SLP, double);
    else if (kernel == G3_SLP && prec == G3_MIXED) G3_ENT(G3_SLP, float);
    else if (kernel == G3_SLP) G3_ENT(G3_SLP, double);
    else if (kernel == G3_DLP && prec == G3_MIXED) G3_ENT(G3_DLP, float);
    else if (kernel == G3_DLP) G3_ENT(G3_DLP, double);
    else return fail(G3_EINVAL, "g3_entries: kernel %d not supported", kernel);
#undef G3_ENT
    ctx->count("k_entries");
    G3_CUDA(cudaGetLastError());
    return G3_OK;
}

// ============================================================================
// Near-field assembly
// ============================================================================

// One CTA per (near block, chunk of kch unique frequencies).  Threads run
// over the M_b * N_b entries of the block; each thread sets up an entry's series
// (below) once and evaluates it at the chunk's frequencies.  Layout of a block:
// [k][j][i] (frequency-major, column-major per frequency: the apply reads a
// column of rows with one coalesced load), complex, starting at offs[b].
//
// The frequencies come in the working precision (FreqT): a float64 pair per
// (entry, frequency) costs two float64-to-float32 conversions, which this part
// issues at its float64 rate.
template <class T>
struct FreqOf {
    using type = double2;
};
template <>
struct FreqOf<float> {
    using type = float2;
};
template <class T>
using FreqT = typename FreqOf<T>::type;

// Four warps per CTA: a 24 x 24 block is 18 warps of entries, 90 % of five rounds (75 %
// of three rounds of eight; 12,288 triangles 2.18 and 2.17 ms, small meshes fill the chip
// better).
constexpr int NEAR_NT = 128;
// Bound by the special-function unit before (float32: 3 results per point and frequency, 21
// per entry; now 3) or by float64 arithmetic; now by the instructions of the
// exponential and the series (140 per entry and frequency, 45 % of them multiply-adds).  12,288 triangles, 65 frequencies, float32: 2.77 -> 2.17 ms;
// 768 triangles, 17 frequencies, float64: 5.58 -> 2.19 ms.
template <int KER, class T>
__global__ void __launch_bounds__(NEAR_NT) k_near(int E, int kch, GeomF gf, GeomD gd, const FreqT<T>* __restrict__ sk,
                                              const BlockRange* __restrict__ ranges,
                                              const long long* __restrict__ offs, int Ku, Cx<T>* __restrict__ out) {
    using S = NearSeries<T>;
    const int b = blockIdx.x;
    const int k0 = blockIdx.y * kch;
    const BlockRange br = ranges[b];
    const int M = br.re - br.rb, N = br.ce - br.cb;
    const int MN = M * N;
    const int kn = min(kch, Ku - k0);
    // whole warps: lanes past the block's entries repeat its last one without storing
    for (int e0 = threadIdx.x & ~31; e0 < MN; e0 += blockDim.x) {
        const int eq = e0 + (threadIdx.x & 31), e = min(eq, MN - 1);
        const int i = br.rb + e % M, j = br.cb + e / M;
        Cx<T>* o = out + offs[b] + (long long)k0 * MN + e;
        const bool self = i == j;   // (DLP: 0; SLP: left to k_near_self, Galerkin: k_near_ss)
        const bool put = eq < MN && (!self || KER == G3_DLP);
        using P = std::conditional_t<KER == G3_GAL_SLP, Pair16<T>, Pair7<T>>;
        P p;
        // (a self entry's lane takes any other pair's geometry: its own has no distance)
        const int jj = !self || E == 1 ? j : (j > 0 ? j - 1 : j + 1);
        if constexpr (KER == G3_GAL_SLP) {
            // regular rule for every off-diagonal pair; pairs with a common
            // vertex are overwritten by k_near_ss
            if constexpr (sizeof(T) == 4)
                gal_setup(gf, i, jj, p);
            else
                gal_setup(gd, i, jj, p);
        } else {
            if constexpr (sizeof(T) == 4)
                pair_setup<KER>(gf, i, jj, p);
            else
                pair_setup<KER>(gd, i, jj, p);
        }
        constexpr int X = SERIES_MORE<KER>;
        T c[S::N2 + X + 1], rc, R;
        series_setup<KER, S::N2 + X, T>(p.r, p.a, c, rc, R);
        for (int kk = 0; kk < kn; ++kk) {
            const FreqT<T> s = sk[k0 + kk];
            const T x = -s.x * R, y = -s.y * R, z2 = fma(x, x, y * y);
            Cx<T> v;
            // one degree for the warp (a NaN distance goes point by point)
            if (__all_sync(0xffffffffu, z2 <= S::Z2 * S::Z2)) {
                Cx<T> w;
                if (__all_sync(0xffffffffu, z2 <= S::Z0 * S::Z0))
                    w = series_sum<S::N0 + X>(c, x, y, z2);
                else if (__all_sync(0xffffffffu, z2 <= S::Z1 * S::Z1))
                    w = series_sum<S::N1 + X>(c, x, y, z2);
                else
                    w = series_sum<S::N2 + X>(c, x, y, z2);
                v = cmul(cexp_acc(s.x, s.y, rc), w);
            } else if constexpr (KER == G3_GAL_SLP) {
                v = gal_eval<T>(p, s.x, s.y);
            } else {
                v = pair_eval<KER, T>(p, s.x, s.y);
            }
            if (self) v = Cx<T>{0, 0};
            if (put) o[(long long)kk * MN] = v;
        }
    }
}

// Galerkin near-field entries of pairs with a common vertex, a common edge or
// identical panels (Sauter-Schwab, SS_N^4 Gauss points per region): one CTA
// per pair.  The points' distances and weights are formed once in float64
// and kept in shared memory (as T); each frequency is then a sum over them
// (exp and sincos in T) reduced across the CTA.
template <class T, int NT>
__global__ void __launch_bounds__(NT) k_near_ss(GeomD gd, SsRule gr, const SsPair* __restrict__ pairs,
                                                 const double2* __restrict__ sd, int Ku, Cx<T>* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* rs = reinterpret_cast<T*>(smem_raw);
    const SsPair pr = pairs[blockIdx.x];
    const int nq = SS_N * SS_N * SS_N * SS_N;
    const int npts = nq * ss_regions(pr.cas);
    T* ws = rs + npts;
    __shared__ SsPanels P;
    if (threadIdx.x == 0) ss_panels(gd, pr.i, pr.j, pr.px, pr.py, P);
    __syncthreads();
    for (int q = threadIdx.x; q < npts; q += NT) {
        const int mreg = q / nq;
        int rem = q % nq;
        double g4[4], gw = 1.0;
        for (int a = 3; a >= 0; --a) {
            g4[a] = gr.x[rem % SS_N];
            gw *= gr.w[rem % SS_N];
            rem /= SS_N;
        }
        double r, w;
        ss_point(P, pr.cas, mreg, g4, gw, r, w);
        rs[q] = (T)r;
        ws[q] = (T)w;
    }
    __syncthreads();
    // each warp owns every (NT / 32)-th frequency: its lanes sum over all the
    // points and the warp reduces, with no block-wide barrier per frequency
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int k = wid; k < Ku; k += NT / 32) {
        const double2 s = sd[k];
        const T sre = (T)s.x, sim = (T)s.y;
        T ax = 0, ay = 0;
        for (int q = lane; q < npts; q += 32) {
            const T r = rs[q];
            const T m = ws[q] * kexp(-sre * r);
            T sn, cs;
            ksincos(sim * r, &sn, &cs);
            ax += m * cs;
            ay -= m * sn;
        }
        ax = warp_sum(ax);
        ay = warp_sum(ay);
        if (lane == 0) out[pr.off + (long long)k * pr.stride] = Cx<T>{ax, ay};
    }
}

// The same in float32, one region's points at a time: the points' distances and
// weights are formed in float-float from the tables (ss_point32; in float64 their
// ~85 operations per point took 25 of the 26 ms of the 5,120-triangle sphere's
// near field, 32 frequencies, 66,000 pairs), the sums over a region added up per
// frequency in shared memory.  Bound by the special-function unit: three results
// per point and frequency.  That near field: 26.3 -> 9.5 ms.
template <int NT>
__global__ void __launch_bounds__(NT) k_near_ss32(GeomD gd, const float4* __restrict__ tab,
                                                  const SsPair* __restrict__ pairs, const float2* __restrict__ sf,
                                                  int Ku, Cx<float>* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* rs = reinterpret_cast<float*>(smem_raw);          // [SS_Q]
    float* ws = rs + SS_Q;                                    // [SS_Q]
    Cx<float>* acc = reinterpret_cast<Cx<float>*>(ws + SS_Q); // [Ku]
    __shared__ SsEdges S;
    const SsPair pr = pairs[blockIdx.x];
    ss_edges(gd, pr, S);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nreg = ss_regions(pr.cas), first = ss_first_region(pr.cas);
    __syncthreads();
    for (int m = 0; m < nreg; ++m) {
        const float4* tm = tab + (size_t)(first + m) * 4 * SS_Q;
        for (int q = threadIdx.x; q < SS_Q; q += NT) {
            float zn;
            ss_point32<false>(S, tm, q, rs[q], ws[q], zn);
        }
        __syncthreads();
        // each warp owns every (NT / 32)-th frequency
        for (int k = wid; k < Ku; k += NT / 32) {
            const float2 s = sf[k];
            float ax = 0, ay = 0;
#pragma unroll 4
            for (int q = lane; q < SS_Q; q += 32) {
                const float r = rs[q];
                const float mm = ws[q] * kexp(-s.x * r);
                float sn, cs;
                ksincos(s.y * r, &sn, &cs);
                ax += mm * cs;
                ay -= mm * sn;
            }
            ax = warp_sum(ax);
            ay = warp_sum(ay);
            if (lane == 0) {
                Cx<float> v{ax, ay};
                if (m > 0) {
                    v.x += acc[k].x;
                    v.y += acc[k].y;
                }
                if (m == nreg - 1) out[pr.off + (long long)k * pr.stride] = v;
                else acc[k] = v;
            }
        }
        __syncthreads();  // the region's points are consumed
    }
}

// Linear continuous elements (element-local degrees of freedom): near-field
// entries of element pairs without a common vertex by the 4-point rule on both
// panels, one thread per element pair: the 16 point distances and weights are
// formed once and every frequency gives the pair's nine local entries; the
// pairs with a common vertex are written by k_near_ss_p1.  One CTA per (near
// block, chunk of KCH unique frequencies), layout [k][j][i] as k_near.
template <int OP, class T, int KCH>
__global__ void __launch_bounds__(256) k_near_p1(GeomF gf, GeomD gd, const int* __restrict__ tv,
                                                 const FreqT<T>* __restrict__ sk, const BlockRange* __restrict__ ranges,
                                                 const long long* __restrict__ offs, int Ku, Cx<T>* __restrict__ out) {
    const int b = blockIdx.x;
    const int k0 = blockIdx.y * KCH;
    const BlockRange br = ranges[b];
    const int M = br.re - br.rb, N = br.ce - br.cb;
    const int Me = M / 3, Ne = N / 3;
    const long long base = offs[b];
    const int kn = min(KCH, Ku - k0);
    for (int e = threadIdx.x; e < Me * Ne; e += blockDim.x) {
        const int pe = br.rb / 3 + e % Me, qe = br.cb / 3 + e / Me;
        bool shared = false;
        for (int x = 0; x < 3; ++x)
            for (int y = 0; y < 3; ++y) shared |= tv[3 * pe + x] == tv[3 * qe + y];
        if (shared) continue;
        T r[16], m[16], gz[16];
        T cab[9], nn = 0;
        if constexpr (sizeof(T) == 4)
            p1_pair_setup<OP>(gf, pe, qe, r, m, gz, cab, nn);
        else
            p1_pair_setup<OP>(gd, pe, qe, r, m, gz, cab, nn);
        const long long e0 = base + (long long)(3 * (qe - br.cb / 3)) * M + 3 * (pe - br.rb / 3);
        for (int kk = 0; kk < kn; ++kk) {
            const FreqT<T> s = sk[k0 + kk];
            Cx<T> v[9];
            p1_pair_eval<OP, T>(r, m, gz, cab, nn, s.x, s.y, v);
            Cx<T>* o = out + (long long)(k0 + kk) * M * N + e0;
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int c = 0; c < 3; ++c) o[a + (long long)c * M] = v[a * 3 + c];
        }
    }
}

// Linear elements, element pairs with a common vertex, a common edge or
// identical panels: the Sauter-Schwab maps (as k_near_ss) with the products
// lambda_a(x) lambda_b(y) of the local functions in the integrand; one CTA per
// element pair writes its 3 x 3 local entries at every frequency.  The points
// of one region (SS_N^4) are set up in float64 (T = float: in float-float from the
// tables) and kept in shared memory (their reference coordinates, distance and
// weight, and for the adjoint double layer
// -((x - y) . n_x) / r^2); each frequency's ten sums (the plain integral and
// the nine weighted ones) are reduced over the CTA and added into acc.
template <int OP, class T, int NT>
__global__ void __launch_bounds__(NT) k_near_ss_p1(GeomD gd, SsRule gr, const float4* __restrict__ tab,
                                                   const SsPair* __restrict__ pairs, const double2* __restrict__ sd,
                                                   const FreqT<T>* __restrict__ sk, int Ku, Cx<T>* __restrict__ out) {
    constexpr int NQ = SS_N * SS_N * SS_N * SS_N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* pt = reinterpret_cast<T*>(smem_raw);                    // [7][NQ]: x1, x2, y1, y2, r, w, g
    Cx<T>* acc = reinterpret_cast<Cx<T>*>(pt + 7 * NQ);         // [Ku][10]
    __shared__ SsPanels P;
    __shared__ SsEdges S32;
    const SsPair pr = pairs[blockIdx.x];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if constexpr (sizeof(T) == 4) ss_edges(gd, pr, S32);
    else if (threadIdx.x == 0) ss_panels(gd, pr.i, pr.j, pr.px, pr.py, P);
    for (int e = threadIdx.x; e < Ku * 10; e += NT) acc[e] = Cx<T>{0, 0};
    double n[3];
    for (int k = 0; k < 3; ++k) n[k] = gd.n[k * gd.E + pr.i];
    __syncthreads();
    const int nreg = ss_regions(pr.cas);
    for (int mreg = 0; mreg < nreg; ++mreg) {
        if constexpr (sizeof(T) == 4) {
            // float32: points in float-float from the tables
            const float4* tm = tab + (size_t)(ss_first_region(pr.cas) + mreg) * 4 * SS_Q;
            for (int q = threadIdx.x; q < NQ; q += NT) {
                float zn;
                ss_point32<OP == G3_GAL_P1KP>(S32, tm, q, pt[4 * NQ + q], pt[5 * NQ + q], zn);
                const float4 c = tm[2 * SS_Q + q], d = tm[3 * SS_Q + q];
                pt[0 * NQ + q] = c.z;
                pt[1 * NQ + q] = c.w;
                pt[2 * NQ + q] = d.x;
                pt[3 * NQ + q] = d.y;
                pt[6 * NQ + q] = -zn;
            }
        } else
        for (int q = threadIdx.x; q < NQ; q += NT) {
            int rem = q;
            double g4[4], gw = 1.0;
            for (int a = 3; a >= 0; --a) {
                g4[a] = gr.x[rem % SS_N];
                gw *= gr.w[rem % SS_N];
                rem /= SS_N;
            }
            double xh[2], yh[2];
            const double f = ss_map(pr.cas, mreg, g4[0], g4[1], g4[2], g4[3], xh, yh);
            double z[3], d2 = 0.0;
            for (int k = 0; k < 3; ++k) {
                const double x = P.P[0][k] + xh[0] * (P.P[1][k] - P.P[0][k]) + xh[1] * (P.P[2][k] - P.P[1][k]);
                const double y = P.Q[0][k] + yh[0] * (P.Q[1][k] - P.Q[0][k]) + yh[1] * (P.Q[2][k] - P.Q[1][k]);
                z[k] = x - y;
                d2 += z[k] * z[k];
            }
            const double r = sqrt(d2);
            pt[0 * NQ + q] = (T)xh[0];
            pt[1 * NQ + q] = (T)xh[1];
            pt[2 * NQ + q] = (T)yh[0];
            pt[3 * NQ + q] = (T)yh[1];
            pt[4 * NQ + q] = (T)r;
            pt[5 * NQ + q] = r > 0.0 ? (T)(gw * f * P.jac / r) : (T)0;
            pt[6 * NQ + q] = r > 0.0 ? (T)(-(z[0] * n[0] + z[1] * n[1] + z[2] * n[2]) / d2) : (T)0;
        }
        __syncthreads();
        // each warp owns every (NT / 32)-th frequency (no block-wide barrier per frequency)
        for (int k = wid; k < Ku; k += NT / 32) {
            const FreqT<T> s = sk[k];
            const T sre = s.x, sim = s.y;
            Cx<T> v[10];
#pragma unroll
            for (int u = 0; u < 10; ++u) v[u] = Cx<T>{0, 0};
            for (int q = lane; q < NQ; q += 32) {
                const T r = pt[4 * NQ + q];
                const T m = pt[5 * NQ + q] * kexp(-sre * r);
                T sn, cs;
                ksincos(sim * r, &sn, &cs);
                Cx<T> E{m * cs, -m * sn};
                if (OP == G3_GAL_P1KP) {
                    const T g = pt[6 * NQ + q], fr = (T)1 + sre * r, fi = sim * r;
                    E = Cx<T>{g * m * (fr * cs + fi * sn), g * m * (fi * cs - fr * sn)};
                }
                const T x1 = pt[q], x2 = pt[NQ + q], y1 = pt[2 * NQ + q], y2 = pt[3 * NQ + q];
                const T lx[3] = {(T)1 - x1, x1 - x2, x2}, ly[3] = {(T)1 - y1, y1 - y2, y2};
                v[9].x += E.x;
                v[9].y += E.y;
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        v[a * 3 + b].x += lx[a] * ly[b] * E.x;
                        v[a * 3 + b].y += lx[a] * ly[b] * E.y;
                    }
            }
#pragma unroll
            for (int u = 0; u < 10; ++u) {
                v[u].x = warp_sum(v[u].x);
                v[u].y = warp_sum(v[u].y);
            }
            if (lane < 10) {  // frequency k belongs to this warp alone
                Cx<T> t{0, 0};
#pragma unroll
                for (int u = 0; u < 10; ++u)
                    if (u == lane) t = v[u];
                acc[k * 10 + lane].x += t.x;
                acc[k * 10 + lane].y += t.y;
            }
        }
        __syncthreads();  // the region's points are consumed before the next region overwrites them
    }
    // local entries (Sauter-Schwab vertex order c, d = local vertices px[c], py[d]);
    // the float64 factors s^2, curl_a . curl_b and n_x . n_y once per CTA, in the
    // buffer of the consumed points
    T* s2 = pt;            // [Ku] Re, then [Ku] Im at NQ
    T* cn = pt + 2 * NQ;   // [9] curl products by (c, d), then n_x . n_y
    if (OP == G3_GAL_P1D) {
        for (int k = threadIdx.x; k < Ku; k += NT) {
            const double2 s = sd[k];
            s2[k] = (T)(s.x * s.x - s.y * s.y);
            s2[NQ + k] = (T)(2.0 * s.x * s.y);
        }
        if (threadIdx.x < 10) {
            const int c = threadIdx.x / 3, dd = threadIdx.x % 3;
            T v = 0;
            for (int kk = 0; kk < 3; ++kk)
                v += threadIdx.x < 9 ? (T)(gd.curl[(pr.px[c] * 3 + kk) * gd.E + pr.i] * gd.curl[(pr.py[dd] * 3 + kk) * gd.E + pr.j])
                                     : (T)(gd.n[kk * gd.E + pr.i] * gd.n[kk * gd.E + pr.j]);
            cn[threadIdx.x] = v;
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < Ku * 9; e += NT) {
        const int k = e / 9, c = (e % 9) / 3, dd = e % 3;
        const int a = pr.px[c], b = pr.py[dd];
        Cx<T> val = acc[k * 10 + c * 3 + dd];
        if (OP == G3_GAL_P1D) {
            const T s2r = s2[k], s2i = s2[NQ + k], cab = cn[c * 3 + dd], nn = cn[9];
            const Cx<T> i0 = acc[k * 10 + 9];
            val = Cx<T>{cab * i0.x + nn * (s2r * val.x - s2i * val.y), cab * i0.y + nn * (s2r * val.y + s2i * val.x)};
        }
        out[pr.off + (long long)k * pr.stride + a + (long long)b * pr.ldm] = val;
    }
}

// The pairs of a near field with a common vertex: one CTA per near block classifies
// its element pairs and appends the records (their order does not matter; one
// counter increment per warp).  p1: blocks of linear elements (three rows per
// element, the record's offset that of local functions (0, 0)).
__global__ void __launch_bounds__(256) k_ss_pairs(const int* __restrict__ tv, const BlockRange* __restrict__ ranges,
                                                  const long long* __restrict__ offs, int p1, SsPair* __restrict__ out,
                                                  int cap, int* __restrict__ count) {
    const int d = p1 ? 3 : 1;
    const BlockRange br = ranges[blockIdx.x];
    const int M = br.re - br.rb, N = br.ce - br.cb, Me = M / d, Ne = N / d;
    const int lane = threadIdx.x & 31;
    for (int e0 = 0; e0 < Me * Ne; e0 += blockDim.x) {
        const int e = e0 + threadIdx.x;
        SsPair q{};
        q.cas = SS_REGULAR;
        if (e < Me * Ne) {
            q.i = br.rb / d + e % Me;
            q.j = br.cb / d + e / Me;
            q.cas = ss_classify(tv + 3 * (size_t)q.i, tv + 3 * (size_t)q.j, q.i == q.j, q.px, q.py);
            q.stride = M * N;
            q.ldm = M;
            q.off = offs[blockIdx.x] + (long long)(d * q.j - br.cb) * M + (d * q.i - br.rb);
        }
        const unsigned mask = __ballot_sync(0xffffffffu, q.cas != SS_REGULAR);
        int base = 0;
        if (lane == 0 && mask) base = atomicAdd(count, __popc(mask));
        base = __shfl_sync(0xffffffffu, base, 0);
        const int at = base + __popc(mask & ((1u << lane) - 1u));
        if (q.cas != SS_REGULAR && at < cap) out[at] = q;
    }
}

g3_status launch_ss_pairs(g3_ctx* ctx, const g3_tree* t, g3_near* nf) {
    // at most one record per (element, element) of every vertex
    std::vector<int> deg(t->nv, 0);
    for (int32_t v : t->tris) ++deg[v];
    long long bound = 0;
    for (int d : deg) bound += (long long)d * d;
    if (bound > INT32_MAX) return fail(G3_EUNSUPPORTED, "assemble_near: too many element pairs with a common vertex");
    const int nb = (int)nf->order.size();
    if (nb == 0) return G3_OK;
    DevBuf cnt;
    G3_CUDA(cnt.alloc(sizeof(int)));
    G3_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int), ctx->stream));
    G3_CUDA(nf->d_ss.alloc((size_t)std::max<long long>(bound, 1) * sizeof(SsPair)));
    k_ss_pairs<<<nb, 256, 0, ctx->stream>>>(t->d_tv.as<int>(), nf->d_ranges.as<BlockRange>(),
                                            nf->d_offs.as<long long>(), t->p1 ? 1 : 0, nf->d_ss.as<SsPair>(),
                                            (int)bound, cnt.as<int>());
    ctx->count("k_ss_pairs");
    G3_CUDA(cudaGetLastError());
    int n = 0;
    G3_CUDA(cudaMemcpyAsync(&n, cnt.p, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    G3_CUDA(cudaStreamSynchronize(ctx->stream));
    if (n > bound) return fail(G3_ECUDA, "assemble_near: %d pairs with a common vertex, at most %lld expected", n, bound);
    nf->n_ss = n;
    return G3_OK;
}

// the Sauter-Schwab point table of the float32 kernels (SsEdges), once per context
static g3_status ss_table(g3_ctx* ctx) {
    if (ctx->ss_tab.p) return G3_OK;
    double gx[SS_N], gw[SS_N];
    gauss_legendre01(SS_N, gx, gw);
    static_assert(SS_Q == SS_N * SS_N * SS_N * SS_N, "points per region");
    std::vector<float> tab((size_t)13 * 4 * SS_Q * 4, 0.f);
    auto put = [&](int reg, int arr, int q, int c, double v) { tab[(((size_t)reg * 4 + arr) * SS_Q + q) * 4 + c] = (float)v; };
    auto put2 = [&](int reg, int arr, int q, int c, double v) {
        const float h = (float)v;
        put(reg, arr, q, c, h);
        put(reg, arr, q, c + 1, v - (double)h);
    };
    for (int cas = SS_VERTEX; cas <= SS_IDENTICAL; ++cas)
        for (int m = 0; m < ss_regions(cas); ++m)
            for (int q = 0; q < SS_Q; ++q) {
                int rem = q;
                double g4[4], w = 1.0;
                for (int a = 3; a >= 0; --a) {
                    g4[a] = gx[rem % SS_N];
                    w *= gw[rem % SS_N];
                    rem /= SS_N;
                }
                double x[2], y[2];
                const double f = ss_map(cas, m, g4[0], g4[1], g4[2], g4[3], x, y);
                const int reg = ss_first_region(cas) + m;
                put2(reg, 0, q, 0, cas == SS_VERTEX ? x[0] : x[0] - y[0]);
                put2(reg, 0, q, 2, cas == SS_IDENTICAL ? x[1] - y[1] : x[1]);
                put2(reg, 1, q, 0, cas == SS_VERTEX ? -y[0] : 0.0);
                put2(reg, 1, q, 2, cas == SS_IDENTICAL ? 0.0 : -y[1]);
                put2(reg, 2, q, 0, w * f);
                put(reg, 2, q, 2, x[0]);
                put(reg, 2, q, 3, x[1]);
                put(reg, 3, q, 0, y[0]);
                put(reg, 3, q, 1, y[1]);
            }
    DevBuf d;
    G3_CUDA(d.alloc(tab.size() * sizeof(float)));
    G3_CUDA(upload(ctx->stream, d.p, tab.data(), tab.size() * sizeof(float)));
    G3_CUDA(cudaStreamSynchronize(ctx->stream));  // (the context may change its stream)
    ctx->ss_tab.take(d);
    return G3_OK;
}

// the unique frequencies in the working precision
template <class T>
static const FreqT<T>* freqs_of(const g3_freqs* f) {
    if constexpr (sizeof(T) == 4) return f->d_sf.as<float2>();
    else return f->d_sd.as<double2>();
}

template <int OP, class T>
static g3_status launch_near_p1_t(g3_ctx* ctx, const g3_tree* t, const g3_freqs* f, g3_near* nf) {
    const int nb = (int)nf->order.size();
    constexpr int KCH = 16;
    dim3 grid(nb, (f->Ku + KCH - 1) / KCH);
    Cx<T>* o = reinterpret_cast<Cx<T>*>(nf->data.p);
    k_near_p1<OP, T, KCH><<<grid, 256, 0, ctx->stream>>>(t->gf, t->gd, t->d_tv.as<int>(), freqs_of<T>(f),
                                                          nf->d_ranges.as<BlockRange>(), nf->d_offs.as<long long>(),
                                                          f->Ku, o);
    ctx->count("k_near_p1");
    G3_CUDA(cudaGetLastError());
    if (nf->n_ss > 0) {
        SsRule gr;
        gauss_legendre01(SS_N, gr.x, gr.w);
        constexpr int NT = 256;
        const size_t smem = 7 * (size_t)SS_N * SS_N * SS_N * SS_N * sizeof(T) + 10 * (size_t)f->Ku * sizeof(Cx<T>);
        if (smem > ctx->smem_optin)
            return fail(G3_EUNSUPPORTED, "assemble_near: %zu bytes of shared memory for the singular pairs", smem);
        G3_CUDA(cudaFuncSetAttribute(k_near_ss_p1<OP, T, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        if (sizeof(T) == 4) {
            const g3_status st = ss_table(ctx);
            if (st != G3_OK) return st;
        }
        k_near_ss_p1<OP, T, NT><<<nf->n_ss, NT, smem, ctx->stream>>>(t->gd, gr, ctx->ss_tab.as<float4>(),
                                                                      nf->d_ss.as<SsPair>(), f->d_sd.as<double2>(),
                                                                      freqs_of<T>(f), f->Ku, o);
        ctx->count("k_near_ss_p1");
        G3_CUDA(cudaGetLastError());
    }
    return G3_OK;
}

// Self entries of the single layer in the near field, in float64: one warp per
// element p; the entry (p, p) of the diagonal leaf block sits at diag_base[p] +
// k * diag_mn[p] (diag_base[p] < 0: not in this tree's blocks).
//
// In polar coordinates about the centroid (slp_self_f64) the entry is
//   V(s) = (1 / 4 pi) sum_q w_q (1 - exp(-s rho_q)) / s
// over the 72 angular points (24 per edge), whose rho_q and w_q do not depend
// on the frequency.  Evaluated as it stands it takes an exponential, a sine
// and a cosine in float64 per point and frequency, on a part with two float64
// lanes per SM.  So the warp forms the points once and their moments
//   m0_n = sum_q w_q rho_q (rho_q / rmax)^n          (about 0)
//   m1_n = sum_q w_q ((rho_q - rc) / rh)^n           (about the middle rc of
//                                                     [rmin, rmax], rh its half width)
// for n < 32, and every lane (one frequency each) sums one of
//   |s| rmax <= 4:  V = (1/4 pi) sum_n (-z)^n / (n+1)! m0_n,            z = s rmax
//   |s| rh <= 4:    V = (1/4 pi s) (m1_0 - e^{-s rc} sum_n (-x)^n / n! m1_n),  x = s rh
// whose first omitted terms are below 4^32 / 32! = 7e-17; larger |s| rh sums the
// points directly.  The terms exceed the sum by up to e^4.  Measured in float64 over
// triangles from right-angled to slivers and all directions of s, against the points
// summed one by one (mean 2.0e-16, largest 1e-15): the first series 2.0e-16 and 7.7e-16
// up to |z| = 3.5, then 2.3e-16 and 8.8e-16; the second up to 4.3e-16 and 5.9e-15.
// Entries that are rounded to float32 take both; float64 entries the first one up to
// 3.5 and the points beyond (of the multistep frequencies none: |z| <= 3.3).
// Bound by the float64 pipe (the moments and the series).  12,288 elements x 65
// frequencies on a GB300: 14.0 -> 1.4 ms, and 1.1 ms with the series as Horner's rule on
// coefficients that hold the factorials (4 operations per term for 8); both that and
// running beside k_near: near field and its product 4.72 -> 4.27 ms.
struct SelfFact {   // 1 / n!
    double v[34];
    constexpr SelfFact() : v{} {
        v[0] = 1.0;
        for (int n = 1; n < 34; ++n) v[n] = v[n - 1] / n;
    }
};
__constant__ SelfFact SELF_IFACT;
constexpr int SELF_NM = 32;   // moments of each kind (one per lane)
constexpr int SELF_NW = 4;    // elements (warps) per CTA
__device__ __forceinline__ Cx<double> self_series(const double* c, double x, double y) {   // sum_n c_n (x + i y)^n
    double ar = c[SELF_NM - 1], ai = 0.0;
#pragma unroll 4
    for (int n = SELF_NM - 2; n >= 0; --n) {
        const double br = fma(x, ar, fma(-y, ai, c[n]));
        ai = fma(x, ai, y * ar);
        ar = br;
    }
    return {ar, ai};
}
template <class T>
__global__ void __launch_bounds__(SELF_NW * 32) k_near_self(GeomD gd, const double2* __restrict__ sd, int E, int Ku,
                                                            const long long* __restrict__ diag_base,
                                                            const int* __restrict__ diag_mn, Cx<T>* __restrict__ out) {
    __shared__ double pts[SELF_NW][2][72];           // rho_q, w_q
    __shared__ double mom[SELF_NW][2][SELF_NM];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = blockIdx.x * SELF_NW + warp;
    if (p >= E || diag_base[p] < 0) return;  // the whole warp (only warp-level synchronisation below)
    double* rho = pts[warp][0];
    double* wq = pts[warp][1];
    double rmin = 1e300, rmax = 0.0;
    for (int q = lane; q < 72; q += 32) {
        slp_self_point(gd, p, q / 24, q % 24, rho[q], wq[q]);
        rmin = fmin(rmin, rho[q]);
        rmax = fmax(rmax, rho[q]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        rmin = fmin(rmin, __shfl_xor_sync(0xffffffffu, rmin, o));
        rmax = fmax(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    }
    __syncwarp();
    const double rc = 0.5 * (rmin + rmax), rh = fmax(0.5 * (rmax - rmin), 1e-9 * rmax);
    {
        // lane = point (up to three per lane), running powers; 32 moments of a
        // kind are summed over the warp by halving exchanges, which leave
        // moment n in lane n
        for (int kind = 0; kind < (sizeof(T) == 4 ? 2 : 1); ++kind) {
            double b[3], t[3], v[SELF_NM];
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                const int q = lane + 32 * u;
                const bool in = q < 72;
                const double r = in ? rho[q] : 0.0, w = in ? wq[q] : 0.0;
                b[u] = kind == 0 ? r / rmax : (in ? (r - rc) / rh : 0.0);
                t[u] = kind == 0 ? w * r : w;
            }
#pragma unroll
            for (int n = 0; n < SELF_NM; ++n) {
                v[n] = t[0] + t[1] + t[2];
#pragma unroll
                for (int u = 0; u < 3; ++u) t[u] *= b[u];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const bool hi = (lane & o) != 0;
#pragma unroll
                for (int n = 0; n < o; ++n) {
                    const double send = hi ? v[n] : v[n + o], keep = hi ? v[n + o] : v[n];
                    v[n] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            mom[warp][kind][lane] = v[0] * SELF_IFACT.v[lane + (kind == 0 ? 1 : 0)];
        }
    }
    __syncwarp();
    const double* m0 = mom[warp][0];
    const double* m1 = mom[warp][1];
    for (int k = lane; k < Ku; k += 32) {
        const double2 s = sd[k];
        const double as = sqrt(s.x * s.x + s.y * s.y);
        Cx<double> v;
        if (as * rmax <= (sizeof(T) == 4 ? 4.0 : 3.5)) {
            v = self_series(m0, -s.x * rmax, -s.y * rmax);
        } else if constexpr (sizeof(T) == 8) {
            v = Cx<double>{0.0, 0.0};
            for (int q = 0; q < 72; ++q) {
                const Cx<double> g = g_expm1_over(Cx<double>{s.x * rho[q], s.y * rho[q]});
                v.x += wq[q] * rho[q] * g.x;
                v.y += wq[q] * rho[q] * g.y;
            }
        } else {
            Cx<double> sum{0.0, 0.0};  // sum_q w_q exp(-s rho_q)
            if (as * rh <= 4.0) {
                const Cx<double> acc = self_series(m1, -s.x * rh, -s.y * rh);
                double sn, cs;
                sincos(s.y * rc, &sn, &cs);
                const double e = exp(-s.x * rc);
                sum = cmul(acc, Cx<double>{e * cs, -e * sn});
            } else {
                for (int q = 0; q < 72; ++q) {
                    double sn, cs;
                    sincos(s.y * rho[q], &sn, &cs);
                    const double e = wq[q] * exp(-s.x * rho[q]);
                    sum.x += e * cs;
                    sum.y -= e * sn;
                }
            }
            v = cdiv(Cx<double>{m1[0] - sum.x, -sum.y}, Cx<double>{s.x, s.y});
        }
        out[diag_base[p] + (long long)k * diag_mn[p]] = Cx<T>{(T)(v.x * G3_INV4PI), (T)(v.y * G3_INV4PI)};
    }
}

// frequencies per CTA of k_near, in equal chunks: at most 24, and in float32 down to 8
// where the blocks alone leave resident CTAs (eight per SM) free.  Forming an entry's
// series costs about as much as four of its frequencies; in float64, where the pipe is
// full with few warps, splitting only adds to it (768 triangles, 17 frequencies: one
// chunk 2.19 ms, two 2.50 ms; float32 on 768 triangles, two of 9: 44 us).
template <class T>
static int near_chunk(const g3_ctx* ctx, int nb, int Ku) {
    int n = (Ku + 23) / 24;
    if (sizeof(T) == 4) n = std::max(n, std::min((Ku + 7) / 8, (8 * ctx->n_sm + nb - 1) / nb));
    return (Ku + n - 1) / n;
}

// Galerkin: near-field pairs with a common vertex (the SsPair records of k_ss_pairs) by
// k_near_ss32 or k_near_ss, after the regular rule for all pairs
template <class T>
static g3_status launch_near_galerkin(g3_ctx* ctx, const g3_tree* t, const g3_freqs* f, g3_near* nf) {
    const int nb = (int)nf->order.size();
    const int kch = near_chunk<T>(ctx, nb, f->Ku);
    dim3 grid(nb, (f->Ku + kch - 1) / kch);
    Cx<T>* o = reinterpret_cast<Cx<T>*>(nf->data.p);
    k_near<G3_GAL_SLP, T><<<grid, NEAR_NT, 0, ctx->stream>>>(t->ne, kch, t->gf, t->gd, freqs_of<T>(f),
                                                               nf->d_ranges.as<BlockRange>(),
                                                               nf->d_offs.as<long long>(), f->Ku, o);
    ctx->count("k_near");
    G3_CUDA(cudaGetLastError());
    if (nf->n_ss > 0) {
        constexpr int NT = 256;
        if constexpr (sizeof(T) == 4) {
            const g3_status st = ss_table(ctx);
            if (st != G3_OK) return st;
            const size_t smem = 2 * SS_Q * sizeof(float) + (size_t)f->Ku * sizeof(Cx<float>);
            k_near_ss32<NT><<<nf->n_ss, NT, smem, ctx->stream>>>(t->gd, ctx->ss_tab.as<float4>(), nf->d_ss.as<SsPair>(),
                                                                 f->d_sf.as<float2>(), f->Ku, o);
        } else {
            SsRule gr;
            gauss_legendre01(SS_N, gr.x, gr.w);
            const size_t smem = 2 * (size_t)SS_N * SS_N * SS_N * SS_N * 6 * sizeof(T);
            G3_CUDA(cudaFuncSetAttribute(k_near_ss<T, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_near_ss<T, NT><<<nf->n_ss, NT, smem, ctx->stream>>>(t->gd, gr, nf->d_ss.as<SsPair>(),
                                                                  f->d_sd.as<double2>(), f->Ku, o);
        }
        ctx->count("k_near_ss");
        G3_CUDA(cudaGetLastError());
    }
    return G3_OK;
}

g3_status launch_near(g3_ctx* ctx, const g3_tree* t, const g3_freqs* f, g3_near* nf, int kernel, int scheme) {
    const int nb = (int)nf->order.size();
    if (nb == 0) return G3_OK;
    if (t->p1) {
        if (kernel == G3_GAL_P1D)
            return nf->prec == G3_MIXED ? launch_near_p1_t<G3_GAL_P1D, float>(ctx, t, f, nf)
                                        : launch_near_p1_t<G3_GAL_P1D, double>(ctx, t, f, nf);
        return nf->prec == G3_MIXED ? launch_near_p1_t<G3_GAL_P1KP, float>(ctx, t, f, nf)
                                    : launch_near_p1_t<G3_GAL_P1KP, double>(ctx, t, f, nf);
    }
    if (scheme == G3_GALERKIN4x4) {
        if (kernel != G3_SLP) return fail(G3_EUNSUPPORTED, "assemble_near: the Galerkin scheme is implemented for G3_SLP");
        return nf->prec == G3_MIXED ? launch_near_galerkin<float>(ctx, t, f, nf)
                                    : launch_near_galerkin<double>(ctx, t, f, nf);
    }
    const BlockRange* rg = nf->d_ranges.as<BlockRange>();
    const long long* of = nf->d_offs.as<long long>();
    const long long* db = nf->d_diag_base.as<long long>();
    const int* dm = nf->d_diag_mn.as<int>();
    auto go = [&](auto zero) -> g3_status {
        using T = decltype(zero);
        Cx<T>* o = nf->data.as<Cx<T>>();
        const int kch = near_chunk<T>(ctx, nb, f->Ku);
        const dim3 grid(nb, (f->Ku + kch - 1) / kch);
        if (kernel == G3_SLP) {
            // the self entries (float64 pipe) run beside the regular ones (float32
            // arithmetic, stores) on the side stream; they write other entries
            G3_CUDA(cudaEventRecord(ctx->fork, ctx->stream));
            G3_CUDA(cudaStreamWaitEvent(ctx->side, ctx->fork, 0));
            k_near_self<T><<<(t->ne + SELF_NW - 1) / SELF_NW, SELF_NW * 32, 0, ctx->side>>>(
                t->gd, f->d_sd.as<double2>(), t->ne, f->Ku, db, dm, o);
            G3_CUDA(cudaEventRecord(ctx->join, ctx->side));
            k_near<G3_SLP, T><<<grid, NEAR_NT, 0, ctx->stream>>>(t->ne, kch, t->gf, t->gd, freqs_of<T>(f), rg, of, f->Ku, o);
            G3_CUDA(cudaStreamWaitEvent(ctx->stream, ctx->join, 0));
            ctx->count("k_near_self");
        } else {
            k_near<G3_DLP, T><<<grid, NEAR_NT, 0, ctx->stream>>>(t->ne, kch, t->gf, t->gd, freqs_of<T>(f), rg, of, f->Ku, o);
        }
        return G3_OK;
    };
    const g3_status st = nf->prec == G3_MIXED ? go(0.0f) : go(0.0);
    if (st != G3_OK) return st;
    ctx->count("k_near");
    G3_CUDA(cudaGetLastError());
    return G3_OK;
}

}  // namespace g3
