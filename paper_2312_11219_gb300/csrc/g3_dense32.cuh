#pragma once
// Float32 blocks with dense faces (M N <= dense_max), one CTA of four warps per
// block, four blocks per SM.
//
// Included by g3_aca_dev.cuh.  The blocks are small (24 x 24 and 48 x 48
// elements on the workloads) and a cross is a chain of short steps: residual
// face, its largest entry, fiber, eq. (norm), stopping test.  Bound by the
// instructions of the entries (28 special-function results each) and, where
// there are few blocks, by that chain: so every reduction takes one barrier,
// the fiber's residual is float-float (not float64), the earlier faces' entries
// are loaded before the entry is evaluated, and eq. (norm) takes four earlier
// crosses per pass: face inner products in float32; those of the fibers, the sum
// over the crosses, ||C^(l)||^2 and the stopping test in float64 (in float32 they
// would overflow from entries of 1e16 on, and the fibers reach the ratio of the
// largest entry to the pivot).  12,288-triangle single layer, 17,450 blocks: 13.1 ms (256
// threads, float64 fiber) -> 6.6 ms after the low-rank launch, which it
// overlaps (the same with the sums in float32).  1, 2, 4 and 8 warps per block: 80.8, 81.0, 80.7 and 82.6 ms for the
// whole set-up there, 1.79, 1.60, 1.49 and 1.46 ms for the step on the
// 768-triangle cube (320 blocks).

namespace g3 {

constexpr int DENSE32_NT = 128;

// per-block state
template <int W>
struct DenseSh {
    AcaArgs<float> A;        // the arguments with the geometry of the block's own mesh
    long long off[KU_MAX];   // pool offsets of the crosses
    Cx<float> hk[KU_MAX];    // f_p[k] during the face, H_p[i_l, j_l] during the fiber
    unsigned used[KU_MAX / 32];
    // the warps' parts of a reduction (two buffers), a broadcast value
    float2 part[2][W][4];    // <H_l, H_d> of four crosses
    double fpart[2][W][8];   // Re, Im of their <f_l, f_d>
    double norm2;            // ||C^(l)||^2
    int stop;
    uint2 key[2][W];
    float4 rel[W];
    long long bc;
};

// eight sums over a warp, the exchanges halving the values a lane carries.  Returns
// value (lane >> 2) (the four lanes of a group).
__device__ __forceinline__ double warp_sum8(double* v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 4, o = 16; n >= 1; n >>= 1, o >>= 1) {
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const double send = hi ? v[i] : v[i + n], keep = hi ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// largest candidate over the block's warps; buf alternates between calls
template <int W>
__device__ __forceinline__ uint2 dkey(DenseSh<W>& sh, ArgMaxT<float> a, int& buf) {
    uint2 k = warp_key(a);
    if ((threadIdx.x & 31) == 0) sh.key[buf][threadIdx.x >> 5] = k;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const uint2 y = sh.key[buf][w];
        if (w == 0 || y.x > k.x || (y.x == k.x && y.y < k.y)) k = y;
    }
    buf ^= 1;
    return k;
}

// The sampled residual of the approximant with ncl crosses at the 32 fixed
// samples over all frequencies (as confirm_stop); rk [SAMPLES / 4][Ku]: residual
// energies, on return [Ku] per frequency, summed in one order.  hs [SAMPLES][ncl]: H_p
// at the samples.
template <int KER, int W>
__device__ __noinline__ bool confirm_dense(DenseSh<W>& sh, const BlockRange br, int ncl, Cx<float> hpiv, Cx<float>* hs,
                                           double* rk) {
    constexpr int NT = 32 * W;
    const AcaArgs<float>& A = sh.A;
    const int tid = threadIdx.x, lane = threadIdx.x & 31;
    const int M = br.re - br.rb, N = br.ce - br.cb, MN = M * N, Ku = A.Ku;
    for (int e = tid; e < SAMPLES * ncl; e += NT) {
        const int p = e / SAMPLES, sm = e % SAMPLES;
        const int i = (2 * sm + 1) * M / (2 * SAMPLES), j = (2 * ((11 * sm) % SAMPLES) + 1) * N / (2 * SAMPLES);
        hs[e] = ldcx(A.pool + sh.off[p] + i + (long long)j * M);
    }
    __syncthreads();
    // squares scaled by a power of two near ||C^(l)||, which the entries do not exceed
    // by much (near the newest pivot, they could exceed it by all of float32's range),
    // float-float sums
    const int ex = min(max(sh.norm2 > 0.0 ? exponent_of(sh.norm2) / 2 : ilogbf(fmaxf(fabsf(hpiv.x), fabsf(hpiv.y))), -100), 100);
    const float sc = scalbnf(1.f, -ex);
    const double back = (double)scalbnf(1.f, ex);
    float2 rt = make_float2(0.f, 0.f), at = rt;
    // items (eight samples apart, frequency), four samples each
    for (int e = tid; e < (SAMPLES / 4) * Ku; e += NT) {
        const int q = e / Ku, k = e - q * Ku;
        float2 rs = make_float2(0.f, 0.f);
        for (int sm = q; sm < SAMPLES; sm += SAMPLES / 4) {
            const int i = (2 * sm + 1) * M / (2 * SAMPLES), j = (2 * ((11 * sm) % SAMPLES) + 1) * N / (2 * SAMPLES);
            const Cx<float> a = ent<KER, float>(A, br.rb + i, br.cb + j, k);
            Cx<float> r = a;
#pragma unroll 4
            for (int p = 0; p < ncl; ++p) {
                const Cx<float> c = cmul(hs[p * SAMPLES + sm], ldcx(A.pool + sh.off[p] + MN + k));
                r.x -= c.x;
                r.y -= c.y;
            }
            const float rx = r.x * sc, ry = r.y * sc, ax = a.x * sc, ay = a.y * sc;
            ff_add_prod(rs, rx, rx);
            ff_add_prod(rs, ry, ry);
            ff_add_prod(at, ax, ax);
            ff_add_prod(at, ay, ay);
        }
        ff_add(rt, rs.x, rs.y);
        rk[e] = ((double)rs.x + (double)rs.y) * back * back;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float rh = __shfl_xor_sync(0xffffffffu, rt.x, o), rl = __shfl_xor_sync(0xffffffffu, rt.y, o);
        const float ah = __shfl_xor_sync(0xffffffffu, at.x, o), al = __shfl_xor_sync(0xffffffffu, at.y, o);
        ff_add(rt, rh, rl);
        ff_add(at, ah, al);
    }
    if (lane == 0) sh.rel[threadIdx.x >> 5] = make_float4(rt.x, rt.y, at.x, at.y);
    __syncthreads();   // (rk is complete, too)
    rt = at = make_float2(0.f, 0.f);
    for (int w = 0; w < W; ++w) {
        const float4 v = sh.rel[w];
        ff_add(rt, v.x, v.y);
        ff_add(at, v.z, v.w);
    }
    sum_items<NT>(rk, SAMPLES / 4, Ku);
    __syncthreads();
    return (double)rt.x + (double)rt.y <= A.eps3 * A.eps3 * ((double)at.x + (double)at.y);
}

__host__ __device__ inline size_t dense_ws_bytes(int Cmax, int Ku) {
    return (((size_t)SAMPLES * (Cmax + 1) * sizeof(Cx<float>) + 255) & ~size_t(255)) +
           (((size_t)(SAMPLES / 4) * Ku * sizeof(double) + 255) & ~size_t(255));
}

// Algorithm 1 with the exact residual face (no low-rank approximation in the
// face, the paper's "No Lwr" variant).  A cross is stored as H (M x N,
// column-major) followed by f (Ku) and recorded with r = -1.
template <int KER>
__global__ void __launch_bounds__(DENSE32_NT, 4) k_dense32(const AcaArgs<float> P) {
    constexpr int NT = DENSE32_NT, W = NT / 32;
    __shared__ DenseSh<W> sh;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const AcaArgs<float>& A = sh.A;
    char* ws = P.ws + (size_t)blockIdx.x * P.ws_stride;
    Cx<float>* hs = reinterpret_cast<Cx<float>*>(ws);
    double* rk = reinterpret_cast<double*>(ws + (((size_t)SAMPLES * (P.Cmax + 1) * sizeof(Cx<float>) + 255) & ~size_t(255)));
    int kbuf = 0, pbuf = 0;
    // thread 0's value for the whole block
    auto bcast = [&](long long v) -> long long {
        if (tid == 0) sh.bc = v;
        __syncthreads();
        v = sh.bc;
        __syncthreads();
        return v;
    };
    for (int iter = 0;; ++iter) {
        int q0 = 0;
        if (tid == 0) {
            if (P.single >= 0)
                q0 = (iter == 0 && blockIdx.x == 0) ? P.single : -1;
            else {
                const int q = atomicAdd(P.queue_head, 1);
                q0 = q < P.n_far ? q : -1;
            }
        }
        const int qi = (int)bcast(q0);
        if (qi < 0) break;
        const int blk = P.queue[qi];
        if (tid == 0) {
            sh.A = P;
            if (P.geos) {
                const GeoDesc g = P.geos[P.bgeo[blk]];
                sh.A.gf = g.gf;
                sh.A.gd = g.gd;
                sh.A.sd = g.sd;
                sh.A.sf = g.sf;
                sh.A.Ku = g.Ku;
                sh.A.k_maxabs = g.k_maxabs;
            }
        }
        if (tid < KU_MAX / 32) sh.used[tid] = 0u;
        if (tid == 0) sh.norm2 = 0.0;
        __syncthreads();
        const BlockRange br = A.ranges[blk];
        const int M = br.re - br.rb, N = br.ce - br.cb, MN = M * N, Ku = A.Ku;
        const unsigned long long t_start = globaltimer_ns();
        long long ph[7] = {0, 0, 0, 0, 0, 0, 0};
        long long tclk = clock64();
        auto lap = [&](int i) {
            const long long tn = clock64();
            ph[i] += tn - tclk;
            tclk = tn;
        };
        int k_l = A.k1 ? A.k1[blk] : 0, nc = 0, computed = 0;
        long long entries = 0;
        bool zero_block = false, spilled = false;
        auto is_used = [&](int k) { return ((sh.used[k >> 5] >> (k & 31)) & 1u) != 0; };
        for (;;) {
            const long long need = (long long)MN + Ku;
            long long off = 0;
            if (tid == 0) {
                const unsigned long long o = atomicAdd(A.pool_ctr, (unsigned long long)need);
                off = (long long)o;
                if ((long long)o + need > A.pool_cap) {
                    atomicOr(A.status, ST_POOL_OVERFLOW);
                    off = -1;
                }
            }
            off = bcast(off);
            if (off < 0) {
                spilled = true;
                break;
            }
            Cx<float>* Hn = A.pool + off;
            Cx<float>* Fn = Hn + MN;
            // ---- face: exact residual at k_l, else up to three more frequencies ----
            const int cand[4] = {k_l, Ku - 1, Ku / 2, A.k_maxabs};
            ArgMaxT<float> am = amax_none<float>();
            int kf = -1;
            for (int c = 0; c < 4 && kf < 0; ++c) {
                const int kk = cand[c];
                bool skip = false;
                for (int d = 1; d < c; ++d) skip |= (cand[d] == kk);
                if (c > 0) skip |= is_used(kk);
                if (skip) continue;
                for (int p = tid; p < nc; p += NT) sh.hk[p] = ldcx(A.pool + sh.off[p] + MN + kk);
                __syncthreads();
                ArgMaxT<float> a = amax_none<float>();
                int i = tid % M, j = tid / M;
                const int di = NT % M, dj = NT / M;
                for (int e = tid; e < MN; e += NT) {
                    // the first eight earlier crosses' entries are on their way while
                    // this entry is evaluated
                    Cx<float> h[8];
#pragma unroll
                    for (int p = 0; p < 8; ++p)
                        if (p < nc) h[p] = ldcx(A.pool + sh.off[p] + e);
                    Cx<float> v = ent<KER, float>(A, br.rb + i, br.cb + j, kk);
#pragma unroll
                    for (int p = 0; p < 8; ++p)
                        if (p < nc) {
                            const Cx<float> x = cmul(sh.hk[p], h[p]);
                            v.x -= x.x;
                            v.y -= x.y;
                        }
#pragma unroll 4
                    for (int p = 8; p < nc; ++p) {
                        const Cx<float> x = cmul(sh.hk[p], ldcx(A.pool + sh.off[p] + e));
                        v.x -= x.x;
                        v.y -= x.y;
                    }
                    Hn[e] = v;
                    a = amax_better(a, ArgMaxT<float>{cabs2(v), i * N + j});
                    i += di;
                    j += dj;
                    if (i >= M) {
                        i -= M;
                        ++j;
                    }
                }
                entries += MN;
                __syncthreads();   // hk and used are read by the whole block up to here
                if (tid == 0) sh.used[kk >> 5] |= 1u << (kk & 31);
                const uint2 key = dkey<W>(sh, a, kbuf);
                __syncthreads();
                if (key.x != 0u && __uint_as_float(key.x - 1u) > tiny_norm2<float>()) {
                    am = ArgMaxT<float>{__uint_as_float(key.x - 1u), (int)key.y};
                    kf = kk;
                }
            }
            lap(0);
            if (kf < 0) {
                zero_block = (nc == 0);
                break;
            }
            k_l = kf;
            ++computed;
            const int ip = am.i / N, jp = am.i % N, ep = ip + jp * M;
            const Cx<float> hpiv = ldcx(Hn + ep);
            for (int p = tid; p < nc; p += NT) sh.hk[p] = ldcx(A.pool + sh.off[p] + ep);
            __syncthreads();
            lap(3);
            // ---- fiber ----
            fiber32<KER, NT>(A, tid, br.rb + ip, br.cb + jp, nc, sh.hk, cff_inv(hpiv),
                             [&](int p) { return A.pool + sh.off[p] + MN; }, Fn);
            entries += Ku;
            __syncthreads();
            lap(4);
            // ---- eq. (norm): four earlier crosses (the last: the new one) at a time ----
            double add = 0.0, own = 0.0;   // (warp 0: lane q of each pass holds cross d0 + q)
            for (int d0 = 0; d0 <= nc; d0 += 4) {
                Cx<float> h[4];
                double f[8];   // Re, Im
                const Cx<float>* Hd[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    h[q] = Cx<float>{0, 0};
                    f[2 * q] = f[2 * q + 1] = 0.0;
                    Hd[q] = d0 + q < nc ? A.pool + sh.off[d0 + q] : Hn;
                }
#pragma unroll 4
                for (int e = tid; e < MN; e += NT) {
                    const Cx<float> a = ldcx(Hn + e);
#pragma unroll
                    for (int q = 0; q < 4; ++q) cfmac(h[q], a, ldcx(Hd[q] + e));
                }
                for (int k = tid; k < Ku; k += NT) {
                    const Cx<double> a = ccast<double>(ldcx(Fn + k));
#pragma unroll
                    for (int q = 0; q < 4; ++q) {   // a conj(b)
                        const Cx<double> b = ccast<double>(ldcx(Hd[q] + MN + k));
                        f[2 * q] = fma(a.x, b.x, fma(a.y, b.y, f[2 * q]));
                        f[2 * q + 1] = fma(a.y, b.x, fma(-a.x, b.y, f[2 * q + 1]));
                    }
                }
                warp_sum_pair(h[0], h[1]);
                warp_sum_pair(h[2], h[3]);
                const double fs = warp_sum8(f);
                if ((lane & 3) == 0) sh.fpart[pbuf][wid][lane >> 2] = fs;
                if (lane == 0) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) sh.part[pbuf][wid][q] = make_float2(h[q].x, h[q].y);
                }
                __syncthreads();
                if (wid == 0 && lane < 4 && d0 + lane <= nc) {
                    float2 hs2 = sh.part[pbuf][0][lane];
                    double fx = sh.fpart[pbuf][0][2 * lane], fy = sh.fpart[pbuf][0][2 * lane + 1];
                    for (int w = 1; w < W; ++w) {
                        const float2 v = sh.part[pbuf][w][lane];
                        hs2.x += v.x;
                        hs2.y += v.y;
                        fx += sh.fpart[pbuf][w][2 * lane];
                        fy += sh.fpart[pbuf][w][2 * lane + 1];
                    }
                    const double re = (double)hs2.x * fx;
                    if (d0 + lane < nc) add += 2.0 * (re - (double)hs2.y * fy);
                    else own = re;
                }
                pbuf ^= 1;
            }
            if (wid == 0) {
                add += __shfl_xor_sync(0xffffffffu, add, 2);   // (lanes 0 to 3 hold them)
                add += __shfl_xor_sync(0xffffffffu, add, 1);
                own = __shfl_sync(0xffffffffu, own, nc & 3);
                if (lane == 0) {
                    const double n2 = sh.norm2 + (add + own);
                    sh.norm2 = n2;
                    sh.stop = fmax(own, 0.0) <= A.eps3 * A.eps3 * fmax(n2, 0.0);
                    sh.off[nc] = off;  // staged for the stop check
                }
            }
            int nu = 0;
            for (int u = 0; u < KU_MAX / 32; ++u) nu += __popc(sh.used[u]);
            const bool all = nu >= Ku;
            __syncthreads();
            const bool stop = sh.stop != 0;
            bool from_samples = false;
            if (stop && A.sample_check && !all) {
                from_samples = !confirm_dense<KER, W>(sh, br, nc + 1, hpiv, hs, rk);
                entries += (long long)SAMPLES * Ku;
                if (from_samples && tid == 0) atomicAdd(&A.counters[6], 1ull);
            }
            if (stop && !from_samples) {
                lap(5);
                break;
            }
            if (tid == 0) A.rec[(size_t)blk * A.Cmax + nc] = CrossRec{off, -1, ip, jp, kf};
            ++nc;
            lap(5);
            if (nc >= A.Cmax || all) break;
            // ---- next frequency: argmax over unused k of |f_l[k]| ----
            ArgMaxT<float> nk = amax_none<float>();
            for (int k = tid; k < Ku; k += NT)
                if (!is_used(k)) nk = amax_better(nk, ArgMaxT<float>{from_samples ? (float)rk[k] : cabs2(ldcx(Fn + k)), k});
            const uint2 key = dkey<W>(sh, nk, kbuf);
            lap(6);
            if (key.x == 0u || (int)key.y >= Ku) break;  // no finite candidate left
            k_l = (int)key.y;
        }
        if (tid == 0) {
            // a block that found the pool full goes to the spill queue and is
            // rerun from its start with a fresh pool segment
            A.r3[blk] = spilled ? 0 : nc;
            if (spilled) {
                const int q = atomicAdd(A.spill_n, 1);
                if (q < A.spill_cap) A.spill[q] = blk;
            }
            for (int i = 0; i < 7; ++i) A.blk_cycles[(size_t)blk * NPH + i] += ph[i];
            A.blk_cycles[(size_t)blk * NPH + 8] = (long long)t_start;
            A.blk_cycles[(size_t)blk * NPH + 9] = (long long)globaltimer_ns();
            atomicAdd(&A.counters[0], (unsigned long long)entries);
            atomicAdd(&A.counters[1], (unsigned long long)computed);
            if (zero_block && !spilled) atomicAdd(&A.counters[2], 1ull);
            for (int i = 0; i < 7; ++i) atomicAdd(&A.counters[8 + i], (unsigned long long)ph[i]);
        }
        __syncthreads();
    }
}

}  // namespace g3
