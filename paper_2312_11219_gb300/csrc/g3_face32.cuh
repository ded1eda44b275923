#pragma once
// Float32 faces of the three-way ACA: the partial-pivot ACA of one residual
// face and its recompression, with the face's columns in shared memory.
//
// Included by g3_aca_dev.cuh (which defines the block state, the line helpers
// and the dense residual working face) and used by the float32 kernels only.
//
// A face of a 192 x 192 block takes 20 to 40 ACA steps, and every step walks
// all earlier columns three times (row, column, norm).  With the columns in
// the global workspace each of those walks is a chain of L2 round trips
// (~25,000 SM cycles per step, measured); in shared memory it is a few hundred
// cycles of multiply-adds, so a step costs two barriers and the latency of one
// row and one column of the dense residual working face.

namespace g3 {

// Columns of the face: column t holds u_t (M values) and then v_t (N values).
// The first ncs columns live in shared memory, the others (faces of higher
// rank than the arena holds) in the CTA's workspace.  ld is 4 modulo 16, so
// that the parts of a gang, which read columns t, t + 1, .. at the same
// element, fall in different banks.
struct ColStore {
    Cx<float>* sm;
    Cx<float>* gm;
    int ncs, ld, M;
};
template <bool SM>
__device__ __forceinline__ Cx<float>* cs_u(const ColStore& c, int t) {
    if constexpr (SM) return c.sm + t * c.ld;
    else return t < c.ncs ? c.sm + t * c.ld : c.gm + (size_t)t * c.ld;
}
template <bool SM>
__device__ __forceinline__ Cx<float>* cs_v(const ColStore& c, int t) {
    return cs_u<SM>(c, t) + c.M;
}
__host__ __device__ inline int cs_ld(int M, int N) {
    const int l = M + N;
    return l + ((4 - l) & 15);   // <= M + N + CS_PAD - 1
}

// four sums over a warp with six exchanges instead of twenty: the halves of
// the warp first split the values between them, then the lanes below.
// Lanes 0-15 get (sum a, sum b), lanes 16-31 (sum c, sum d).
__device__ __forceinline__ float2 warp_sum4(float a, float b, float c, float d) {
    const int lane = threadIdx.x & 31;
    const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
    float x = h16 ? c : a, y = h16 ? d : b;
    x += __shfl_xor_sync(0xffffffffu, h16 ? a : c, 16);
    y += __shfl_xor_sync(0xffffffffu, h16 ? b : d, 16);
    float z = (h8 ? y : x) + __shfl_xor_sync(0xffffffffu, h8 ? x : y, 8);
    z += __shfl_xor_sync(0xffffffffu, z, 4);
    z += __shfl_xor_sync(0xffffffffu, z, 2);
    z += __shfl_xor_sync(0xffffffffu, z, 1);
    // every lane of a half holds its x sum (lanes 0-7, 16-23) or its y sum
    const float w = __shfl_xor_sync(0xffffffffu, z, 8);
    return h8 ? make_float2(w, z) : make_float2(z, w);
}

// two complex sums over a warp, known to every lane
__device__ __forceinline__ void warp_sum_pair(Cx<float>& p, Cx<float>& q) {
    const float2 v = warp_sum4(p.x, p.y, q.x, q.y);
    const bool hi = (threadIdx.x & 16) != 0;
    const float ox = __shfl_xor_sync(0xffffffffu, v.x, 16), oy = __shfl_xor_sync(0xffffffffu, v.y, 16);
    p = hi ? Cx<float>{ox, oy} : Cx<float>{v.x, v.y};
    q = hi ? Cx<float>{v.x, v.y} : Cx<float>{ox, oy};
}

// warp argmax of non-negative float32 values, ties to the smallest index:
// {value bits + 1 (0: no candidate), index}
__device__ __forceinline__ uint2 warp_key(ArgMaxT<float> a) {
    const unsigned enc = a.v >= 0.f ? __float_as_uint(a.v + 0.f) + 1u : 0u;
    const unsigned mx = __reduce_max_sync(0xffffffffu, enc);
    const unsigned ix = __reduce_min_sync(0xffffffffu, enc == mx ? (unsigned)a.i : 0xffffffffu);
    return make_uint2(mx, ix);
}
// the block's candidate from its warps' (after a barrier)
template <int NT>
__device__ __forceinline__ ArgMaxT<float> block_key(const uint2* k) {
    uint2 b = k[0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) {
        const uint2 y = k[w];
        if (y.x > b.x || (y.x == b.x && y.y < b.y)) b = y;
    }
    if (b.x == 0u) return amax_none<float>();
    return ArgMaxT<float>{__uint_as_float(b.x - 1u), (int)b.y};
}

// rows already taken by the face ACA: a bit mask in shared memory (blocks of
// more than 32 USED_W rows: bytes in the workspace)
__device__ __forceinline__ bool row_used(const BlockSh<float>& S, const Ws<float>& w, int i) {
    return S.M <= 32 * USED_W ? (S.usedm[i >> 5] >> (i & 31)) & 1u : w.used[i] != 0;
}

// the part of a gang in sum_t u_t[fix] conj(v_t[v]) (ROW) or
// sum_t u_t[v] conj(v_t[fix]) over the face's columns t < m
template <bool ROW>
__device__ __forceinline__ Cx<float> cur_sum(const ColStore& c, int fix, int v, int m, int part, int G) {
    Cx<float> s0{0, 0}, s1{0, 0}, s2{0, 0}, s3{0, 0};
    const int ou = ROW ? fix : v, ov = c.M + (ROW ? v : fix);
    const int ms = min(m, c.ncs);
    int t = part;
    for (; t + 3 * G < ms; t += 4 * G) {
        const Cx<float>* p = c.sm + t * c.ld;
        const int st = G * c.ld;
        const Cx<float> a0 = ldcx(p + ou), a1 = ldcx(p + st + ou), a2 = ldcx(p + 2 * st + ou), a3 = ldcx(p + 3 * st + ou);
        const Cx<float> b0 = ldcx(p + ov), b1 = ldcx(p + st + ov), b2 = ldcx(p + 2 * st + ov), b3 = ldcx(p + 3 * st + ov);
        cfmac(s0, a0, b0);
        cfmac(s1, a1, b1);
        cfmac(s2, a2, b2);
        cfmac(s3, a3, b3);
    }
    for (; t < ms; t += G) {
        const Cx<float>* p = c.sm + t * c.ld;
        cfmac(s0, ldcx(p + ou), ldcx(p + ov));
    }
    for (; t < m; t += G) {  // columns beyond the arena
        const Cx<float>* p = c.gm + (size_t)t * c.ld;
        cfmac(s1, ldcx(p + ou), ldcx(p + ov));
    }
    return Cx<float>{(s0.x + s1.x) + (s2.x + s3.x), (s0.y + s1.y) + (s2.y + s3.y)};
}

// One residual row (ROW: fixed row `fix`) or column of the face:
//   ENTRY - sum_p f_p[kf] (U_p V_p^H) - sum_{t<m} u_t v_t^H
// read from the dense residual working face D (which holds the first two
// terms), or evaluated with the earlier crosses' tables.  G threads share an
// element.  Writes the line to out and returns the thread's largest |.|^2
// (columns: over the rows not yet used, `skip` being used too).
template <int KER, int NT, bool ROW>
__device__ __forceinline__ ArgMaxT<float> line32(const AcaArgs<float>& A, const Ws<float>& w, BlockSh<float>& S,
                                                 const FaceTab<float>& F, const ColStore& c, int fix, int skip, int kf,
                                                 int m, Cx<float>* out, const Cx<float>* D, float* n2 = nullptr) {
    const int tid = threadIdx.x;
    const int M = S.M, N = S.N;
    const int L = ROW ? N : M;
    // D: one pass over the line where it fits; else as many passes as the
    // entries and tables want (gang_size)
    const int G = D ? (L * 4 <= NT ? 4 : (L * 2 <= NT ? 2 : 1)) : gang_size<NT>(L);
    const int per = NT / G, part = tid % G;
    ArgMaxT<float> am = amax_none<float>();
    for (int base = 0; base < L; base += per) {
        const int v = base + tid / G;
        Cx<float> acc{0, 0};
        bool cand = false;
        if (v < L) {
            if (D) {
                if (part == 0) acc = ldcx(D + (ROW ? (size_t)fix * N + v : (size_t)v * N + fix));
            } else {
                const long long te = tid == 0 ? clock64() : 0;
                acc = ent_part<KER, float>(A, S.rb + (ROW ? fix : v), S.cb + (ROW ? v : fix), kf, part, G);
                if (tid == 0) S.sub[10] += clock64() - te;
                Cx<float> s0{0, 0}, s1{0, 0}, s2{0, 0}, s3{0, 0};
                cross_sum<float, ROW>(A, F, v, part, G, s0, s1, s2, s3);
                acc.x -= (s0.x + s1.x) + (s2.x + s3.x);
                acc.y -= (s0.y + s1.y) + (s2.y + s3.y);
            }
            cand = part == 0 && (ROW || (v != skip && !row_used(S, w, v)));
            const Cx<float> q = cur_sum<ROW>(c, fix, v, m, part, G);
            acc.x -= q.x;
            acc.y -= q.y;
        }
        for (int o = G >> 1; o > 0; o >>= 1) {
            const Cx<float> y = shfl_xor_c(acc, o);
            acc.x += y.x;
            acc.y += y.y;
        }
        if (part == 0 && v < L) {
            out[v] = acc;
            if (n2) *n2 += cabs2(acc);
            if (cand) am = amax_better(am, ArgMaxT<float>{cabs2(acc), v});
        }
    }
    if (tid == 0) S.entries += L;
    return am;
}

// The residual of the face approximant (m columns) at the 32 fixed samples,
// one warp per sample; |R_s|^2 to S.samp.
template <int KER, int NT>
__device__ void samples32(const AcaArgs<float>& A, BlockSh<float>& S, const FaceTab<float>& F, const ColStore& c,
                          int kf, int m, const Cx<float>* D) {
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int M = S.M, N = S.N;
    for (int sm = wid; sm < SAMPLES; sm += NT / 32) {
        const int i = (2 * sm + 1) * M / (2 * SAMPLES), j = (2 * ((11 * sm) % SAMPLES) + 1) * N / (2 * SAMPLES);
        Cx<float> e{0, 0};
        if (lane == 0) e = D ? ldcx(D + (size_t)i * N + j) : ent<KER, float>(A, S.rb + i, S.cb + j, kf);
        Cx<float> acc{0, 0};
        for (int q = lane; q < F.ncol; q += 32)
            cfma(acc, S.fk[F.colP[q]], cmulc(A.pool[F.colU[q] + i], A.pool[F.colV[q] + j]));
        for (int t = lane; t < m; t += 32) cfmac(acc, ldcx(cs_u<false>(c, t) + i), ldcx(cs_v<false>(c, t) + j));
        acc.x = warp_sum(acc.x);
        acc.y = warp_sum(acc.y);
        if (lane == 0) S.samp[sm] = cabs2d(Cx<float>{e.x - acc.x, e.y - acc.y});
    }
    if (threadIdx.x == 0) S.entries += SAMPLES;
    __syncthreads();
}

// max(eps_face^2 ||S_m||_F^2, floor^2)
__device__ __forceinline__ double face_bound2(const AcaArgs<float>& A, const BlockSh<float>& S) {
    return fmax(A.eps_face * A.eps_face * fmax(S.fsn2, 0.0), A.face_floor * A.face_floor * (S.norm2 * S.iku));
}
__device__ __forceinline__ FaceThr face_thr(double b) {
    const int e = b > 0.0 ? min(max(exponent_of(b), -120), 120) : 0;
    b = fmin(b * pow2_of(-e), 3e38);
    const float h = (float)b;
    return FaceThr{make_float2(h, (float)(b - (double)h)), scalbnf(1.f, -e)};
}
// nu2 nv2 <= bound (an overflowing left side exceeds it, a vanishing one does not)
__device__ __forceinline__ bool face_passes(const FaceThr& t, float nu2, float nv2) {
    const float a = nu2 * t.scale, p = a * nv2;
    return (p - t.v.x) + (fmaf(a, nv2, -p) - t.v.y) <= 0.f;
}

// Partial-pivot ACA of the residual face at frequency kf.  Returns the rank m;
// c holds the crosses.  Rows, columns and tests as in the float64 face_aca:
//   ||u_m|| ||v_m|| <= eps_face ||S_m||_F  (or the absolute floor), confirmed on
//   the sample entries.
// Two barriers per step: the residual row and its largest entry; then the
// column of that entry, the norms of both and the test.  With the dense
// residual working face D, ||D||_F stands for ||S_m||_F: the two agree to
// eps_face where the test can pass, and D's norm is a by-product of forming it.
// Without D, ||S_m||_F is the recursive
//   ||S_m||^2 = ||S_{m-1}||^2 + 2 Re sum_t (u_t^H u_m)(v_m^H v_t) + ||u_m||^2 ||v_m||^2
// (two more barriers; the sum over t took a third of the step's instructions).
// The sums over a vector are float32; their products and what is summed of them are
// float64 in one warp, as in face_aca, and with D the test is taken in float-float on a
// scaled bound that one warp forms per face and every step reads from shared memory
// (float64 in every warp would hold each step for its pipe; the bound in registers
// costs 1 % of the whole launch in spills: 12,288-triangle single layer 72.4 and
// 71.3 ms).
template <int KER, int NT>
__device__ int face32(const AcaArgs<float>& A, const Ws<float>& w, BlockSh<float>& S, int kf, unsigned char* arena,
                      ColStore& c) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int M = S.M, N = S.N, nc = S.ncross;
    const int cap = min(min(M, N), A.RF);
    c = ColStore{nullptr, w.uw, 0, cs_ld(M, N), M};
    if (kf < 0 || kf >= A.Ku) {  // cannot happen: every caller passes a checked index
        if (tid == 0) atomicOr(A.status, ST_BAD_INDEX);
        return 0;
    }
    for (int p = tid; p < nc; p += NT) S.fk[p] = Fp(A, S, p)[kf];
    long long tf = clock64();
    FaceTab<float> F = facetab_build<float, NT>(A, w, S, arena);
    if (M <= 32 * USED_W) {
        if (tid < USED_W) S.usedm[tid] = 0u;
    } else {
        for (int i = tid; i < M; i += NT) w.used[i] = 0;
    }
    __syncthreads();
    const Cx<float>* D = nullptr;
    size_t off = (facetab_smem_bytes<float>() + 255) & ~size_t(255);
    if constexpr (KER != G3_SEPARABLE) {
        if (w.dres && (long long)M * N <= A.drf_max) {
            face_dense_residual<KER, float, NT>(A, w.dres, S, F, kf);
            D = w.dres;
            // the tables are not needed any more: only the row buffer stays
            F.ncol = 0;
            F.row = N <= ROWMAX ? reinterpret_cast<Cx<float>*>(arena) : w.row;
            off = N <= ROWMAX ? ((size_t)N * sizeof(Cx<float>) + 15) & ~size_t(15) : 0;
            sublap(S, 11, tf);
        }
    }
    c.sm = reinterpret_cast<Cx<float>*>(arena + off);
    c.ncs = (size_t)A.arena_bytes > off ? (int)(((size_t)A.arena_bytes - off) / ((size_t)c.ld * sizeof(Cx<float>))) : 0;
    c.ncs = min(c.ncs, A.RF);
    int m = 0, irow = 0;
    bool converged = false;
    // own <= max(eps^2 ||S||^2, floor^2); S.fsn2: ||S_m||_F^2
    if (wid == 0) {
        double n2 = D && lane < NW ? S.crs[lane] : 0.0;
        n2 = warp_sum(n2);
        if (lane == 0) {
            S.fsn2 = n2;
            S.thr = face_thr(face_bound2(A, S));
        }
    }
    __syncthreads();
    while (m < cap) {
        // ---- the residual row ----
        if (F.ncol > 0) {
            // (the current columns' coefficients are read from c directly)
            for (int q = tid; q < F.ncol; q += NT) F.coef[q] = cmul(S.fk[F.colP[q]], A.pool[F.colU[q] + irow]);
            __syncthreads();
        }
        ArgMaxT<float> am = line32<KER, NT, true>(A, w, S, F, c, irow, -1, kf, m, F.row, D);
        {
            const uint2 k = warp_key(am);
            if (lane == 0) S.key[0][wid] = k;
        }
        if (tid == 0) {
            if (M <= 32 * USED_W) S.usedm[irow >> 5] |= 1u << (irow & 31);
            else w.used[irow] = 1;
        }
        __syncthreads();
        am = block_key<NT>(S.key[0]);
        // a row counts as nonzero when |delta|^2 is a normal number of the
        // working precision (below that the entries are far under any tolerance)
        if (!(am.v > tiny_norm2<float>())) {
            // zero residual row: next unused row in index order
            ArgMaxT<float> un = amax_none<float>();
            for (int i = tid; i < M; i += NT)
                if (!row_used(S, w, i)) un = amax_better(un, ArgMaxT<float>{0.f, i});
            un = block_argmax<NT>(un, S.am);
            if (un.v < 0.f) break;  // no row with a nonzero residual left
            irow = un.i;
            continue;
        }
        const int jp = am.i;
        sublap(S, 6, tf);
        // ---- v = conj(row / delta), the column of the pivot ----
        // delta is scaled to magnitude ~1 first, so that a tiny pivot of a strongly
        // damped face cannot overflow 1 / |delta|^2 (|row[j]| <= |delta|)
        const Cx<float> delta = F.row[jp];
        const float sc = 1.f / fmaxf(fabsf(delta.x), fabsf(delta.y));
        const Cx<float> ds{delta.x * sc, delta.y * sc};
        const float dn = 1.f / cabs2(ds);
        if (F.ncol > 0) {
            for (int q = tid; q < F.ncol; q += NT) F.coef[q] = cmul(S.fk[F.colP[q]], cconj(A.pool[F.colV[q] + jp]));
            __syncthreads();
        }
        Cx<float>* um = cs_u<false>(c, m);
        Cx<float>* vm = um + M;
        float nv2 = 0, nu2 = 0;
        for (int j = tid; j < N; j += NT) {
            const Cx<float> rj = F.row[j];
            const Cx<float> q = cmulc(Cx<float>{rj.x * sc, rj.y * sc}, ds);  // (row / s) conj(delta / s)
            const Cx<float> v{q.x * dn, -q.y * dn};                          // conj(row / delta)
            vm[j] = v;
            nv2 += cabs2(v);
        }
        ArgMaxT<float> nx = line32<KER, NT, false>(A, w, S, F, c, jp, irow, kf, m, um, D, &nu2);
        {
            const uint2 k = warp_key(nx);
            nu2 = warp_sum(nu2);
            nv2 = warp_sum(nv2);
            if (lane == 0) {
                S.key[1][wid] = k;
                S.nrm[wid] = make_float2(nu2, nv2);
            }
        }
        __syncthreads();
        nx = block_key<NT>(S.key[1]);
        nu2 = nv2 = 0;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const float2 x = S.nrm[q];
            nu2 += x.x;
            nv2 += x.y;
        }
        sublap(S, 7, tf);
        if (!D) {
            // the recursive norm's cross terms
            double part = 0.0;
            for (int t = wid; t < m; t += NW) {
                const Cx<float>* ut = cs_u<false>(c, t);
                const Cx<float>* vt = ut + M;
                Cx<float> gu{0, 0}, gv{0, 0};
#pragma unroll 4
                for (int i = lane; i < M; i += 32) cfmac(gu, ldcx(um + i), ldcx(ut + i));  // conj(u_t) u_m
#pragma unroll 4
                for (int i = lane; i < N; i += 32) cfmac(gv, ldcx(vt + i), ldcx(vm + i));  // conj(v_m) v_t
                // lanes 0-15: Re gu, Re gv; lanes 16-31: Im gu, Im gv
                const float2 g = warp_sum4(gu.x, gv.x, gu.y, gv.y);
                part = fma((lane & 16) ? -2.0 * (double)g.x : 2.0 * (double)g.x, (double)g.y, part);
            }
            part += __shfl_xor_sync(0xffffffffu, part, 16);
            if (lane == 0) S.crs[wid] = part;
            __syncthreads();
            if (wid == 0) {
                double add = lane < NW ? S.crs[lane] : 0.0;
                add = warp_sum(add);
                if (lane == 0) {
                    const double own = (double)nu2 * (double)nv2;
                    S.fsn2 += add + own;
                    S.fconv = own <= face_bound2(A, S);
                }
            }
            __syncthreads();
            sublap(S, 8, tf);
        }
        ++m;
        if (D ? face_passes(S.thr, nu2, nv2) : S.fconv != 0) {
            if (!A.sample_check) {
                converged = true;
                break;
            }
            // confirm on the sample entries: partial pivoting can miss a block
            // of the face that no visited row or column reaches
            samples32<KER, NT>(A, S, F, c, kf, m, D);
            static_assert(SAMPLES == 32, "one sample per lane");
            if (wid == 0) {
                const double sv = S.samp[lane];
                const double tot = warp_sum(sv);
                ArgMaxT<float> b{(float)sv, lane};
                b = warp_argmax(b);
                if (lane == 0) {
                    S.fconv = (double)M * (double)N / SAMPLES * tot <= face_bound2(A, S);
                    S.fbs = b.i;
                }
            }
            __syncthreads();
            const bool ok = S.fconv;
            const int bs = S.fbs;
            __syncthreads();  // both are rewritten by the next test
            sublap(S, 9, tf);
            if (ok) {
                converged = true;
                break;
            }
            if (tid == 0) atomicAdd(&A.counters[5], 1ull);
            irow = (2 * bs + 1) * M / (2 * SAMPLES);
            continue;
        }
        if (nx.v < 0.f) break;  // every row used
        irow = nx.i;
    }
    if (tid == 0) S.raw += m;
    if (!converged && m == A.RF && m < min(M, N)) {
        if (tid == 0) {
            atomicOr(A.status, ST_FACE_CAPPED);
            atomicAdd(&A.counters[3], 1ull);
        }
    }
    __syncthreads();
    return m;
}

// ---- recompression ----------------------------------------------------------------------
// The r crosses of c are replaced in place by the factors of a truncated
// H = U V^H (Section 4, second implementation remark), all in float32 and in
// shared memory when the columns and two r x r matrices fit:
//   1. V = Q R by modified Gram-Schmidt (R unit upper triangular, Q's columns
//      orthogonal with norms n_b), one barrier per column.  v_t = conj(row /
//      pivot) vanishes at the earlier pivot columns, so V is well conditioned;
//   2. W = U R^H diag(n), row by row in place: H = W (Q diag(1/n))^H, and W has
//      the column norms of the core R_U R_V^H without a QR of U;
//   3. column-pivoted QR of W by modified Gram-Schmidt, stopped when the
//      largest remaining column norm falls below eps_face times the first one:
//      dropping the remaining columns removes exactly their norms, as a
//      truncated SVD removes its dropped singular values.  One barrier per step:
//      every warp picks the pivot from the column norms (double-buffered) and
//      forms its norm itself.
// U' = W's pivot columns (normalised), V' = Q diag(1/n) J, J = Pi R_W^H.
// Modified Gram-Schmidt keeps A = Q R to rounding whatever the orthogonality
// of Q, so U' V'^H + (the dropped columns) is H to float32 rounding; a Gram
// (Cholesky) QR squares the condition number and needs float64, at 4x the cycles.
// On residual faces of both layers (L-shapes, sphere) the two add the same rounding
// error, 1.2 to 1.4e-7 of the face, at the same ranks.
// RT [r][ldr]: conj(R) transposed; JT [r][ldr].  Returns the kept rank;
// S.sel, S.rk32: pivot columns and their norms.  A face that breaks down (values that
// are not finite, or no column left of a face with crosses) is reported in the status
// and counted: the columns are overwritten by then, so what was found up to there is
// kept.
template <int NT, bool SM>
__device__ int recompress32_t(const AcaArgs<float>& A, BlockSh<float>& S, const ColStore& c, int r, Cx<float>* RT,
                              Cx<float>* JT, int ldr) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int M = S.M, N = S.N;
    long long tc = clock64();
    for (int e = tid; e < r * ldr; e += NT) RT[e] = JT[e] = Cx<float>{0, 0};
    if (wid == 0) {
        const Cx<float>* v = cs_v<SM>(c, 0);
        float s2 = 0;
        for (int i = lane; i < N; i += 32) s2 += cabs2(ldcx(v + i));
        s2 = warp_sum(s2);
        if (lane == 0) S.n2[0] = s2;
    }
    __syncthreads();
    // ---- 1. V = Q R ----
    for (int k = 0; k < r; ++k) {
        const float n2 = S.n2[k];
        const float inv = n2 > 0.f ? 1.f / n2 : 0.f;
        const Cx<float>* vk = cs_v<SM>(c, k);
        if (tid == 0) RT[k * ldr + k] = Cx<float>{1.f, 0.f};
        // two columns per warp and pass
        for (int j = k + 1 + wid; j < r; j += 2 * NW) {
            const bool two = j + NW < r;
            Cx<float>* va = cs_v<SM>(c, j);
            Cx<float>* vb = two ? cs_v<SM>(c, j + NW) : va;
            Cx<float> ga{0, 0}, gb{0, 0};
#pragma unroll 2
            for (int i = lane; i < N; i += 32) {
                const Cx<float> q = ldcx(vk + i);
                cfmac(ga, ldcx(va + i), q);  // conj(v_k) v_j
                cfmac(gb, ldcx(vb + i), q);
            }
            warp_sum_pair(ga, gb);
            ga.x *= inv;
            ga.y *= inv;
            gb.x *= inv;
            gb.y *= inv;
            float s2 = 0;
#pragma unroll 2
            for (int i = lane; i < N; i += 32) {
                const Cx<float> q = ldcx(vk + i);
                Cx<float> x = ldcx(va + i);
                x.x -= q.x * ga.x - q.y * ga.y;
                x.y -= q.x * ga.y + q.y * ga.x;
                va[i] = x;
                s2 += cabs2(x);
                if (two) {
                    Cx<float> y = ldcx(vb + i);
                    y.x -= q.x * gb.x - q.y * gb.y;
                    y.y -= q.x * gb.y + q.y * gb.x;
                    vb[i] = y;
                }
            }
            if (j == k + 1) {  // the next step's column
                s2 = warp_sum(s2);
                if (lane == 0) S.n2[j] = s2;
            }
            if (lane == 0) {
                RT[j * ldr + k] = cconj(ga);
                if (two) RT[(j + NW) * ldr + k] = cconj(gb);
            }
        }
        __syncthreads();
    }
    for (int b = tid; b < r; b += NT) {
        const float n = sqrtf(S.n2[b]);
        S.nv[b] = n;
        S.rnv[b] = n > 0.f ? 1.f / n : 0.f;
    }
    __syncthreads();
    sublap(S, 0, tc);
    // ---- 2. W = U R^H diag(n) in place: W[i][b] = n_b sum_{c >= b} U[i][c] conj(R[b][c]) ----
    {
        // G threads (one warp's neighbours) per row, four columns b each per pass; a
        // pass overwrites columns that no later pass reads
        const int G = M * 4 <= NT ? 4 : (M * 2 <= NT ? 2 : 1);
        const int per = NT / G, part = tid % G;
        for (int base = 0; base < M; base += per) {
            const int i = base + tid / G;
            for (int b0 = 0; b0 < r; b0 += 4 * G) {
                const int b = b0 + 4 * part;
                Cx<float> acc[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] = Cx<float>{0, 0};
                if (i < M && b < r) {
                    for (int cc = b; cc < r; ++cc) {
                        const Cx<float> u = ldcx(cs_u<SM>(c, cc) + i);
                        const float4 r0 = *reinterpret_cast<const float4*>(RT + cc * ldr + b);
                        const float4 r1 = *reinterpret_cast<const float4*>(RT + cc * ldr + b + 2);
                        cfma(acc[0], u, Cx<float>{r0.x, r0.y});
                        cfma(acc[1], u, Cx<float>{r0.z, r0.w});
                        cfma(acc[2], u, Cx<float>{r1.x, r1.y});
                        cfma(acc[3], u, Cx<float>{r1.z, r1.w});
                    }
                }
                __syncwarp();
                if (i < M) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (b + q < r) {
                            const float n = S.nv[b + q];
                            cs_u<SM>(c, b + q)[i] = Cx<float>{acc[q].x * n, acc[q].y * n};
                        }
                }
                __syncwarp();
            }
        }
    }
    __syncthreads();
    sublap(S, 1, tc);
    // ---- 3. column-pivoted QR of W ----
    for (int j = wid; j < r; j += NW) {
        const Cx<float>* x = cs_u<SM>(c, j);
        float s2 = 0;
        for (int i = lane; i < M; i += 32) s2 += cabs2(ldcx(x + i));
        s2 = warp_sum(s2);
        if (lane == 0) S.cn[0][j] = s2;
    }
    __syncthreads();
    const float sfloor = (float)A.trunc_floor * S.rms;
    float r00 = 0.f;
    int k = 0;
    for (; k < r; ++k) {
        const float* cn = S.cn[k & 1];
        float* cx = S.cn[(k & 1) ^ 1];
        ArgMaxT<float> best = amax_none<float>();
        for (int q = lane; q < r; q += 32) best = amax_better(best, ArgMaxT<float>{cn[q], q});
        const uint2 key = warp_key(best);
        if (key.x == 0u) break;
        const int pv = (int)key.y;
        const Cx<float>* qv = cs_u<SM>(c, pv);
        float s2 = 0;
        for (int i = lane; i < M; i += 32) s2 += cabs2(ldcx(qv + i));
        s2 = warp_sum(s2);
        const float rkk = sqrtf(s2);
        if (k == 0) r00 = rkk;
        if (!(rkk > 0.f) || !isfinite(rkk) || rkk < (float)A.eps_face * r00 || (k > 0 && rkk < sfloor)) break;
        const float inv = 1.f / rkk;
        if (tid == 0) {
            S.sel[k] = pv;
            S.rk32[k] = rkk;
            JT[pv * ldr + k] = Cx<float>{rkk, 0.f};
        }
        for (int j = wid; j < r; j += 2 * NW) {
            const int j2 = j + NW;
            const float c1 = cn[j], c2 = j2 < r ? cn[j2] : -1.f;
            const bool o1 = c1 >= 0.f && j != pv, o2 = c2 >= 0.f && j2 != pv;
            Cx<float>* xa = cs_u<SM>(c, j);
            Cx<float>* xb = o2 ? cs_u<SM>(c, j2) : xa;
            Cx<float> ga{0, 0}, gb{0, 0};
            if (o1 || o2) {
#pragma unroll 2
                for (int i = lane; i < M; i += 32) {
                    const Cx<float> q = ldcx(qv + i);
                    cfmac(ga, ldcx(xa + i), q);
                    cfmac(gb, ldcx(xb + i), q);
                }
                warp_sum_pair(ga, gb);
                ga.x *= inv;
                ga.y *= inv;
                gb.x *= inv;
                gb.y *= inv;
#pragma unroll 2
                for (int i = lane; i < M; i += 32) {
                    Cx<float> q = ldcx(qv + i);
                    q.x *= inv;
                    q.y *= inv;
                    if (o1) {
                        Cx<float> x = ldcx(xa + i);
                        x.x -= q.x * ga.x - q.y * ga.y;
                        x.y -= q.x * ga.y + q.y * ga.x;
                        xa[i] = x;
                    }
                    if (o2) {
                        Cx<float> y = ldcx(xb + i);
                        y.x -= q.x * gb.x - q.y * gb.y;
                        y.y -= q.x * gb.y + q.y * gb.x;
                        xb[i] = y;
                    }
                }
            }
            if (lane == 0) {
                cx[j] = o1 ? fmaxf(c1 - cabs2(ga), 0.f) : -1.f;
                if (o1) JT[j * ldr + k] = cconj(ga);
                if (j2 < r) {
                    cx[j2] = o2 ? fmaxf(c2 - cabs2(gb), 0.f) : -1.f;
                    if (o2) JT[j2 * ldr + k] = cconj(gb);
                }
            }
        }
        __syncthreads();
    }
    __syncthreads();
    if (wid == 0) {
        const float* cn = S.cn[k & 1];
        bool bad = k == 0;
        for (int q = lane; q < r; q += 32) bad |= !isfinite(cn[q]);
        if (__any_sync(0xffffffffu, bad) && lane == 0) {
            atomicOr(A.status, ST_CHOL_FALLBACK);
            atomicAdd(&A.counters[4], 1ull);
        }
    }
    sublap(S, 3, tc);
    // fold Q's normalisation into J
    for (int e = tid; e < r * ldr; e += NT) {
        const float n = S.rnv[e / ldr];
        JT[e].x *= n;
        JT[e].y *= n;
    }
    __syncthreads();
    return k;
}

// U' and V' of the recompressed face into the pool (M x rn, N x rn, column-major)
template <int NT, bool SM>
__device__ void form32_t(BlockSh<float>& S, const ColStore& c, int r, int rn, const Cx<float>* JT, int ldr,
                         Cx<float>* Un, Cx<float>* Vn) {
    const int tid = threadIdx.x;
    const int M = S.M, N = S.N;
    for (int e = tid; e < rn * M; e += NT) {
        const int b = e / M, i = e - b * M;
        const float inv = 1.f / S.rk32[b];
        const Cx<float> x = ldcx(cs_u<SM>(c, S.sel[b]) + i);
        Un[e] = Cx<float>{x.x * inv, x.y * inv};
    }
    const int nb = (rn + 3) / 4;
    for (int e = tid; e < N * nb; e += NT) {
        const int b = (e / N) * 4, j = e % N;
        Cx<float> acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = Cx<float>{0, 0};
#pragma unroll 2
        for (int a = 0; a < r; ++a) {
            const Cx<float> v = ldcx(cs_v<SM>(c, a) + j);
            const float4 r0 = *reinterpret_cast<const float4*>(JT + a * ldr + b);
            const float4 r1 = *reinterpret_cast<const float4*>(JT + a * ldr + b + 2);
            cfma(acc[0], v, Cx<float>{r0.x, r0.y});
            cfma(acc[1], v, Cx<float>{r0.z, r0.w});
            cfma(acc[2], v, Cx<float>{r1.x, r1.y});
            cfma(acc[3], v, Cx<float>{r1.z, r1.w});
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (b + q < rn) Vn[(long long)(b + q) * N + j] = acc[q];
    }
}

// where the recompression's two r x r matrices go, and whether everything is
// in shared memory
struct Recomp32 {
    Cx<float>* RT;
    Cx<float>* JT;
    int ldr;
    bool sm;
};
__device__ __forceinline__ Recomp32 recomp32_place(const AcaArgs<float>& A, const Ws<float>& w, const ColStore& c, int r,
                                                   unsigned char* arena) {
    Recomp32 p;
    p.ldr = (r + 3) & ~3;
    const size_t one = (size_t)r * p.ldr;
    unsigned char* end = reinterpret_cast<unsigned char*>(c.sm + (size_t)r * c.ld);
    p.sm = r <= c.ncs && (size_t)(end - arena) + 2 * one * sizeof(Cx<float>) <= (size_t)A.arena_bytes;
    p.RT = p.sm ? reinterpret_cast<Cx<float>*>(end) : reinterpret_cast<Cx<float>*>(w.RU);
    p.JT = p.sm ? p.RT + one : reinterpret_cast<Cx<float>*>(w.RV);
    return p;
}
template <int NT>
__device__ int recompress32(const AcaArgs<float>& A, BlockSh<float>& S, const ColStore& c, int r, const Recomp32& p,
                            unsigned char* arena) {
    // (addresses formed from the arena, so that they stay shared-memory accesses)
    if (p.sm) {
        Cx<float>* RT = reinterpret_cast<Cx<float>*>(arena + (reinterpret_cast<unsigned char*>(p.RT) - arena));
        return recompress32_t<NT, true>(A, S, c, r, RT, RT + (size_t)r * p.ldr, p.ldr);
    }
    return recompress32_t<NT, false>(A, S, c, r, p.RT, p.JT, p.ldr);
}
template <int NT>
__device__ void form32(BlockSh<float>& S, const ColStore& c, int r, int rn, bool raw, const Recomp32& p, Cx<float>* Un,
                       Cx<float>* Vn) {
    if (raw) {
        const int M = S.M, N = S.N;
        for (int e = threadIdx.x; e < rn * M; e += NT) Un[e] = cs_u<false>(c, e / M)[e % M];
        for (int e = threadIdx.x; e < rn * N; e += NT) Vn[e] = cs_v<false>(c, e / N)[e % N];
    } else if (p.sm) {
        form32_t<NT, true>(S, c, r, rn, p.JT, p.ldr, Un, Vn);
    } else {
        form32_t<NT, false>(S, c, r, rn, p.JT, p.ldr, Un, Vn);
    }
}

// ---- float-float helpers of the fiber ------------------------------------------------------
// a complex number as two float-float values
struct Cff {
    float2 x, y;
};
// a - h f for float32 h, f: the products exact, the sum to ~2^-48
__device__ __forceinline__ void cff_sub_prod(Cff& a, Cx<float> h, Cx<float> f) {
    ff_add_prod(a.x, -h.x, f.x);
    ff_add_prod(a.x, h.y, f.y);
    ff_add_prod(a.y, -h.x, f.y);
    ff_add_prod(a.y, -h.y, f.x);
}

// 1 / h to ~2^-46: one Newton step in float-float from the float32 reciprocal of
// |h|^2, h scaled to magnitude ~1 by a power of two
__device__ __forceinline__ Cff cff_inv(Cx<float> h) {
    const int e = min(max(ilogbf(fmaxf(fabsf(h.x), fabsf(h.y))), -120), 120);
    const float sc = scalbnf(1.f, -e);
    const float x = h.x * sc, y = h.y * sc;
    float2 n = make_float2(0.f, 0.f);
    ff_add_prod(n, x, x);
    ff_add_prod(n, y, y);
    const float r0 = 1.f / n.x;
    // r = r0 + r0 (1 - n r0)
    float2 d = ff_neg(ff_mul(n, make_float2(r0, 0.f)));
    ff_add(d, 1.f, 0.f);
    float2 r = make_float2(r0, 0.f);
    const float2 c = ff_mul(d, make_float2(r0, 0.f));
    ff_add(r, c.x, c.y);
    const float2 rx = ff_mul(r, make_float2(x, 0.f)), ry = ff_mul(r, make_float2(-y, 0.f));
    return Cff{make_float2(rx.x * sc, rx.y * sc), make_float2(ry.x * sc, ry.y * sc)};
}

// The fiber of the new cross at the pivot (elements gi, gj), float32 blocks:
//   f[k] = (ENTRY(gi, gj, k) - sum_p H_p f_p[k]) / H_l   (H at the pivot).
// The residual is formed in float-float (its operands are float32, so every
// product is exact and the sum good to ~2^-48; the same values in float64 cost
// 19 SM cycles per warp instruction on this part's float64 pipe, which bound
// the blocks with dense faces).  G threads share a frequency: its quadrature
// points and its crosses.  hp[p] = H_p at the pivot, inv = 1 / H_l, fptr(p): the
// fiber of cross p; tid of NT threads (whole warps).
template <int KER, int NT, class FP>
__device__ __forceinline__ void fiber32(const AcaArgs<float>& A, int tid, int gi, int gj, int nc, const Cx<float>* hp,
                                        const Cff inv, FP fptr, Cx<float>* Fn) {
    const int Ku = A.Ku;
    // the gang of 1, 2 or 4 with the fewest passes per frequency
    int G = 1, best = 4 * ((Ku + NT - 1) / NT);
#pragma unroll
    for (int g = 2; g <= 4; g *= 2) {
        const int c = (4 / g) * ((Ku * g + NT - 1) / NT);
        if (c < best) {
            best = c;
            G = g;
        }
    }
    const int part = tid % G;
    for (int k0 = 0; k0 < Ku; k0 += NT / G) {
        const int k = k0 + tid / G;
        Cff e{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (k < Ku) {
            const Cx<float> a = ent_part<KER, float>(A, gi, gj, k, part, G);
            e.x.x = a.x;
            e.y.x = a.y;
#pragma unroll 2
            for (int p = part; p < nc; p += G) cff_sub_prod(e, hp[p], ldcx(fptr(p) + k));
        }
        for (int o = G >> 1; o > 0; o >>= 1) {
            const float xh = __shfl_xor_sync(0xffffffffu, e.x.x, o), xl = __shfl_xor_sync(0xffffffffu, e.x.y, o);
            const float yh = __shfl_xor_sync(0xffffffffu, e.y.x, o), yl = __shfl_xor_sync(0xffffffffu, e.y.y, o);
            ff_add(e.x, xh, xl);
            ff_add(e.y, yh, yl);
        }
        if (k < Ku && part == 0) {
            float2 re = ff_mul(e.x, inv.x), im = ff_mul(e.x, inv.y);
            const float2 a = ff_neg(ff_mul(e.y, inv.y)), b = ff_mul(e.y, inv.x);
            ff_add(re, a.x, a.y);
            ff_add(im, b.x, b.y);
            Fn[k] = Cx<float>{re.x + re.y, im.x + im.y};
        }
    }
}

// ---- the new cross's factors in shared memory --------------------------------------------
// U' and V' (just written to the pool) staged once for the pivot search and
// eq. (norm): column b at su + b ldu (ldu is 8 modulo 16 and at least M + 8, zero
// beyond M; sv likewise), when the arena holds them.
struct NewFac {
    Cx<float>* su;
    Cx<float>* sv;
    int ldu, ldv;
    bool sm;
};
template <int NT>
__device__ __forceinline__ NewFac stage_new(const AcaArgs<float>& A, const BlockSh<float>& S, const Cx<float>* Un,
                                            const Cx<float>* Vn, int rn, unsigned char* arena) {
    NewFac f;
    f.ldu = ((S.M + 15) & ~15) + 8;
    f.ldv = ((S.N + 15) & ~15) + 8;
    f.su = reinterpret_cast<Cx<float>*>(arena);
    f.sv = f.su + (size_t)rn * f.ldu;
    f.sm = (size_t)rn * (f.ldu + f.ldv) * sizeof(Cx<float>) <= (size_t)A.arena_bytes;
    if (f.sm) {
        // one warp per column, all of its loads in flight together
        const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int b = wid; b < 2 * rn; b += NT / 32) {
            const bool u = b < rn;
            const int L = u ? S.M : S.N, ld = u ? f.ldu : f.ldv;
            const Cx<float>* src = u ? Un + (long long)b * S.M : Vn + (long long)(b - rn) * S.N;
            Cx<float>* dst = u ? f.su + b * f.ldu : f.sv + (b - rn) * f.ldv;
#pragma unroll 8
            for (int i = lane; i < ld; i += 32) dst[i] = i < L ? ldcx(src + i) : Cx<float>{0, 0};
        }
    }
    return f;
}

// largest |U' V'^H| entry of a thread's 4 x 4 tiles (staged factors)
template <int NT>
__device__ __forceinline__ ArgMaxT<float> pivot32(const BlockSh<float>& S, const NewFac& f, int rn) {
    ArgMaxT<float> best = amax_none<float>();
    const int M = S.M, N = S.N, tx = (N + 3) / 4, nt = ((M + 3) / 4) * tx;
    for (int q = threadIdx.x; q < nt; q += NT) {
        const int ti = (q / tx) * 4, tj = (q % tx) * 4;
        Cx<float> acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][c] = Cx<float>{0, 0};
        const Cx<float>* pu = f.su + ti;
        const Cx<float>* pv = f.sv + tj;
        for (int b = 0; b < rn; ++b, pu += f.ldu, pv += f.ldv) {
            const float4 u0 = *reinterpret_cast<const float4*>(pu), u1 = *reinterpret_cast<const float4*>(pu + 2);
            const float4 v0 = *reinterpret_cast<const float4*>(pv), v1 = *reinterpret_cast<const float4*>(pv + 2);
            const Cx<float> uu[4] = {{u0.x, u0.y}, {u0.z, u0.w}, {u1.x, u1.y}, {u1.z, u1.w}};
            const Cx<float> vv[4] = {{v0.x, v0.y}, {v0.z, v0.w}, {v1.x, v1.y}, {v1.z, v1.w}};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 4; ++c) cfmac(acc[a][c], uu[a], vv[c]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (ti + a < M && tj + c < N)
                    best = amax_better(best, ArgMaxT<float>{cabs2(acc[a][c]), (ti + a) * N + tj + c});
    }
    return best;
}

// ---- eq. (norm) inner products, float32 ----------------------------------------------------
// hh[d] = <H_l, H_d>_F = sum_{a in cross d, b} (U_d^H U_l)[a][b] conj((V_d^H V_l)[a][b]),
// hself = ||H_l||_F^2 (a over the columns of cross l), as norm_grams, on the
// tensor cores (the three-term TF32 split): a warp takes 16 columns a of
// [U_1 .. U_nc U_l] against 16 columns b of U_l at a time, streams its columns
// from L2 straight into the A fragments (32-byte sectors, four k-steps of loads
// in flight) and reads U_l from the staged copy; no barrier until the sums per
// column are complete (the tiled version staged every column and synchronised
// four times per 64 rows).  The k slots of a step are the rows i0 + 2t and
// i0 + 2t + 1 of lane group t, so that both operands load 16 adjacent bytes.
// Sums per column in float32, over crosses in float64.  colv: a value per column.
template <int NT, bool SM>
__device__ void norm32_t(const AcaArgs<float>& A, BlockSh<float>& S, const Cx<float>* Un, const Cx<float>* Vn, int rn,
                         const NewFac& f, Cx<float>* colv) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int M = S.M, N = S.N, nc = S.ncross;
    const int n0 = S.pre[nc], na = n0 + rn;
    for (int a0 = wid * 16; a0 < na; a0 += NW * 16) {
        // the lane's two columns (g, g + 8): U then V; absent ones repeat the last
        const Cx<float>* pu[2];
        const Cx<float>* pv[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int a = min(a0 + g + 8 * h, na - 1);
            if (a < n0) {
                int lo = 0, hi = nc - 1;   // the cross d with pre[d] <= a < pre[d + 1]
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (S.pre[mid] <= a) lo = mid;
                    else hi = mid - 1;
                }
                const int tt = a - S.pre[lo];
                pu[h] = A.pool + S.off[lo] + (long long)tt * M;
                pv[h] = A.pool + S.off[lo] + (long long)S.r[lo] * M + (long long)tt * N;
            } else {
                pu[h] = Un + (long long)(a - n0) * M;
                pv[h] = Vn + (long long)(a - n0) * N;
            }
        }
        float sx[2] = {0, 0}, sy[2] = {0, 0};   // the two columns' sums over b (this lane's b)
        for (int b0 = 0; b0 < rn; b0 += 16) {
            float z[2][2][2][4];   // [U, V][b tile][re, im][fragment]
#pragma unroll
            for (int side = 0; side < 2; ++side) {
#pragma unroll
                for (int bt = 0; bt < 2; ++bt)
#pragma unroll
                    for (int q = 0; q < 4; ++q) z[side][bt][0][q] = z[side][bt][1][q] = 0.f;
                const int L = side == 0 ? M : N;
                const int ldb = side == 0 ? f.ldu : f.ldv;
                const Cx<float>* bs = side == 0 ? f.su : f.sv;
                const Cx<float>* bg = side == 0 ? Un : Vn;
                const Cx<float>* c0 = side == 0 ? pu[0] : pv[0];
                const Cx<float>* c1 = side == 0 ? pu[1] : pv[1];
                const bool two = b0 + 8 < rn;
                for (int i0 = 0; i0 < L; i0 += 32) {
                    Cx<float> x[4][4];   // [k-step][(g, 2t), (g + 8, 2t), (g, 2t + 1), (g + 8, 2t + 1)]
#pragma unroll
                    for (int st = 0; st < 4; ++st) {
                        const int i = i0 + 8 * st + 2 * t;
                        x[st][0] = i < L ? ldcx(c0 + i) : Cx<float>{0, 0};
                        x[st][1] = i < L ? ldcx(c1 + i) : Cx<float>{0, 0};
                        x[st][2] = i + 1 < L ? ldcx(c0 + i + 1) : Cx<float>{0, 0};
                        x[st][3] = i + 1 < L ? ldcx(c1 + i + 1) : Cx<float>{0, 0};
                    }
#pragma unroll
                    for (int st = 0; st < 4; ++st) {
                        if (i0 + 8 * st >= L) break;
                        const int i = i0 + 8 * st + 2 * t;
                        unsigned arh[4], arl[4], aih[4], ail[4], nih[4], nil[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const Tf32Pair r = tf32_split(x[st][q].x), m = tf32_split(x[st][q].y);
                            arh[q] = r.hi;
                            arl[q] = r.lo;
                            aih[q] = m.hi;
                            ail[q] = m.lo;
                        }
                        tf32_neg4(aih, nih);
                        tf32_neg4(ail, nil);
#pragma unroll
                        for (int bt = 0; bt < 2; ++bt) {
                            if (bt == 1 && !two) break;
                            const int b = b0 + 8 * bt + g;
                            Cx<float> y[2] = {{0, 0}, {0, 0}};
                            if (b < rn) {
                                if constexpr (SM) {
                                    const float4 v = *reinterpret_cast<const float4*>(bs + b * ldb + i);
                                    y[0] = Cx<float>{v.x, v.y};
                                    y[1] = Cx<float>{v.z, v.w};
                                } else {
                                    const Cx<float>* p = bg + (long long)b * L + i;
                                    if (i < L) y[0] = ldcx(p);
                                    if (i + 1 < L) y[1] = ldcx(p + 1);
                                }
                            }
                            unsigned brh[2], brl[2], bih[2], bil[2];
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const Tf32Pair r = tf32_split(y[q].x), m = tf32_split(y[q].y);
                                brh[q] = r.hi;
                                brl[q] = r.lo;
                                bih[q] = m.hi;
                                bil[q] = m.lo;
                            }
                            float* re = z[side][bt][0];
                            float* im = z[side][bt][1];
                            // conj(a) b: Re = ar br + ai bi, Im = ar bi - ai br
                            mma_tf32(re, arh, brl);
                            mma_tf32(im, arh, bil);
                            mma_tf32(re, arl, brh);
                            mma_tf32(im, arl, bih);
                            mma_tf32(re, aih, bil);
                            mma_tf32(im, nih, brl);
                            mma_tf32(re, ail, bih);
                            mma_tf32(im, nil, brh);
                            mma_tf32(re, arh, brh);
                            mma_tf32(im, arh, bih);
                            mma_tf32(re, aih, bih);
                            mma_tf32(im, nih, brh);
                        }
                    }
                }
            }
            // zu conj(zv) summed over the lane's columns b (absent ones are zero)
#pragma unroll
            for (int bt = 0; bt < 2; ++bt)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float ux = z[0][bt][0][q], uy = z[0][bt][1][q], vx = z[1][bt][0][q], vy = z[1][bt][1][q];
                    sx[q >> 1] += ux * vx + uy * vy;
                    sy[q >> 1] += uy * vx - ux * vy;
                }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                sx[h] += __shfl_xor_sync(0xffffffffu, sx[h], o);
                sy[h] += __shfl_xor_sync(0xffffffffu, sy[h], o);
            }
            const int a = a0 + g + 8 * h;
            if (t == 0 && a < na) colv[a] = Cx<float>{sx[h], sy[h]};
        }
    }
    __syncthreads();
    for (int d = wid; d <= nc; d += NW) {
        const int lo = S.pre[d], hi = d < nc ? S.pre[d + 1] : na;
        float x = 0, y = 0;
        for (int a = lo + lane; a < hi; a += 32) {
            const Cx<float> v = colv[a];
            x += v.x;
            y += v.y;
        }
        x = warp_sum(x);
        y = warp_sum(y);
        if (lane == 0) {
            if (d < nc) S.hh[d] = Cx<double>{(double)x, (double)y};
            else S.hself = (double)x;
        }
    }
    __syncthreads();
}

}  // namespace g3
