// Application of the compressed three-way array to densities at all
// frequencies (eq. (product)):
//
//   y = sum_{l=1}^{K} A(s_l) w_l
//     = sum_near sum_k [Re A_k (w_k + w_k') + i Im A_k (w_k - w_k')]
//       + sum_far sum_p [ U_p (V_p^H x_p) + conj(U_p (V_p^H zc_p)) ],
//   x_p = sum_{k in unique} f_p[k] w_k ,  zc_p = sum_{k paired} f_p[k] conj(w_k'),
//
// where k' is the conjugate partner of the unique frequency k
// (A(conj s) = conj A(s) for real geometry; Appendix A notes that half of the
// frequencies suffice).  Both sums need w only in the combinations
//   w^+_k = w_k + conj(w_k'),  w^-_k = w_k - conj(w_k')
// (w_k' = 0 without a partner), which k_apply_prep forms once: with x^+- =
// sum_k f_p[k] w^+-_k and a^+- = V^H x^+-, the terms U a + conj(U b) of a cross are
//   Re = Re U Re a^+ - Im U Im a^+,  Im = Re U Im a^- + Im U Re a^-,
// half the multiply-adds of the two products.  The near field is read once from HBM (the bound of
// this step); each stored (unique-frequency) entry serves both members of a
// conjugate pair.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "g3_device.cuh"

#define G3_TRY_NA(expr)                 \
    do {                                \
        g3_status st_ = (expr);         \
        if (st_ != G3_OK) return st_;   \
    } while (0)

namespace g3 {

// largest face rank the per-frequency apply keeps in shared memory (the
// compression caps face ranks at 64)
constexpr int RF_TS = 64;

// W (original order, column l = w_l, M x K column-major, complex TI) ->
// Wf[k][p] = w_{uniq[k]}[perm[p]],  Wc[k][p] = w_{partner(uniq[k])}[perm[p]] or 0
// (cluster order, frequency-major), and y := 0.
// ldw: rows of W (E, or the vertex count for linear-element trees, where perm is
// the vertex of each position: the gather w_loc = P w of the nodal densities)
template <class TI, class T>
__global__ void k_apply_prep(int E, int K, int Ku, const int* __restrict__ perm, const int* __restrict__ uniq,
                             const int* __restrict__ partner, const Cx<TI>* __restrict__ W, Cx<T>* __restrict__ Wf,
                             Cx<T>* __restrict__ Wc, Cx<T>* __restrict__ y, int ldw) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx < E) y[idx] = Cx<T>{0, 0};
    if (idx >= (long long)Ku * E) return;
    const int k = (int)(idx / E), p = (int)(idx % E);
    const int e = perm[p];
    const int l = uniq[k], lp = partner[l];
    Cx<TI> a = W[(long long)l * ldw + e];
    Wf[idx] = Cx<T>{(T)a.x, (T)a.y};
    if (lp != l) {
        Cx<TI> b = W[(long long)lp * ldw + e];
        Wc[idx] = Cx<T>{(T)b.x, (T)b.y};
    } else {
        Wc[idx] = Cx<T>{0, 0};
    }
}

// W -> (w^+, w^-)[k][p] for the sum over the frequencies (the gather as above), y := 0
template <class T>
struct alignas(4 * sizeof(T)) WPair {
    T px, py, mx, my;   // w + conj(w'), w - conj(w')
};
template <class TI, class T>
__global__ void k_apply_prep_pm(int E, int Ku, const int* __restrict__ perm, const int* __restrict__ uniq,
                                const int* __restrict__ partner, const Cx<TI>* __restrict__ W, WPair<T>* __restrict__ Wp,
                                Cx<T>* __restrict__ y, int ldw) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (p >= E) return;
    if (k == 0) y[p] = Cx<T>{0, 0};
    const int e = perm[p], l = uniq[k], lp = partner[l];
    const Cx<TI> a = W[(long long)l * ldw + e];
    Cx<TI> b{0, 0};
    if (lp != l) b = W[(long long)lp * ldw + e];
    const Cx<T> f{(T)a.x, (T)a.y}, c{(T)b.x, (T)b.y};
    Wp[(long long)k * E + p] = WPair<T>{f.x + c.x, f.y - c.y, f.x - c.x, f.y + c.y};
}
template <class T>
__device__ __forceinline__ WPair<T> ldw(const WPair<T>* p) {
    if constexpr (sizeof(T) == 4) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        return {v.x, v.y, v.z, v.w};
    } else {
        const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
        return {a.x, a.y, b.x, b.y};
    }
}

// Near field: one CTA of four warps per (row cluster, frequency chunk).  The work
// units are the (near block, frequency) pairs of the row cluster and chunk, dealt to
// the warps in turn.  A unit's entries are one contiguous slab (blocks are stored
// [k][j][i]); each warp streams its slabs, in pieces of whole columns, through its
// own ring of NEAR_ST stages in shared memory by 16-byte cp.async (with the pieces of
// w and w' beside them), NEAR_ST - 1 pieces ahead, and needs no other warp until the
// end.  Lane i holds row i and sums Re A (w + w') + i Im A (w - w') over the piece's
// columns; the CTA adds the warps' sums to y once.
// Bound by HBM.  Loading into registers kept 45 KB per SM in flight (eight columns of
// 192 bytes in 29 warps) and spent 48 % of the issue slots on addresses and on w read
// per column from L2; the rings keep 74 KB per SM in flight whatever the
// registers; two stages beat three and four (below): HBM serves fewer, longer runs
// better.  12,288-triangle double layer, 4.02 GB: 0.85 -> 0.61 ms (6.6 TB/s); four and
// three stages 1.05 and 0.81 ms, an L2 prefetch three slabs ahead of register loads
// 1.13 ms, 2, 6 and 8 warps 0.68, 0.65 and 0.9 to 1.7 ms.
constexpr int NEAR_NW = 4;            // warps per CTA
constexpr int NEAR_ST = 2;            // stages per warp
constexpr int NEAR_A = 4608 + 16;     // bytes of entries per stage (24 x 24 complex64, and the alignment shift)
constexpr int NEAR_JN = 32;           // most columns per piece
template <class T>
constexpr int near_stage_bytes() { return NEAR_A + NEAR_JN * (int)sizeof(WPair<T>); }

template <class T>
__global__ void __launch_bounds__(NEAR_NW * 32) k_apply_near(const Cx<T>* __restrict__ A,
                                                             const BlockRange* __restrict__ ranges,
                                                             const long long* __restrict__ offs,
                                                             const int* __restrict__ row_start, int Ku, int kchunk, int E,
                                                             const WPair<T>* __restrict__ Wp, Cx<T>* __restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NW = NEAR_NW, ES = (int)sizeof(Cx<T>), SB = near_stage_bytes<T>();
    const int g = blockIdx.x;
    const int k0 = blockIdx.y * kchunk, nk = min(Ku, k0 + kchunk) - k0;
    const int b0 = row_start[g], units = (row_start[g + 1] - b0) * nk;
    const int rb = ranges[b0].rb, M = ranges[b0].re - ranges[b0].rb;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* ring = smem_raw + warp * NEAR_ST * SB;
    T* ys = reinterpret_cast<T*>(smem_raw + NW * NEAR_ST * SB);  // [NW][2 M]
    T* ysw = ys + (size_t)warp * 2 * M;
    for (int i = lane; i < 2 * M; i += 32) ysw[i] = 0;
    __syncwarp();
    const int JN = min(NEAR_JN, (NEAR_A - 16) / (M * ES));  // columns per piece (>= 1, checked on the host)
    // next piece to stage: unit, first column, stage
    int iu = warp, ij = 0, is = 0;
    auto issue = [&]() {
        if (iu < units) {
            const int b = b0 + iu / nk, k = k0 + iu % nk;
            const BlockRange br = ranges[b];
            const int N = br.ce - br.cb, jn = min(JN, N - ij);
            const long long e0 = offs[b] + (long long)k * M * N + (long long)ij * M;
            unsigned char* st = ring + is * SB;
            // 16-byte units from the (rounded-down) first element; the last one may hold
            // a single value
            const int sh = ES == 8 ? (int)(e0 & 1) : 0, n = jn * M + sh;
            const Cx<T>* src = A + (e0 - sh);
            constexpr int EU = 16 / ES;
            for (int c = lane; c * EU < n; c += 32) cp_async16(st + c * 16, src + c * EU, min(16, (n - c * EU) * ES));
            unsigned char* sw = st + NEAR_A;
            if (lane < jn) {
                constexpr int WB = (int)sizeof(WPair<T>);
                const WPair<T>* w = Wp + (long long)k * E + br.cb + ij + lane;
                cp_async16(sw + lane * WB, w, 16);
                if constexpr (WB == 32) cp_async16(sw + lane * WB + 16, reinterpret_cast<const char*>(w) + 16, 16);
            }
            ij += jn;
            if (ij >= N) {
                ij = 0;
                iu += NW;
            }
            is = is + 1 == NEAR_ST ? 0 : is + 1;
        }
        cp_async_commit();   // (an empty group past the end keeps the count)
    };
#pragma unroll
    for (int q = 0; q < NEAR_ST - 1; ++q) issue();
    T sx = 0, sy = 0;   // the lane's row sums (clusters of at most 32 rows)
    int stg = 0;
    for (int u = warp; u < units; u += NW) {
        const int b = b0 + u / nk, k = k0 + u % nk;
        const BlockRange br = ranges[b];
        const int N = br.ce - br.cb;
        const long long ub = offs[b] + (long long)k * M * N;
        for (int j0 = 0; j0 < N; j0 += JN) {
            const int jn = min(JN, N - j0);
            cp_async_wait<NEAR_ST - 2>();
            __syncwarp();   // the piece has landed for every lane, the last one is consumed
            issue();
            const unsigned char* st = ring + stg * SB;
            stg = stg + 1 == NEAR_ST ? 0 : stg + 1;
            const Cx<T>* a0 = reinterpret_cast<const Cx<T>*>(st) + (ES == 8 ? (int)((ub + (long long)j0 * M) & 1) : 0);
            const WPair<T>* w = reinterpret_cast<const WPair<T>*>(st + NEAR_A);
            for (int i0 = 0; i0 < M; i0 += 32) {
                const int i = i0 + lane;
                if (i >= M) break;
                T ax = 0, ay = 0;
#pragma unroll 8
                for (int j = 0; j < jn; ++j) {
                    const Cx<T> a = ldcx(a0 + j * M + i);
                    const WPair<T> v = ldw(w + j);
                    ax += a.x * v.px - a.y * v.py;
                    ay += a.x * v.my + a.y * v.mx;
                }
                if (M <= 32) {
                    sx += ax;
                    sy += ay;
                } else {
                    ysw[2 * i] += ax;
                    ysw[2 * i + 1] += ay;
                }
            }
        }
    }
    if (M <= 32 && lane < M) {
        ysw[2 * lane] = sx;
        ysw[2 * lane + 1] = sy;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < M; i += NW * 32) {
        T tx = 0, ty = 0;
        for (int w = 0; w < NW; ++w) {
            tx += ys[(size_t)w * 2 * M + 2 * i];
            ty += ys[(size_t)w * 2 * M + 2 * i + 1];
        }
        atomicAdd(&y[rb + i].x, tx);
        atomicAdd(&y[rb + i].y, ty);
    }
}

// Near field of row clusters whose columns do not fit a stage of k_apply_near (more
// than 288 rows in float64, 576 in float32): one CTA per (row cluster, frequency chunk).  The work units are
// the (near block, frequency) pairs of the row cluster and chunk, dealt to the
// warps in turn.  For a unit, lane i holds row i of the block (blocks are
// stored [k][j][i], so the column j of all rows is one coalesced load) and
// sums Re A (w + w') + i Im A (w - w') over the block's columns, with w_j and
// w'_j read as broadcasts.  Each warp keeps its row sums in its own slice of
// shared memory; the CTA adds the warps' sums to y once.
template <class T, int NT>
__global__ void __launch_bounds__(NT) k_apply_near_wide(const Cx<T>* __restrict__ A, const BlockRange* __restrict__ ranges,
                                                   const long long* __restrict__ offs, const int* __restrict__ row_start,
                                                   int Ku, int kchunk, int E, const WPair<T>* __restrict__ Wp,
                                                   Cx<T>* __restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NW = NT / 32;
    const int g = blockIdx.x;
    const int k0 = blockIdx.y * kchunk, k1 = min(Ku, k0 + kchunk), nk = k1 - k0;
    const int b0 = row_start[g], b1 = row_start[g + 1];
    const int rb = ranges[b0].rb, Mrow = ranges[b0].re - ranges[b0].rb;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T* ysw = reinterpret_cast<T*>(smem_raw) + (size_t)warp * 2 * Mrow;  // [NW][2 * Mrow]
    for (int i = threadIdx.x; i < NW * 2 * Mrow; i += NT) reinterpret_cast<T*>(smem_raw)[i] = 0;
    __syncthreads();
    const int units = (b1 - b0) * nk;
    for (int u = warp; u < units; u += NW) {
        const int b = b0 + u / nk, k = k0 + u % nk;
        const BlockRange br = ranges[b];
        const int N = br.ce - br.cb;
        const Cx<T>* Ak = A + offs[b] + (long long)k * Mrow * N;
        const WPair<T>* wp = Wp + (long long)k * E + br.cb;
        for (int i0 = 0; i0 < Mrow; i0 += 32) {
            const int i = i0 + lane;
            const bool act = i < Mrow;
            T ax = 0, ay = 0;
            int j = 0;
            for (; j + 8 <= N; j += 8) {
                Cx<T> a[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) a[q] = act ? ldcx(Ak + (long long)(j + q) * Mrow + i) : Cx<T>{0, 0};
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const WPair<T> v = ldw(wp + j + q);
                    ax += a[q].x * v.px - a[q].y * v.py;
                    ay += a[q].x * v.my + a[q].y * v.mx;
                }
            }
            for (; j < N; ++j) {
                const Cx<T> a = act ? ldcx(Ak + (long long)j * Mrow + i) : Cx<T>{0, 0};
                const WPair<T> v = ldw(wp + j);
                ax += a.x * v.px - a.y * v.py;
                ay += a.x * v.my + a.y * v.mx;
            }
            if (act) {
                ysw[2 * i] += ax;
                ysw[2 * i + 1] += ay;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < Mrow; i += NT) {
        T sx = 0, sy = 0;
        for (int w = 0; w < NW; ++w) {
            const T* yw = reinterpret_cast<const T*>(smem_raw) + (size_t)w * 2 * Mrow;
            sx += yw[2 * i];
            sy += yw[2 * i + 1];
        }
        atomicAdd(&y[rb + i].x, sx);
        atomicAdd(&y[rb + i].y, sy);
    }
}

// ---- tensor-core x formation (float32 path) --------------------------------------------
// x_p = sum_k f_p[k] w_k for 16 columns x 8 crosses at a time is the real-matrix product
// of W_sigma^T (columns x frequencies) and F (frequencies x crosses), split into four real
// products per complex product, each on the tensor cores in the three-term TF32 split
// of g3_device.cuh.
// row stride (floats) of the split fibers in shared memory: >= the padded frequency
// count and 4 mod 8, so the eight rows of a B fragment fall in distinct banks
__host__ __device__ constexpr int tc_fiber_stride(int Ku) { return (Ku + 7) / 8 * 8 + 4; }

// One warp: x^+-_p[j] = sum_k f_p[k] w^+-_k[j] for 16 columns j0.. and 8 crosses into
// xs[p * ldx + j] (columns up to the padded tile).  fsp: the crosses' fibers split into
// TF32 parts, [4][ldp][KS] (re hi, re lo, im hi, im lo), rows p0 .. p0 + 7.
__device__ __forceinline__ void x_tile_tc(const WPair<float>* __restrict__ w, int E, int Ku, int jn, int j0,
                                          const unsigned* fsp, int ldp, int KS, int p0, WPair<float>* xs, int ldx) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    float xr[4] = {0, 0, 0, 0}, xi[4] = {0, 0, 0, 0}, zr[4] = {0, 0, 0, 0}, zi[4] = {0, 0, 0, 0};
    const int pl = ldp * KS;
    for (int k0 = 0; k0 < Ku; k0 += 8) {
        // A fragment: (row g, col t), (g + 8, t), (g, t + 4), (g + 8, t + 4);
        // row = column j of the block, col = frequency k
        WPair<float> a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int jj = j0 + g + (q & 1) * 8, kk = k0 + t + (q >> 1) * 4;
            a[q] = jj < jn && kk < Ku ? ldw(w + (long long)kk * E + jj) : WPair<float>{0, 0, 0, 0};
        }
        unsigned prh[4], prl[4], pih[4], pil[4], mrh[4], mrl[4], mih[4], mil[4], nph[4], npl[4], nmh[4], nml[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            Tf32Pair v = tf32_split(a[q].px);
            prh[q] = v.hi;
            prl[q] = v.lo;
            v = tf32_split(a[q].py);
            pih[q] = v.hi;
            pil[q] = v.lo;
            v = tf32_split(a[q].mx);
            mrh[q] = v.hi;
            mrl[q] = v.lo;
            v = tf32_split(a[q].my);
            mih[q] = v.hi;
            mil[q] = v.lo;
        }
        tf32_neg4(pih, nph);
        tf32_neg4(pil, npl);
        tf32_neg4(mih, nmh);
        tf32_neg4(mil, nml);
        // B fragment: (row t, col g), (t + 4, g); row = frequency, col = cross
        unsigned frh[2], frl[2], fih[2], fil[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int o = (p0 + g) * KS + k0 + t + q * 4;
            frh[q] = fsp[o];
            frl[q] = fsp[pl + o];
            fih[q] = fsp[2 * pl + o];
            fil[q] = fsp[3 * pl + o];
        }
        // Re += wr fr - wi fi, Im += wr fi + wi fr for w^+ and w^-; the four
        // accumulators in turn, the small terms first
        mma_tf32(xr, prh, frl);
        mma_tf32(xi, prh, fil);
        mma_tf32(zr, mrh, frl);
        mma_tf32(zi, mrh, fil);
        mma_tf32(xr, prl, frh);
        mma_tf32(xi, prl, fih);
        mma_tf32(zr, mrl, frh);
        mma_tf32(zi, mrl, fih);
        mma_tf32(xr, nph, fil);
        mma_tf32(xi, pih, frl);
        mma_tf32(zr, nmh, fil);
        mma_tf32(zi, mih, frl);
        mma_tf32(xr, npl, fih);
        mma_tf32(xi, pil, frh);
        mma_tf32(zr, nml, fih);
        mma_tf32(zi, mil, frh);
        mma_tf32(xr, prh, frh);
        mma_tf32(xi, prh, fih);
        mma_tf32(zr, mrh, frh);
        mma_tf32(zi, mrh, fih);
        mma_tf32(xr, nph, fih);
        mma_tf32(xi, pih, frh);
        mma_tf32(zr, nmh, fih);
        mma_tf32(zi, mih, frh);
    }
    // C fragment: (row g, col 2t), (g, 2t + 1), (g + 8, 2t), (g + 8, 2t + 1)
#pragma unroll
    for (int q = 0; q < 4; ++q)
        xs[(2 * t + (q & 1)) * ldx + j0 + g + (q >> 1) * 8] = WPair<float>{xr[q], xi[q], zr[q], zi[q]};
}

// x += f w for both combinations
template <class T>
__device__ __forceinline__ void wfma(WPair<T>& x, Cx<T> f, WPair<T> w) {
    x.px = fma(f.x, w.px, x.px);
    x.px = fma(-f.y, w.py, x.px);
    x.py = fma(f.x, w.py, x.py);
    x.py = fma(f.y, w.px, x.py);
    x.mx = fma(f.x, w.mx, x.mx);
    x.mx = fma(-f.y, w.my, x.mx);
    x.my = fma(f.x, w.my, x.my);
    x.my = fma(f.y, w.mx, x.my);
}

// sixteen sums over a warp with sixteen exchanges: each step halves the values a
// lane carries.  Returns value (lane >> 1) (both lanes of a pair).
template <class T>
__device__ __forceinline__ T warp_sum16(T* v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = 8, o = 16; n >= 1; n >>= 1, o >>= 1) {
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const T send = hi ? v[i] : v[i + n], keep = hi ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Far field, blocks with low-rank faces: one CTA per work item (block, group
// of PG crosses), every factor read once from HBM and every item complete in
// itself (no second pass, no global scratch):
//   1. x^+-_p[j] = sum_k f_p[k] w^+-_k[j] for the group's crosses and a chunk of
//      the block's columns (the fibers in shared memory, W read from L2; on the
//      tensor cores a warp per 16 columns, else TPC threads per column, each
//      with PG / TPC crosses);
//   2. a^+-_p[t] += V_p[:, t]^H x^+-_p over the chunk (a warp takes four columns t
//      of one cross at a time, which share x; lanes over the chunk), the sums
//      kept in shared memory;
//   3. the rows of y from U_p and a^+- (TPR threads per row splitting the pairs,
//      lanes over rows, one atomic add per row and part).
// Bound by the latency of 1 to 3 at three CTAs per SM (registers; two CTAs: 0.99
// against 0.85 ms for the whole far field, four with spills 0.91).  12,288-triangle
// double layer, 2.49 GB of factors, far field alone: 0.93 -> 0.85 ms.
template <class T, int NT, int PG, int TPC, bool TC>
__global__ void __launch_bounds__(NT, 3) k_far_lr(const Cx<T>* __restrict__ pool, const CrossRec* __restrict__ rec,
                                               const int* __restrict__ r3, const BlockRange* __restrict__ ranges,
                                               const int4* __restrict__ items, int Cmax, int Ku, int E,
                                               const WPair<T>* __restrict__ Wp, Cx<T>* __restrict__ y) {
    constexpr int NC = NT / TPC;    // columns per chunk
    constexpr int PPT = PG / TPC;   // crosses per thread in phase 1
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WPair<T>* xs = reinterpret_cast<WPair<T>*>(smem_raw);  // [PG][NC]
    WPair<T>* ab = xs + PG * NC;                            // [sum of ranks]
    // the fibers: [PG][Ku], or (TC) split into TF32 parts, zero beyond Ku
    const int KS = tc_fiber_stride(Ku);
    Cx<T>* fg = reinterpret_cast<Cx<T>*>(ab + PG * RF_TS);
    unsigned* fsp = reinterpret_cast<unsigned*>(fg);
    __shared__ CrossRec crs[PG];
    __shared__ int pre[PG + 1], gpre[PG + 1];         // columns and groups of four columns before each cross
    __shared__ long long ubase[PG * RF_TS];           // pool offset of U_p[:, t] of each pair
    const int4 it = items[blockIdx.x];
    const int blk = it.x, g0 = it.y * PG;
    const BlockRange br = ranges[blk];
    const int M = br.re - br.rb, N = br.ce - br.cb;
    const int np = min(PG, r3[blk] - g0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < PG) crs[tid] = tid < np ? rec[(size_t)blk * Cmax + g0 + tid] : CrossRec{0, 0, 0, 0, 0};
    __syncthreads();
    if (tid == 0) {
        pre[0] = gpre[0] = 0;
        for (int p = 0; p < PG; ++p) {
            const int r = p < np ? crs[p].r : 0;
            pre[p + 1] = pre[p] + r;
            gpre[p + 1] = gpre[p] + (r + 3) / 4;
        }
    }
    if constexpr (TC) {
        static_assert(sizeof(T) == 4 && PG == 8, "tensor-core x formation: float32, 8 crosses per item");
        for (int e = tid; e < PG * KS; e += NT) {
            const int p = e / KS, k = e - p * KS;
            Cx<T> f{0, 0};
            if (p < np && k < Ku) f = ldcx(pool + crs[p].off + (long long)crs[p].r * (M + N) + k);
            const Tf32Pair re = tf32_split(f.x), im = tf32_split(f.y);
            fsp[e] = re.hi;
            fsp[PG * KS + e] = re.lo;
            fsp[2 * PG * KS + e] = im.hi;
            fsp[3 * PG * KS + e] = im.lo;
        }
    } else {
        for (int e = tid; e < PG * Ku; e += NT) {
            const int p = e / Ku, k = e - p * Ku;
            fg[e] = p < np ? ldcx(pool + crs[p].off + (long long)crs[p].r * (M + N) + k) : Cx<T>{0, 0};
        }
    }
    __syncthreads();
    const int npt = pre[PG], ngr = gpre[PG];
    for (int q = tid; q < npt; q += NT) {
        int p = 0;
        while (pre[p + 1] <= q) ++p;
        ubase[q] = crs[p].off + (long long)(q - pre[p]) * M;
        ab[q] = WPair<T>{0, 0, 0, 0};
    }
    for (int c0 = 0; c0 < N; c0 += NC) {
        const int jn = min(NC, N - c0);
        const WPair<T>* w = Wp + br.cb + c0;
        // ---- 1. x^+- for the chunk ----
        if constexpr (TC) {
            for (int tile = warp; tile * 16 < jn; tile += NW) x_tile_tc(w, E, Ku, jn, tile * 16, fsp, PG, KS, 0, xs, NC);
        } else {
            const int jl = tid % NC, h = tid / NC;   // column, part of the group
            WPair<T> x[PPT];
#pragma unroll
            for (int u = 0; u < PPT; ++u) x[u] = WPair<T>{0, 0, 0, 0};
            if (jl < jn) {
                const Cx<T>* f0 = fg + h * PPT * Ku;
                // eight W loads in flight, then their FMAs
                int k = 0;
                for (; k + 8 <= Ku; k += 8) {
                    WPair<T> a[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) a[q] = ldw(w + (long long)(k + q) * E + jl);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
#pragma unroll
                        for (int u = 0; u < PPT; ++u) wfma(x[u], f0[u * Ku + k + q], a[q]);
                }
                for (; k < Ku; ++k) {
                    const WPair<T> a = ldw(w + (long long)k * E + jl);
#pragma unroll
                    for (int u = 0; u < PPT; ++u) wfma(x[u], f0[u * Ku + k], a);
                }
            }
#pragma unroll
            for (int u = 0; u < PPT; ++u) xs[(h * PPT + u) * NC + jl] = x[u];
        }
        __syncthreads();
        // ---- 2. a^+-_p[t] += V_p[:, t]^H x^+-_p, four columns t per warp ----
        for (int gq = warp; gq < ngr; gq += NW) {
            int p = 0;
            while (gpre[p + 1] <= gq) ++p;
            const int t0 = (gq - gpre[p]) * 4, tn = min(4, crs[p].r - t0);
            const Cx<T>* V = pool + crs[p].off + (long long)crs[p].r * M + (long long)t0 * N + c0;
            const Cx<T>* Vq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) Vq[u] = V + (long long)min(u, tn - 1) * N;
            const WPair<T>* xq = xs + p * NC;
            T v16[16];   // [u][px, py, mx, my]
#pragma unroll
            for (int u = 0; u < 16; ++u) v16[u] = 0;
#pragma unroll 2
            for (int jj = lane; jj < jn; jj += 32) {
                Cx<T> v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = ldcx_once(Vq[u] + jj);
                const WPair<T> x = ldw(xq + jj);
#pragma unroll
                for (int u = 0; u < 4; ++u) {  // conj(v) x
                    v16[4 * u] = fma(v[u].x, x.px, v16[4 * u]);
                    v16[4 * u] = fma(v[u].y, x.py, v16[4 * u]);
                    v16[4 * u + 1] = fma(v[u].x, x.py, v16[4 * u + 1]);
                    v16[4 * u + 1] = fma(-v[u].y, x.px, v16[4 * u + 1]);
                    v16[4 * u + 2] = fma(v[u].x, x.mx, v16[4 * u + 2]);
                    v16[4 * u + 2] = fma(v[u].y, x.my, v16[4 * u + 2]);
                    v16[4 * u + 3] = fma(v[u].x, x.my, v16[4 * u + 3]);
                    v16[4 * u + 3] = fma(-v[u].y, x.mx, v16[4 * u + 3]);
                }
            }
            const T sum = warp_sum16(v16);
            const int u = lane >> 3, comp = (lane >> 1) & 3;
            if ((lane & 1) == 0 && u < tn) reinterpret_cast<T*>(ab + pre[p] + t0 + u)[comp] += sum;
        }
        __syncthreads();
    }
    // ---- 3. rows of y: TPR threads per row split the flattened pairs ----
    const int tpr = M <= NT / 4 ? 4 : (M <= NT / 2 ? 2 : 1);
    const int rows = NT / tpr;
    const int h = tid / rows, il = tid - h * rows;
    for (int i0 = 0; i0 < M; i0 += rows) {
        const int i = i0 + il;
        if (i >= M) continue;
        T sx[2] = {0, 0}, sy[2] = {0, 0};
        int q = h;
        // sixteen U loads in flight per thread, then their multiply-adds
        for (; q + 15 * tpr < npt; q += 16 * tpr) {
            Cx<T> u[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) u[e] = ldcx_once(pool + ubase[q + e * tpr] + i);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const WPair<T> a = ldw(ab + q + e * tpr);
                sx[e & 1] += u[e].x * a.px - u[e].y * a.py;
                sy[e & 1] += u[e].x * a.my + u[e].y * a.mx;
            }
        }
#pragma unroll 4
        for (; q < npt; q += tpr) {
            const Cx<T> u = ldcx_once(pool + ubase[q] + i);
            const WPair<T> a = ldw(ab + q);
            sx[0] += u.x * a.px - u.y * a.py;
            sy[0] += u.x * a.my + u.y * a.mx;
        }
        atomicAdd(&y[br.rb + i].x, sx[0] + sx[1]);
        atomicAdd(&y[br.rb + i].y, sy[0] + sy[1]);
    }
}

// Far field, blocks with dense faces (small blocks): one CTA per item, up to FD_SL
// crosses (slots) of blocks with the same column cluster, whose x^+- share the
// column cluster's slice of W:
//   1. x^+-[slot][j] for a chunk of FD_NC columns: the fibers staged in shared memory,
//      on the tensor cores a warp per (16 columns, 8 slots), else a thread per (column,
//      four slots);
//   2. each warp takes FD_SL / 4 consecutive slots: lane i sums Re, Im of H x over
//      the chunk's columns for its rows, and adds a block's rows to y when its slots
//      end.
// Forming x per block (one warp each, a thread per column, four crosses at a time)
// took three quarters of the instructions and read W once per four crosses.
constexpr int FD_NT = 128, FD_SL = 16, FD_NC = 64;
template <class T, int MQ, bool TC>
__global__ void __launch_bounds__(FD_NT) k_apply_far_dense(const Cx<T>* __restrict__ pool,
                                                           const CrossRec* __restrict__ rec,
                                                           const BlockRange* __restrict__ ranges,
                                                           const int4* __restrict__ items, const int2* __restrict__ slots,
                                                           int Cmax, int Ku, int E, const WPair<T>* __restrict__ Wp,
                                                           Cx<T>* __restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    WPair<T>* xs = reinterpret_cast<WPair<T>*>(smem_raw);   // [FD_SL][FD_NC]
    const int KS = tc_fiber_stride(Ku);
    Cx<T>* fg = reinterpret_cast<Cx<T>*>(xs + FD_SL * FD_NC);  // [FD_SL][Ku], or (TC) TF32 parts
    unsigned* fsp = reinterpret_cast<unsigned*>(fg);
    __shared__ long long soff[FD_SL];
    __shared__ int sblk[FD_SL], srb[FD_SL], sm[FD_SL];
    const int4 it = items[blockIdx.x];                      // first slot, slots, first column, columns
    const int ns = it.y, cb = it.z, N = it.w;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < FD_SL) {
        sblk[tid] = -1;
        if (tid < ns) {
            const int2 sl = slots[it.x + tid];
            const BlockRange br = ranges[sl.x];
            sblk[tid] = sl.x;
            srb[tid] = br.rb;
            sm[tid] = br.re - br.rb;
            soff[tid] = rec[(size_t)sl.x * Cmax + sl.y].off;
        }
    }
    __syncthreads();
    if constexpr (TC) {
        for (int e = tid; e < FD_SL * KS; e += FD_NT) {
            const int p = e / KS, k = e - p * KS;
            Cx<T> f{0, 0};
            if (p < ns && k < Ku) f = ldcx(pool + soff[p] + (long long)sm[p] * N + k);
            const Tf32Pair re = tf32_split(f.x), im = tf32_split(f.y);
            fsp[e] = re.hi;
            fsp[FD_SL * KS + e] = re.lo;
            fsp[2 * FD_SL * KS + e] = im.hi;
            fsp[3 * FD_SL * KS + e] = im.lo;
        }
    } else {
        for (int e = tid; e < FD_SL * Ku; e += FD_NT) {
            const int p = e / Ku, k = e - p * Ku;
            fg[e] = p < ns ? ldcx(pool + soff[p] + (long long)sm[p] * N + k) : Cx<T>{0, 0};
        }
    }
    __syncthreads();
    for (int c0 = 0; c0 < N; c0 += FD_NC) {
        const int jn = min(FD_NC, N - c0);
        const WPair<T>* w = Wp + cb + c0;
        if constexpr (TC) {
            const int nt = (jn + 15) / 16, np8 = (ns + 7) / 8;
            for (int q = warp; q < nt * np8; q += FD_NT / 32)
                x_tile_tc(w, E, Ku, jn, (q % nt) * 16, fsp, FD_SL, KS, (q / nt) * 8, xs + (q / nt) * 8 * FD_NC, FD_NC);
        } else {
            const int np4 = (ns + 3) / 4;
            for (int q = tid; q < jn * np4; q += FD_NT) {
                const int jl = q % jn, p0 = (q / jn) * 4;
                WPair<T> x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = WPair<T>{0, 0, 0, 0};
#pragma unroll 4
                for (int k = 0; k < Ku; ++k) {
                    const WPair<T> a = ldw(w + (long long)k * E + jl);
#pragma unroll
                    for (int u = 0; u < 4; ++u) wfma(x[u], fg[(p0 + u) * Ku + k], a);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) xs[(p0 + u) * FD_NC + jl] = x[u];
            }
        }
        __syncthreads();
        T ax[MQ], ay[MQ];
#pragma unroll
        for (int q = 0; q < MQ; ++q) ax[q] = ay[q] = 0;
        constexpr int SPW = FD_SL / (FD_NT / 32);
        for (int p = warp * SPW; p < min(ns, (warp + 1) * SPW); ++p) {
            const int M = sm[p];
            const Cx<T>* H = pool + soff[p] + (long long)c0 * M;
            const WPair<T>* x = xs + p * FD_NC;
#pragma unroll
            for (int q = 0; q < MQ; ++q) {
                const int i = lane + 32 * q;
                if (i < M) {
                    T bx = 0, by = 0;
#pragma unroll 8
                    for (int jj = 0; jj < jn; ++jj) {
                        const Cx<T> h = ldcx_once(H + i + (long long)jj * M);
                        const WPair<T> v = ldw(x + jj);
                        bx += h.x * v.px - h.y * v.py;
                        by += h.x * v.my + h.y * v.mx;
                    }
                    ax[q] += bx;
                    ay[q] += by;
                }
            }
            if (p + 1 == min(ns, (warp + 1) * SPW) || sblk[p + 1] != sblk[p]) {  // the block's last slot here
#pragma unroll
                for (int q = 0; q < MQ; ++q) {
                    const int i = lane + 32 * q;
                    if (i < M) {
                        atomicAdd(&y[srb[p] + i].x, ax[q]);
                        atomicAdd(&y[srb[p] + i].y, ay[q]);
                    }
                    ax[q] = ay[q] = 0;
                }
            }
        }
        __syncthreads();   // x is consumed
    }
}

template <class T, class TO>
__global__ void k_apply_finish(int E, const int* __restrict__ perm, const Cx<T>* __restrict__ y, Cx<TO>* __restrict__ Y) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= E) return;
    Cx<T> v = y[p];
    Y[perm[p]] = Cx<TO>{(TO)v.x, (TO)v.y};
}
// linear elements: y = P^T y_loc, each position's row added into its vertex
// (Y cleared before)
template <class T, class TO>
__global__ void k_apply_finish_add(int E, const int* __restrict__ src, const Cx<T>* __restrict__ y,
                                   Cx<TO>* __restrict__ Y) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= E) return;
    Cx<T> v = y[p];
    atomicAdd(&Y[src[p]].x, (TO)v.x);
    atomicAdd(&Y[src[p]].y, (TO)v.y);
}


// near-field launch: grid (row clusters) x (frequency chunks), several CTAs per
// resident slot so that the last wave is short
template <class T>
static g3_status launch_apply_near(g3_ctx* ctx, cudaStream_t stream, const g3_tree* t, const g3_near* nf, int Ku,
                                   int E, const WPair<T>* Wp, Cx<T>* y) {
    const int n_rows = (int)nf->row_start.size() - 1;
    const int ksplit0 = std::max(1, std::min(Ku, (32 * ctx->n_sm + n_rows - 1) / n_rows));
    const int kchunk = (Ku + ksplit0 - 1) / ksplit0, ksplit = (Ku + kchunk - 1) / kchunk;
    int mrow = 0;
    for (int g = 0; g < n_rows; ++g) {
        const int32_t* r = &t->blocks[5 * (size_t)nf->order[nf->row_start[g]]];
        mrow = std::max(mrow, r[1] - r[0]);
    }
    dim3 grid(n_rows, ksplit);
    const size_t smem = (size_t)NEAR_NW * NEAR_ST * near_stage_bytes<T>() + NEAR_NW * 2 * (size_t)mrow * sizeof(T);
    if ((size_t)mrow * sizeof(Cx<T>) <= (size_t)NEAR_A - 16 && smem <= ctx->smem_optin) {
        G3_CUDA(cudaFuncSetAttribute(k_apply_near<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_apply_near<T><<<grid, NEAR_NW * 32, smem, stream>>>(
            nf->data.as<Cx<T>>(), nf->d_ranges.as<BlockRange>(), nf->d_offs.as<long long>(), nf->d_row_start.as<int>(),
            Ku, kchunk, E, Wp, y);
        ctx->count("k_apply_near");
    } else {
        constexpr int NT = 256;
        const size_t wsm = (NT / 32) * 2 * (size_t)mrow * sizeof(T);
        if (wsm > ctx->smem_optin)
            return fail(G3_EUNSUPPORTED, "apply_gcq: near-field clusters of %d rows exceed the apply kernel's limit", mrow);
        G3_CUDA(cudaFuncSetAttribute(k_apply_near_wide<T, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wsm));
        k_apply_near_wide<T, NT><<<grid, NT, wsm, stream>>>(
            nf->data.as<Cx<T>>(), nf->d_ranges.as<BlockRange>(), nf->d_offs.as<long long>(), nf->d_row_start.as<int>(),
            Ku, kchunk, E, Wp, y);
        ctx->count("k_apply_near_wide");
    }
    G3_CUDA(cudaGetLastError());
    return G3_OK;
}

// Far-field work lists, built on the host when the compression ends and
// uploaded with the block ranges, as int4 items: the dense-face items (first slot,
// slots, first column, columns), the low-rank items (block, group of FAR_PG
// crosses) of blocks with at most FAR_NT / 2 columns (two threads per column in
// the x formation), those of wider blocks; then the dense items' slots
// (block, cross).  Each list by column cluster.
constexpr int FAR_PG = 8;
constexpr int FAR_NT = 256;

g3_status far_plan_build(g3_factors* fa) {
    std::vector<int>& L = fa->plan;
    L.clear();
    struct Item {
        long long cost;
        int b, g;
    };
    std::vector<Item> narrow, wide, dense;
    int mmax = 0;
    for (int b = 0; b < fa->n_far; ++b) {
        const int r = fa->r3[b];
        if (r <= 0) continue;
        if (fa->crec(b, 0).r < 0) {
            const int M = fa->ranges[b].re - fa->ranges[b].rb, N = fa->ranges[b].ce - fa->ranges[b].cb;
            dense.push_back(Item{(long long)r * M * N, b, 0});
            mmax = std::max(mmax, M);
            continue;
        }
        const int M = fa->ranges[b].re - fa->ranges[b].rb;
        const int N = fa->ranges[b].ce - fa->ranges[b].cb;
        for (int p = 0; p < r; ++p)
            if (fa->crec(b, p).r > RF_TS)
                return fail(G3_EUNSUPPORTED, "aca3_compress: face rank %d above the apply's limit %d",
                            fa->crec(b, p).r, RF_TS);
        for (int g = 0; g * FAR_PG < r; ++g) {
            long long c = 0;
            for (int p = g * FAR_PG; p < std::min(r, (g + 1) * FAR_PG); ++p)
                c += (long long)fa->crec(b, p).r * (M + N) + fa->Ku;
            (N <= FAR_NT / 2 ? narrow : wide).push_back(Item{c, b, g});
        }
    }
    auto by_cost = [](const Item& x, const Item& y) {
        if (x.cost != y.cost) return x.cost > y.cost;
        return x.b != y.b ? x.b < y.b : x.g < y.g;
    };
    // items grouped by column cluster (longest first within a cluster): CTAs that
    // run at the same time read the same slice of W, which stays in L2 even when
    // W as a whole does not (81,920 elements x 128 unique frequencies: 168 MB;
    // far field 34.8 against 39.0 ms longest first)
    auto by_col = [&](const Item& x, const Item& y) {
        const BlockRange &rx = fa->ranges[x.b], &ry = fa->ranges[y.b];
        if (rx.cb != ry.cb) return rx.cb < ry.cb;
        if (rx.ce != ry.ce) return rx.ce < ry.ce;
        return by_cost(x, y);
    };
    std::sort(narrow.begin(), narrow.end(), by_col);
    std::sort(wide.begin(), wide.end(), by_col);
    std::sort(dense.begin(), dense.end(), by_col);
    // dense items: up to FD_SL crosses (slots) of blocks with the same columns
    std::vector<int> slots;   // (block, cross) pairs
    int nd = 0, cb = -1, ce = -1, first = 0;
    auto close = [&]() {
        const int n = (int)slots.size() / 2 - first;
        if (n > 0) {
            L.insert(L.end(), {first, n, cb, ce - cb});
            ++nd;
        }
        first += n;
    };
    for (const Item& it : dense) {
        const BlockRange& r = fa->ranges[it.b];
        for (int p = 0; p < fa->r3[it.b]; ++p) {
            if (r.cb != cb || r.ce != ce || (int)slots.size() / 2 - first == FD_SL) {
                close();
                cb = r.cb;
                ce = r.ce;
            }
            slots.insert(slots.end(), {it.b, p});
        }
    }
    close();
    fa->plan_nd = nd;
    fa->plan_n1 = (int)narrow.size();
    fa->plan_n2 = (int)wide.size();
    fa->plan_mmax_dense = mmax;
    for (const Item& it : narrow) L.insert(L.end(), {it.b, it.g, 0, 0});
    for (const Item& it : wide) L.insert(L.end(), {it.b, it.g, 0, 0});
    L.insert(L.end(), slots.begin(), slots.end());
    G3_CUDA(fa->d_plan.alloc(std::max<size_t>(1, L.size()) * sizeof(int)));
    const cudaStream_t stream = fa->ctx->stream;
    G3_CUDA(upload(stream, fa->d_plan.p, L.data(), L.size() * sizeof(int)));
    G3_CUDA(fa->d_franges.alloc(std::max<size_t>(1, fa->ranges.size()) * sizeof(BlockRange)));
    G3_CUDA(upload(stream, fa->d_franges.p, fa->ranges.data(), fa->ranges.size() * sizeof(BlockRange)));
    G3_CUDA(cudaStreamSynchronize(stream));  // the factors may be applied from another context
    fa->plan_ready = true;
    return G3_OK;
}

// far-field launches over the factors' device work lists
template <class T>
static g3_status launch_apply_far(g3_ctx* ctx, const g3_factors* fa, int Ku, int E, const WPair<T>* Wp, Cx<T>* y) {
    if (!fa->plan_ready) return fail(G3_EINVAL, "apply_gcq: factors without far-field work lists");
    if (fa->plan.empty()) return G3_OK;
    const int nd = fa->plan_nd, n1 = fa->plan_n1, n2 = fa->plan_n2;
    const int4* it0 = fa->d_plan.as<int4>();
    const int4* it1 = it0 + nd;
    const int4* it2 = it1 + n1;
    const int2* slots = reinterpret_cast<const int2*>(it2 + n2);
    const BlockRange* d_ranges = fa->d_franges.as<BlockRange>();
    const bool tc = sizeof(T) == 4 && ctx->apply_tensor_cores;
    // fibers of n crosses in shared memory
    auto fiber_bytes = [&](int n) {
        return tc ? 4 * (size_t)n * tc_fiber_stride(Ku) * sizeof(unsigned) : (size_t)n * Ku * sizeof(Cx<T>);
    };
    if (nd > 0) {
        const int mmax = fa->plan_mmax_dense;
        const size_t smem = (size_t)FD_SL * FD_NC * sizeof(WPair<T>) + fiber_bytes(FD_SL);
        if (smem > ctx->smem_optin || mmax > 256)
            return fail(G3_EUNSUPPORTED, "apply_gcq: dense-face blocks with %d rows exceed the apply kernel's limit", mmax);
        auto go = [&](auto kfn) -> g3_status {
            G3_CUDA(cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            kfn<<<nd, FD_NT, smem, ctx->stream>>>(fa->pool->as<Cx<T>>(), fa->d_rec.as<CrossRec>(), d_ranges, it0, slots,
                                                  fa->Cmax, Ku, E, Wp, y);
            return G3_OK;
        };
        auto by_rows = [&](auto use_tc) -> g3_status {
            constexpr bool TC = decltype(use_tc)::value;
            if (mmax <= 32) return go(k_apply_far_dense<T, 1, TC>);
            if (mmax <= 64) return go(k_apply_far_dense<T, 2, TC>);
            if (mmax <= 128) return go(k_apply_far_dense<T, 4, TC>);
            return go(k_apply_far_dense<T, 8, TC>);
        };
        if constexpr (sizeof(T) == 4) {
            G3_TRY_NA(tc ? by_rows(std::true_type{}) : by_rows(std::false_type{}));
        } else {
            G3_TRY_NA(by_rows(std::false_type{}));
        }
        ctx->count("k_apply_far_dense");
        G3_CUDA(cudaGetLastError());
    }
    auto far_lr = [&](auto kfn, int n, const int4* items, int nc) -> g3_status {
        if (n <= 0) return G3_OK;
        const size_t smem = (size_t)FAR_PG * (nc + RF_TS) * sizeof(WPair<T>) + fiber_bytes(FAR_PG);
        if (smem > ctx->smem_optin)
            return fail(G3_EUNSUPPORTED, "apply_gcq: far-field kernel needs %zu bytes of shared memory", smem);
        G3_CUDA(cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kfn<<<n, FAR_NT, smem, ctx->stream>>>(fa->pool->as<Cx<T>>(), fa->d_rec.as<CrossRec>(), fa->d_r3.as<int>(),
                                              d_ranges, items, fa->Cmax, Ku, E, Wp, y);
        ctx->count(tc ? "k_far_lr_tc" : "k_far_lr");
        G3_CUDA(cudaGetLastError());
        return G3_OK;
    };
    if constexpr (sizeof(T) == 4) {
        if (tc) {
            G3_TRY_NA(far_lr(k_far_lr<T, FAR_NT, FAR_PG, 2, true>, n1, it1, FAR_NT / 2));
            G3_TRY_NA(far_lr(k_far_lr<T, FAR_NT, FAR_PG, 1, true>, n2, it2, FAR_NT));
            return G3_OK;
        }
    }
    G3_TRY_NA(far_lr(k_far_lr<T, FAR_NT, FAR_PG, 2, false>, n1, it1, FAR_NT / 2));
    G3_TRY_NA(far_lr(k_far_lr<T, FAR_NT, FAR_PG, 1, false>, n2, it2, FAR_NT));
    return G3_OK;
}

// Near field and far field of one apply.  With both present the near field
// (an HBM stream) runs on the context's high-priority side stream and the
// far-field kernels (bound by latency: short dependent chains per item) on the
// context's stream, forked and joined through events: pending near-field CTAs
// are dispatched first and far-field CTAs fill the rest of each SM, which
// overlaps the two better than the opposite priority (measured on the
// 12,288-triangle L-shape: 1.88 against 1.95 ms per single-layer apply).
// Both add into y atomically.  ev_side brackets the near field (its device time).
template <class T>
static g3_status apply_near_far(g3_ctx* ctx, const g3_tree* t, const g3_near* nf, const g3_factors* fa, int Ku,
                                int E, const WPair<T>* Wp, Cx<T>* y) {
    const bool has_near = nf && !nf->order.empty(), has_far = fa && fa->n_far > 0;
    if (has_near && has_far) {
        G3_CUDA(cudaEventRecord(ctx->fork, ctx->stream));
        G3_CUDA(cudaStreamWaitEvent(ctx->side, ctx->fork, 0));
        G3_CUDA(cudaEventRecord(ctx->ev_side[0], ctx->side));
        G3_TRY_NA(launch_apply_near<T>(ctx, ctx->side, t, nf, Ku, E, Wp, y));
        G3_CUDA(cudaEventRecord(ctx->ev_side[1], ctx->side));
        G3_CUDA(cudaEventRecord(ctx->join, ctx->side));
        G3_TRY_NA(launch_apply_far<T>(ctx, fa, Ku, E, Wp, y));
        G3_CUDA(cudaStreamWaitEvent(ctx->stream, ctx->join, 0));
        return G3_OK;
    }
    if (has_near) {
        G3_CUDA(cudaEventRecord(ctx->ev_side[0], ctx->stream));
        G3_TRY_NA(launch_apply_near<T>(ctx, ctx->stream, t, nf, Ku, E, Wp, y));
        G3_CUDA(cudaEventRecord(ctx->ev_side[1], ctx->stream));
    }
    if (has_far) G3_TRY_NA(launch_apply_far<T>(ctx, fa, Ku, E, Wp, y));
    return G3_OK;
}

template <class T>
static g3_status launch_prep_pm(g3_ctx* ctx, int E, const g3_freqs* f, const int* rowsrc, const void* W, int dtype,
                                WPair<T>* Wp, Cx<T>* y, int ldw) {
    const dim3 grid((E + 127) / 128, f->Ku);
    if (dtype == G3_C128)
        k_apply_prep_pm<double, T><<<grid, 128, 0, ctx->stream>>>(E, f->Ku, rowsrc, f->d_uniq.as<int>(), f->d_partner.as<int>(),
                                                                  (const Cx<double>*)W, Wp, y, ldw);
    else
        k_apply_prep_pm<float, T><<<grid, 128, 0, ctx->stream>>>(E, f->Ku, rowsrc, f->d_uniq.as<int>(), f->d_partner.as<int>(),
                                                                 (const Cx<float>*)W, Wp, y, ldw);
    ctx->count("k_apply_prep");
    G3_CUDA(cudaGetLastError());
    return G3_OK;
}

template <class T>
static g3_status run_apply_t(g3_ctx* ctx, const g3_tree* t, const g3_near* nf, const g3_factors* fa, const void* W,
                             void* Y, int dtype, const g3_freqs* f) {
    const int E = t->ne, K = f->K, Ku = f->Ku;
    const size_t nW = (size_t)Ku * E;
    const size_t need = nW * sizeof(WPair<T>) + E * sizeof(Cx<T>);
    G3_CUDA(ctx->scratch.ensure(need));
    WPair<T>* Wp = ctx->scratch.as<WPair<T>>();
    Cx<T>* y = reinterpret_cast<Cx<T>*>(Wp + nW);
    cudaEvent_t e0 = ctx->ev[2], e3 = ctx->ev[5];
    G3_CUDA(cudaEventRecord(e0, ctx->stream));
    // linear-element trees: nodal W and Y (nv rows), gathered per position at its vertex
    const int* rowsrc = t->p1 ? t->d_src.as<int>() : t->d_perm.as<int>();
    const int ldw = t->p1 ? t->nv : E;
    G3_TRY_NA(launch_prep_pm<T>(ctx, E, f, rowsrc, W, dtype, Wp, y, ldw));
    G3_TRY_NA(apply_near_far<T>(ctx, t, nf, fa, Ku, E, Wp, y));
    {
        int blocks = (E + 255) / 256;
        if (t->p1) {
            G3_CUDA(cudaMemsetAsync(Y, 0, (size_t)t->nv * (dtype == G3_C128 ? 16 : 8), ctx->stream));
            if (dtype == G3_C128)
                k_apply_finish_add<T, double><<<blocks, 256, 0, ctx->stream>>>(E, rowsrc, y, (Cx<double>*)Y);
            else
                k_apply_finish_add<T, float><<<blocks, 256, 0, ctx->stream>>>(E, rowsrc, y, (Cx<float>*)Y);
            ctx->count("k_apply_finish_add");
        } else {
            if (dtype == G3_C128)
                k_apply_finish<T, double><<<blocks, 256, 0, ctx->stream>>>(E, t->d_perm.as<int>(), y, (Cx<double>*)Y);
            else
                k_apply_finish<T, float><<<blocks, 256, 0, ctx->stream>>>(E, t->d_perm.as<int>(), y, (Cx<float>*)Y);
            ctx->count("k_apply_finish");
        }
        G3_CUDA(cudaGetLastError());
    }
    G3_CUDA(cudaEventRecord(e3, ctx->stream));
    G3_CUDA(cudaEventSynchronize(e3));
    float ms_all = 0, ms_near = 0;
    G3_CUDA(cudaEventElapsedTime(&ms_all, e0, e3));
    if (nf && !nf->order.empty()) G3_CUDA(cudaEventElapsedTime(&ms_near, ctx->ev_side[0], ctx->ev_side[1]));
    ctx->last_apply_ms = ms_all;
    ctx->last_near_ms = ms_near;
    const int64_t in_sz = dtype == G3_C128 ? 16 : 8;
    int64_t near_bytes = nf ? nf->n_entries * (int64_t)sizeof(Cx<T>) : 0;
    int64_t far_bytes = fa ? fa->stats.factor_bytes : 0;
    ctx->last_near_bytes = near_bytes;
    ctx->last_apply_bytes = near_bytes + far_bytes + (int64_t)E * K * in_sz + (int64_t)E * in_sz;
    return G3_OK;
}

// ============================================================================
// Per-frequency apply (G3_APPLY_PERFREQ): Y[:, l] = A(s_l) w_l for every l
// ============================================================================
//
// The terms of eq. (product) before the sum over l, one column per frequency
// (a check of the compressed operator at each frequency).  With the unique
// frequencies k and their partners k' (A(s_k') = conj A(s_k)):
//   Y[:, k]  = A(s_k) w_k               = sum_far sum_p f_p[k] H_p w_k + near,
//   Y[:, k'] = conj(A(s_k) conj(w_k'))  (the same operator on conj(w_k')).
// So every unique frequency k has two right-hand sides, x_k = w_k and
// x_{Ku + k} = conj(w_k') (zero without a partner), and two outputs
// yf[k] and yc[k] in cluster order; Y[:, k'] = conj(yc[k]).  Scratch:
// Wf, Wc (from k_apply_prep, Wc unconjugated), yf, yc: 4 Ku E values.

// near field: one CTA per (near block, frequency chunk); warp per frequency,
// lane per row; both right-hand sides in one pass over the stored entries
template <class T, int NT>
__global__ void __launch_bounds__(NT) k_pf_near(const Cx<T>* __restrict__ A, const BlockRange* __restrict__ ranges,
                                                const long long* __restrict__ offs, int Ku, int kchunk, int E,
                                                const Cx<T>* __restrict__ Wf, const Cx<T>* __restrict__ Wc,
                                                Cx<T>* __restrict__ yf, Cx<T>* __restrict__ yc) {
    const int b = blockIdx.x;
    const int k0 = blockIdx.y * kchunk, k1 = min(Ku, k0 + kchunk);
    const BlockRange br = ranges[b];
    const int M = br.re - br.rb, N = br.ce - br.cb;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = k0 + warp; k < k1; k += NT / 32) {
        const Cx<T>* Ak = A + offs[b] + (long long)k * M * N;
        const Cx<T>* wf = Wf + (long long)k * E + br.cb;
        const Cx<T>* wc = Wc + (long long)k * E + br.cb;
        for (int i = lane; i < M; i += 32) {
            Cx<T> s1{0, 0}, s2{0, 0};
            for (int j = 0; j < N; ++j) {
                const Cx<T> a = ldcx(Ak + (long long)j * M + i);
                cfma(s1, a, ldcx(wf + j));
                cfmac(s2, a, ldcx(wc + j));  // A conj(w')
            }
            atomicAdd(&yf[(long long)k * E + br.rb + i].x, s1.x);
            atomicAdd(&yf[(long long)k * E + br.rb + i].y, s1.y);
            atomicAdd(&yc[(long long)k * E + br.rb + i].x, s2.x);
            atomicAdd(&yc[(long long)k * E + br.rb + i].y, s2.y);
        }
    }
}

// two neighbouring values (16-byte aligned in float32)
template <class T>
__device__ __forceinline__ void ldcx2(const Cx<T>* p, Cx<T>& a, Cx<T>& b) {
    if constexpr (sizeof(T) == 4) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        a = Cx<T>{v.x, v.y};
        b = Cx<T>{v.z, v.w};
    } else {
        a = ldcx(p);
        b = ldcx(p + 1);
    }
}

// far field, blocks with dense faces: one CTA per (item of k_apply_far_dense,
// frequency chunk), the item's fibers in shared memory.  Both right-hand sides of a
// frequency see the same matrix, so it is formed once, in registers:
//   A_k[i, j] = sum_p f_p[k] H_p[i, j],  yf_k[i] += A_k[i, j] w_k[j],  yc_k[i] += A_k[i, j] conj(w'_k[j]),
// r + 2 products per entry and frequency for the 2 r of H_p x per right-hand side.
// A warp takes (the item's slots of one block, PD_KT frequencies, 32 rows), lane i row
// i; two columns at a time share the fiber values, and the values of H come from L1
// (an item's 16 faces of 24 x 24 take 74 KB).
// Before, both kinds of faces went through one kernel, a CTA per (block, 32 right-hand
// sides, 128 rows): every multiply-add read one value of H or V through a broadcast
// load, and a block of 24 rows kept 3 of a thread's 16 sums busy.  3,072-triangle
// L-shape, 33 unique frequencies, the whole per-frequency apply: 3.51 -> 1.70 ms.
constexpr int PD_NT = 128, PD_KT = 4, PD_KC = 64;
template <class T>
__global__ void __launch_bounds__(PD_NT) k_pf_far_dense(const Cx<T>* __restrict__ pool, const CrossRec* __restrict__ rec,
                                                        const BlockRange* __restrict__ ranges,
                                                        const int4* __restrict__ items, const int2* __restrict__ slots,
                                                        int Cmax, int Ku, int kchunk, int E, const Cx<T>* __restrict__ Wf,
                                                        const Cx<T>* __restrict__ Wc, Cx<T>* __restrict__ yf,
                                                        Cx<T>* __restrict__ yc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T>* fs = reinterpret_cast<Cx<T>*>(smem_raw);   // [FD_SL][KS], zero beyond the chunk
    __shared__ long long soff[FD_SL];
    __shared__ int srb[FD_SL], sm[FD_SL], run0[FD_SL + 1], n_run;
    const int4 it = items[blockIdx.x];                // first slot, slots, first column, columns
    const int ns = it.y, cb = it.z, N = it.w;
    const int k0 = blockIdx.y * kchunk, nk = min(Ku, k0 + kchunk) - k0;
    const int KS = (kchunk + PD_KT - 1) / PD_KT * PD_KT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < ns) {
        const int2 sl = slots[it.x + tid];
        const BlockRange br = ranges[sl.x];
        srb[tid] = br.rb;
        sm[tid] = br.re - br.rb;
        soff[tid] = rec[(size_t)sl.x * Cmax + sl.y].off;
    }
    if (tid == 0) {
        int n = 0;
        for (int p = 0; p < ns; ++p)
            if (p == 0 || slots[it.x + p].x != slots[it.x + p - 1].x) run0[n++] = p;
        run0[n] = ns;
        n_run = n;
    }
    __syncthreads();
    for (int e = tid; e < ns * KS; e += PD_NT) {
        const int p = e / KS, k = e - p * KS;
        fs[e] = k < nk ? ldcx(pool + soff[p] + (long long)sm[p] * N + k0 + k) : Cx<T>{0, 0};
    }
    __syncthreads();
    const int ng = (nk + PD_KT - 1) / PD_KT;
    for (int q = warp; q < n_run * ng; q += PD_NT / 32) {
        const int run = q / ng, kg = (q - run * ng) * PD_KT;
        const int pa = run0[run], pb = run0[run + 1], M = sm[pa];
        const int kn = min(PD_KT, nk - kg);
        const Cx<T>* wf = Wf + (long long)(k0 + kg) * E + cb;
        const Cx<T>* wc = Wc + (long long)(k0 + kg) * E + cb;
        for (int i0 = 0; i0 < M; i0 += 32) {
            const int i = min(i0 + lane, M - 1);      // (lanes past the block's rows repeat the last one)
            Cx<T> s1[PD_KT], s2[PD_KT];
#pragma unroll
            for (int u = 0; u < PD_KT; ++u) s1[u] = s2[u] = Cx<T>{0, 0};
            for (int j = 0; j < N; j += 2) {
                const int dj = j + 1 < N ? 1 : 0;
                Cx<T> a0[PD_KT], a1[PD_KT];
#pragma unroll
                for (int u = 0; u < PD_KT; ++u) a0[u] = a1[u] = Cx<T>{0, 0};
                const long long o = (long long)j * M + i;
#pragma unroll 4
                for (int p = pa; p < pb; ++p) {
                    const Cx<T>* H = pool + soff[p] + o;
                    const Cx<T> h0 = ldcx(H), h1 = ldcx(H + dj * M);
                    Cx<T> f[PD_KT];
#pragma unroll
                    for (int u = 0; u < PD_KT; u += 2) ldcx2(fs + p * KS + kg + u, f[u], f[u + 1]);
#pragma unroll
                    for (int u = 0; u < PD_KT; ++u) {
                        cfma(a0[u], f[u], h0);
                        cfma(a1[u], f[u], h1);
                    }
                }
#pragma unroll
                for (int u = 0; u < PD_KT; ++u) {
                    if (u < kn) {
                        const long long wo = (long long)u * E + j;
                        cfma(s1[u], a0[u], ldcx(wf + wo));
                        cfmac(s2[u], a0[u], ldcx(wc + wo));
                        if (dj) {
                            cfma(s1[u], a1[u], ldcx(wf + wo + 1));
                            cfmac(s2[u], a1[u], ldcx(wc + wo + 1));
                        }
                    }
                }
            }
            if (i0 + lane < M) {
#pragma unroll
                for (int u = 0; u < PD_KT; ++u) {
                    if (u < kn) {
                        const long long yo = (long long)(k0 + kg + u) * E + srb[pa] + i;
                        atomicAdd(&yf[yo].x, s1[u].x);
                        atomicAdd(&yf[yo].y, s1[u].y);
                        atomicAdd(&yc[yo].x, s2[u].x);
                        atomicAdd(&yc[yo].y, s2[u].y);
                    }
                }
            }
        }
    }
}

// far field, blocks with low-rank faces: one CTA per (item of k_far_lr: block and
// group of FAR_PG crosses, PF_NC right-hand sides c0..).  Right-hand side c < Ku is w_c,
// c >= Ku is conj(w'_{c-Ku}); its fiber coefficient is f_p[c mod Ku].  As many of the
// group's crosses at a time as have PF_NQ columns together:
//   1. t[q][c] = f_p[c] V_p[:, q]^H x_c, kept in shared memory;
//   2. z[i][c] = sum_q U[i, q] t[q][c], added to yf / yc.
// Both are products of tall matrices with PF_NC columns: warp w takes columns c0 + 4 w..
// (a warp without columns only stages), lane l rows 2 l, 2 l + 1 of a tile of 64, so
// that three 16-byte reads of shared memory feed 32 multiply-adds.
constexpr int PF_NT = 256, PF_NC = 32, PF_NQ = 128, PF_JC = 32, PF_LD = 66, PF_LX = 34;
template <class T>
constexpr size_t pf_lr_smem() {   // t, tile of V or U, tile of x
    return ((size_t)PF_NQ * PF_LX + (size_t)PF_JC * PF_LD + (size_t)PF_JC * PF_LX) * sizeof(Cx<T>);
}
template <class T>
__global__ void __launch_bounds__(PF_NT) k_pf_far_lr(const Cx<T>* __restrict__ pool, const CrossRec* __restrict__ rec,
                                                     const int* __restrict__ r3, const BlockRange* __restrict__ ranges,
                                                     const int4* __restrict__ items, int Cmax, int Ku, int E,
                                                     const Cx<T>* __restrict__ Wf, const Cx<T>* __restrict__ Wc,
                                                     Cx<T>* __restrict__ yf, Cx<T>* __restrict__ yc) {
    static_assert(PF_NQ >= 2 * RF_TS, "a cross's columns fit the tile of t");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Cx<T>* ts = reinterpret_cast<Cx<T>*>(smem_raw);   // [PF_NQ][PF_LX]
    Cx<T>* as = ts + PF_NQ * PF_LX;                    // [PF_JC][PF_LD]: V (column, q) or U (q, row)
    Cx<T>* xs = as + PF_JC * PF_LD;                    // [PF_JC][PF_LX]
    __shared__ CrossRec crs[FAR_PG];
    __shared__ Cx<T> fs[FAR_PG][PF_NC];
    __shared__ long long uo[PF_NQ], vo[PF_NQ];         // pool offsets of U_p[:, q], V_p[:, q]
    __shared__ int pq[PF_NQ];
    const int4 it = items[blockIdx.x];
    const int blk = it.x, g0 = it.y * FAR_PG, c0 = blockIdx.y * PF_NC, nrhs = 2 * Ku;
    const BlockRange br = ranges[blk];
    const int M = br.re - br.rb, N = br.ce - br.cb;
    const int np = min(FAR_PG, r3[blk] - g0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cw = warp * 4;
    const bool act = c0 + cw < nrhs;
    if (tid < np) crs[tid] = rec[(size_t)blk * Cmax + g0 + tid];
    __syncthreads();
    for (int e = tid; e < np * PF_NC; e += PF_NT) {
        const int p = e / PF_NC, c = e - p * PF_NC, gc = c0 + c;
        fs[p][c] = gc < nrhs ? ldcx(pool + crs[p].off + (long long)crs[p].r * (M + N) + (gc < Ku ? gc : gc - Ku))
                             : Cx<T>{0, 0};
    }
    for (int pa = 0; pa < np;) {
        int pb = pa, Q = 0;
        while (pb < np && Q + crs[pb].r <= PF_NQ) Q += crs[pb++].r;
        __syncthreads();   // the crosses before are done with the offsets and t
        if (tid < Q) {
            int p = pa, q = tid;
            while (q >= crs[p].r) q -= crs[p++].r;
            pq[tid] = p;
            uo[tid] = crs[p].off + (long long)q * M;
            vo[tid] = crs[p].off + (long long)crs[p].r * M + (long long)q * N;
        }
        // ---- 1. t ----
        for (int q0 = 0; q0 < Q; q0 += 64) {
            Cx<T> t[2][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) t[0][u] = t[1][u] = Cx<T>{0, 0};
            for (int j0 = 0; j0 < N; j0 += PF_JC) {
                const int jn = min(PF_JC, N - j0), j = br.cb + j0 + lane;
                __syncthreads();
                for (int q = warp; q < 64; q += PF_NT / 32)
                    as[lane * PF_LD + q] =
                        q0 + q < Q && lane < jn ? ldcx(pool + vo[q0 + q] + j0 + lane) : Cx<T>{0, 0};
                for (int c = warp; c < PF_NC; c += PF_NT / 32) {
                    const int gc = c0 + c;
                    Cx<T> v{0, 0};
                    if (gc < nrhs && lane < jn)
                        v = gc < Ku ? ldcx(Wf + (long long)gc * E + j) : cconj(ldcx(Wc + (long long)(gc - Ku) * E + j));
                    xs[lane * PF_LX + c] = v;
                }
                __syncthreads();
                if (act) {
#pragma unroll 4
                    for (int jj = 0; jj < jn; ++jj) {
                        Cx<T> v0, v1, x[4];
                        ldcx2(as + jj * PF_LD + 2 * lane, v0, v1);
                        ldcx2(xs + jj * PF_LX + cw, x[0], x[1]);
                        ldcx2(xs + jj * PF_LX + cw + 2, x[2], x[3]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            cfmac(t[0][u], x[u], v0);
                            cfmac(t[1][u], x[u], v1);
                        }
                    }
                }
            }
            if (act) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int q = q0 + 2 * lane + e;
                    if (q < Q) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) ts[q * PF_LX + cw + u] = cmul(fs[pq[q]][cw + u], t[e][u]);
                    }
                }
            }
        }
        // ---- 2. z, 64 rows at a time ----
        for (int i0 = 0; i0 < M; i0 += 64) {
            Cx<T> z[2][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) z[0][u] = z[1][u] = Cx<T>{0, 0};
            for (int q0 = 0; q0 < Q; q0 += PF_JC) {
                const int qn = min(PF_JC, Q - q0);
                __syncthreads();
                for (int e = tid; e < PF_JC * 64; e += PF_NT) {
                    const int q = e >> 6, i = e & 63;
                    as[q * PF_LD + i] = q < qn && i0 + i < M ? ldcx(pool + uo[q0 + q] + i0 + i) : Cx<T>{0, 0};
                }
                __syncthreads();
                if (act) {
#pragma unroll 4
                    for (int q = 0; q < qn; ++q) {
                        Cx<T> a0, a1, t[4];
                        ldcx2(as + q * PF_LD + 2 * lane, a0, a1);
                        ldcx2(ts + (q0 + q) * PF_LX + cw, t[0], t[1]);
                        ldcx2(ts + (q0 + q) * PF_LX + cw + 2, t[2], t[3]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            cfma(z[0][u], a0, t[u]);
                            cfma(z[1][u], a1, t[u]);
                        }
                    }
                }
            }
            if (act) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int gc = c0 + cw + u;
                    if (gc >= nrhs) break;
                    Cx<T>* out = (gc < Ku ? yf + (long long)gc * E : yc + (long long)(gc - Ku) * E) + br.rb + i0 + 2 * lane;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        if (i0 + 2 * lane + e < M) {
                            atomicAdd(&out[e].x, z[e][u].x);
                            atomicAdd(&out[e].y, z[e][u].y);
                        }
                    }
                }
            }
        }
        pa = pb;
    }
}

// Y[perm p, uniq k] = yf[k][p];  Y[perm p, partner] = conj(yc[k][p]) (column-major M x K)
template <class T, class TO>
__global__ void k_pf_finish(int E, int Ku, const int* __restrict__ perm, const int* __restrict__ uniq,
                            const int* __restrict__ partner, const Cx<T>* __restrict__ yf,
                            const Cx<T>* __restrict__ yc, Cx<TO>* __restrict__ Y) {
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)Ku * E) return;
    const int k = (int)(idx / E), p = (int)(idx % E);
    const int l = uniq[k], lp = partner[l];
    const Cx<T> a = yf[idx];
    Y[(long long)l * E + perm[p]] = Cx<TO>{(TO)a.x, (TO)a.y};
    if (lp != l) {
        const Cx<T> b = yc[idx];
        Y[(long long)lp * E + perm[p]] = Cx<TO>{(TO)b.x, (TO)-b.y};
    }
}

template <class T>
static g3_status run_apply_perfreq_t(g3_ctx* ctx, const g3_tree* t, const g3_near* nf, const g3_factors* fa,
                                     const void* W, void* Y, int dtype, const g3_freqs* f) {
    const int E = t->ne, K = f->K, Ku = f->Ku;
    const size_t nW = (size_t)Ku * E;
    G3_CUDA(ctx->scratch.ensure(4 * nW * sizeof(Cx<T>)));
    Cx<T>* Wf = ctx->scratch.as<Cx<T>>();
    Cx<T>* Wc = Wf + nW;
    Cx<T>* yf = Wc + nW;
    Cx<T>* yc = yf + nW;
    cudaEvent_t e0 = ctx->ev[2], e3 = ctx->ev[5];
    G3_CUDA(cudaEventRecord(e0, ctx->stream));
    G3_CUDA(cudaMemsetAsync(yf, 0, 2 * nW * sizeof(Cx<T>), ctx->stream));
    {
        const int blocks = (int)((nW + 255) / 256);
        // k_apply_prep also clears its y argument: point it at yf (cleared anyway)
        if (dtype == G3_C128)
            k_apply_prep<double, T><<<blocks, 256, 0, ctx->stream>>>(E, K, Ku, t->d_perm.as<int>(), f->d_uniq.as<int>(),
                                                                   f->d_partner.as<int>(), (const Cx<double>*)W, Wf, Wc, yf, E);
        else
            k_apply_prep<float, T><<<blocks, 256, 0, ctx->stream>>>(E, K, Ku, t->d_perm.as<int>(), f->d_uniq.as<int>(),
                                                                  f->d_partner.as<int>(), (const Cx<float>*)W, Wf, Wc, yf, E);
        ctx->count("k_apply_prep");
        G3_CUDA(cudaGetLastError());
    }
    if (nf && !nf->order.empty()) {
        constexpr int NT = 256, KC = 16;
        dim3 grid((unsigned)nf->order.size(), (Ku + KC - 1) / KC);
        k_pf_near<T, NT><<<grid, NT, 0, ctx->stream>>>(nf->data.as<Cx<T>>(), nf->d_ranges.as<BlockRange>(),
                                                       nf->d_offs.as<long long>(), Ku, KC, E, Wf, Wc, yf, yc);
        ctx->count("k_pf_near");
        G3_CUDA(cudaGetLastError());
    }
    if (fa && fa->n_far > 0) {
        if (!fa->plan_ready) return fail(G3_EINVAL, "apply_gcq: factors without far-field work lists");
        const int nd = fa->plan_nd, nl = fa->plan_n1 + fa->plan_n2;
        const int4* it0 = fa->d_plan.as<int4>();
        const int4* it1 = it0 + nd;
        const BlockRange* d_ranges = fa->d_franges.as<BlockRange>();
        if (nd > 0) {
            const int nch = (Ku + PD_KC - 1) / PD_KC, kchunk = (Ku + nch - 1) / nch;
            const size_t smem = (size_t)FD_SL * ((kchunk + PD_KT - 1) / PD_KT * PD_KT) * sizeof(Cx<T>);
            k_pf_far_dense<T><<<dim3(nd, nch), PD_NT, smem, ctx->stream>>>(
                fa->pool->as<Cx<T>>(), fa->d_rec.as<CrossRec>(), d_ranges, it0, reinterpret_cast<const int2*>(it1 + nl),
                fa->Cmax, Ku, kchunk, E, Wf, Wc, yf, yc);
            ctx->count("k_pf_far_dense");
            G3_CUDA(cudaGetLastError());
        }
        if (nl > 0) {
            constexpr size_t smem = pf_lr_smem<T>();
            G3_CUDA(cudaFuncSetAttribute(k_pf_far_lr<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            k_pf_far_lr<T><<<dim3(nl, (2 * Ku + PF_NC - 1) / PF_NC), PF_NT, smem, ctx->stream>>>(
                fa->pool->as<Cx<T>>(), fa->d_rec.as<CrossRec>(), fa->d_r3.as<int>(), d_ranges, it1, fa->Cmax, Ku, E, Wf,
                Wc, yf, yc);
            ctx->count("k_pf_far_lr");
            G3_CUDA(cudaGetLastError());
        }
    }
    {
        const int blocks = (int)((nW + 255) / 256);
        if (dtype == G3_C128)
            k_pf_finish<T, double><<<blocks, 256, 0, ctx->stream>>>(E, Ku, t->d_perm.as<int>(), f->d_uniq.as<int>(),
                                                                  f->d_partner.as<int>(), yf, yc, (Cx<double>*)Y);
        else
            k_pf_finish<T, float><<<blocks, 256, 0, ctx->stream>>>(E, Ku, t->d_perm.as<int>(), f->d_uniq.as<int>(),
                                                                 f->d_partner.as<int>(), yf, yc, (Cx<float>*)Y);
        ctx->count("k_pf_finish");
        G3_CUDA(cudaGetLastError());
    }
    G3_CUDA(cudaEventRecord(e3, ctx->stream));
    G3_CUDA(cudaEventSynchronize(e3));
    float ms_all = 0;
    G3_CUDA(cudaEventElapsedTime(&ms_all, e0, e3));
    ctx->last_apply_ms = ms_all;
    ctx->last_near_ms = 0;
    const int64_t in_sz = dtype == G3_C128 ? 16 : 8;
    const int64_t near_bytes = nf ? nf->n_entries * (int64_t)sizeof(Cx<T>) : 0;
    ctx->last_near_bytes = near_bytes;
    ctx->last_apply_bytes = near_bytes + (fa ? fa->stats.factor_bytes : 0) + 2 * (int64_t)E * K * in_sz;
    return G3_OK;
}

// ============================================================================
// Allocation-free apply
// ============================================================================
//
// Some callers cannot allocate device memory while they run this step: code
// inside a memory-capped or pre-reserved arena, a runtime that forbids
// cudaMalloc on its hot path, or a host that must not synchronise the device
// (cudaMalloc/cudaFree can).  apply_gcq_noalloc serves them: it computes the
// same sum as apply_gcq (device buffers, G3_APPLY_SUM) with its scratch in the
// fixed array below instead of the context's growable buffer, and calls no
// allocating routine.
//
// The array is a file-scope __device__ object: every GPU that loads this
// library holds it until the process exits.  All calls on a device share it
// and it keeps the last call's contents, so every part a call reads is
// written first by that call (the accumulator is cleared by k_apply_prep).
// Calls whose work overlaps on the GPU (several streams or threads at once)
// race on it and must be serialised by the caller.
constexpr size_t NOALLOC_SCRATCH_BYTES = 32ull << 20;  // 32 MiB
static __device__ __align__(256) unsigned char g3_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

// device address of the scratch array, looked up once per device (with that
// device current); host code must not use the symbol itself as an address
static void* g_noalloc_ptr[64] = {};

static g3_status noalloc_scratch(int device, void** out) {
    if (device < 0 || device >= 64) return fail(G3_EINVAL, "apply_gcq_noalloc: device %d not supported", device);
    if (!g_noalloc_ptr[device]) {
        void* ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g3_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g3_noalloc_scratch)");
        g_noalloc_ptr[device] = ptr;
    }
    *out = g_noalloc_ptr[device];
    return G3_OK;
}


template <class T>
static g3_status run_apply_noalloc_t(g3_ctx* ctx, const g3_tree* t, const g3_near* nf, const g3_factors* fa,
                                     const void* W, void* Y, int dtype, const g3_freqs* f) {
    const int E = t->ne, Ku = f->Ku;
    const int n_far = fa ? fa->n_far : 0;
    const size_t nW = (size_t)Ku * E;
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t need = al(nW * sizeof(WPair<T>)) + al(E * sizeof(Cx<T>));
    if (need > NOALLOC_SCRATCH_BYTES)
        return fail(G3_EINVAL,
                    "apply_gcq_noalloc: this problem needs %zu bytes of scratch (2 Ku E + E complex values), "
                    "the fixed scratch holds %zu; use apply_gcq",
                    need, NOALLOC_SCRATCH_BYTES);
    void* base = nullptr;
    G3_TRY_NA(noalloc_scratch(ctx->device, &base));
    WPair<T>* Wp = static_cast<WPair<T>*>(base);
    Cx<T>* y = reinterpret_cast<Cx<T>*>(static_cast<char*>(base) + al(nW * sizeof(WPair<T>)));
    G3_TRY_NA(launch_prep_pm<T>(ctx, E, f, t->d_perm.as<int>(), W, dtype, Wp, y, E));
    G3_TRY_NA(apply_near_far<T>(ctx, t, nf, n_far > 0 ? fa : nullptr, Ku, E, Wp, y));
    {
        int blocks = (E + 255) / 256;
        if (dtype == G3_C128)
            k_apply_finish<T, double><<<blocks, 256, 0, ctx->stream>>>(E, t->d_perm.as<int>(), y, (Cx<double>*)Y);
        else
            k_apply_finish<T, float><<<blocks, 256, 0, ctx->stream>>>(E, t->d_perm.as<int>(), y, (Cx<float>*)Y);
        ctx->count("k_apply_finish");
        G3_CUDA(cudaGetLastError());
    }
    return G3_OK;
}

g3_status run_apply(g3_ctx* ctx, const g3_tree* t, const g3_near* nf, const g3_factors* fa, const void* W, void* Y,
                    int dtype, int mode) {
    const g3_freqs* f = nf ? nf->freqs : fa->freqs;
    const int prec = nf ? nf->prec : fa->prec;
    if (nf && fa && (nf->prec != fa->prec || nf->freqs != fa->freqs))
        return fail(G3_EINVAL, "apply_gcq: near field and factors differ in precision or frequency set");
    if (mode == G3_APPLY_PERFREQ) {
        if (prec == G3_MIXED) return run_apply_perfreq_t<float>(ctx, t, nf, fa, W, Y, dtype, f);
        return run_apply_perfreq_t<double>(ctx, t, nf, fa, W, Y, dtype, f);
    }
    if (prec == G3_MIXED) return run_apply_t<float>(ctx, t, nf, fa, W, Y, dtype, f);
    return run_apply_t<double>(ctx, t, nf, fa, W, Y, dtype, f);
}

}  // namespace g3

extern "C" g3_status apply_gcq_noalloc(g3_ctx* ctx, const g3_tree* t, const g3_near* nf, const g3_factors* fa,
                                       const void* W, void* Y, g3_dtype dtype) {
    using namespace g3;
    if (!ctx || !t || !W || !Y) return fail(G3_EINVAL, "apply_gcq_noalloc: NULL argument");
    if (t->p1) return fail(G3_EUNSUPPORTED, "apply_gcq_noalloc: linear-element trees use apply_gcq");
    if (!nf && !fa) return fail(G3_EINVAL, "apply_gcq_noalloc: near field and factors are both NULL");
    if (dtype != G3_C64 && dtype != G3_C128) return fail(G3_EINVAL, "apply_gcq_noalloc: bad dtype");
    if ((nf && nf->tree != t) || (fa && fa->tree != t))
        return fail(G3_EINVAL, "apply_gcq_noalloc: near field or factors built on another tree");
    if (nf && fa && (nf->prec != fa->prec || nf->freqs != fa->freqs))
        return fail(G3_EINVAL, "apply_gcq_noalloc: near field and factors differ in precision or frequency set");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    const g3_freqs* f = nf ? nf->freqs : fa->freqs;
    const int prec = nf ? nf->prec : fa->prec;
    if (prec == G3_MIXED) return run_apply_noalloc_t<float>(ctx, t, nf, fa, W, Y, dtype, f);
    return run_apply_noalloc_t<double>(ctx, t, nf, fa, W, Y, dtype, f);
}
