// Differentiation of the solver's outputs.
//
//  * Gradients of the smooth loss L(Omega, X) = -sum log w_ii + tr(Omega S Omega)/2
//    + lambda2/2 ||Omega||_F^2, S = X^T X / n, at the (symmetric) iterate:
//      dL/dOmega = -diag(1/w_ii) + (Omega S + S Omega)/2 + lambda2 Omega   (Alg. 1 step 4's G, dense)
//      dL/dX     = X Omega^2 / n = Y Omega / n,  Y = X Omega.
//    dL/dOmega is one kernel over pairs of tiles (I <= J): W[I, J] and W[J, I] in
//    the screening pass's canonical FMA order (so G agrees bitwise with the solver's
//    G on its candidates), symmetrised, with the support terms, written once.
//    X Omega^2 / n is two row-split SpMMs on X^T, the second writing its result
//    transposed.
//  * The implicit lambda-gradient of a held-out loss on the support A: the
//    support-restricted products (E S)_ij by gathers, the Hessian-vector product
//      H[E]_ij = ((E S)_ij + (E S)_ji)/2 + lambda2 E_ij + [i=j] E_ii / w_ii^2,
//    and conjugate gradients in FP64 with fixed-order reductions (the vectors
//    live on the nnz entries of A, so FP64 costs little there).  The held-out
//    loss's gradient needs (Omega S_val)_ij on A only: a row-split SpMM
//    Y^T = Omega X_val^T and one dot product of rows of Y^T and X_val^T per entry,
//    so S_val (p x p) is never formed.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.cuh"

namespace hpc {
namespace {

constexpr int kW = 8;   // warps per block

__device__ __forceinline__ float fmaT(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mulT(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulT(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

template <typename TO, typename TI>
__device__ __forceinline__ TO to_t(TI v) { return (TO)v; }
template <>
__device__ __forceinline__ float to_t<float, __nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ double to_t<double, __nv_bfloat16>(__nv_bfloat16 v) {
    return (double)__bfloat162float(v);
}

// C[i, c] = sum_k w_ik B[k, c], canonical order: w_ii B[i, c] first, then the
// off-diagonal k ascending.  Warp per row, lanes over 32 * 4 consecutive columns.
template <typename T>
__global__ void __launch_bounds__(256)
k_spmm_dense(int p, Csr<T> om, const int4* __restrict__ rinfo, const T* __restrict__ rdv, const T* __restrict__ B,
             int64_t ldb, int64_t m, T* __restrict__ C, int64_t ldc) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kW + (threadIdx.x >> 5);
    if (i >= p) return;
    const int64_t c0 = (int64_t)blockIdx.y * 128;
    const int4 info = rinfo[i];
    const T dv = rdv[i];
    T acc[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int64_t c = c0 + lane + 32 * v;
        acc[v] = c < m ? mulT(dv, B[(int64_t)i * ldb + c]) : T(0);
    }
    for (int q = info.x; q < info.y; ++q) {
        if (q == info.z) continue;
        const int k = om.ci[q];
        const T w = om.cv[q];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t c = c0 + lane + 32 * v;
            if (c < m) acc[v] = fmaT(w, B[(int64_t)k * ldb + c], acc[v]);
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int64_t c = c0 + lane + 32 * v;
        if (c < m) C[(int64_t)i * ldc + c] = acc[v];
    }
}

// C^T scaled: C = Omega B as in k_spmm_dense (same order per element), for a tile of 32
// rows i x 128 columns c staged in shared memory, then written as Ct[c, i] = scale C[i, c]
// (Ct m x p, row pitch ldt), so a transpose never re-reads C.
template <typename T>
__global__ void __launch_bounds__(256)
k_spmm_dense_t(int p, Csr<T> om, const int4* __restrict__ rinfo, const T* __restrict__ rdv, const T* __restrict__ B,
               int64_t ldb, int64_t m, T* __restrict__ Ct, int64_t ldt, T scale) {
    __shared__ T tile[32][129];
    const int lane = threadIdx.x & 31;
    const int i0 = blockIdx.x * 32;
    const int64_t c0 = (int64_t)blockIdx.y * 128;
    for (int y = threadIdx.x >> 5; y < 32; y += kW) {
        const int i = i0 + y;
        T acc[4] = {T(0), T(0), T(0), T(0)};
        if (i < p) {
            const int4 info = rinfo[i];
            const T dv = rdv[i];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int64_t c = c0 + lane + 32 * v;
                acc[v] = c < m ? mulT(dv, B[(int64_t)i * ldb + c]) : T(0);
            }
            for (int q = info.x; q < info.y; ++q) {
                if (q == info.z) continue;
                const int k = om.ci[q];
                const T w = om.cv[q];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int64_t c = c0 + lane + 32 * v;
                    if (c < m) acc[v] = fmaT(w, B[(int64_t)k * ldb + c], acc[v]);
                }
            }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) tile[y][lane + 32 * v] = acc[v];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < 32 * 128; idx += 256) {
        const int cl = idx >> 5, il = idx & 31;
        const int64_t c = c0 + cl;
        if (c < m && i0 + il < p) Ct[c * ldt + i0 + il] = tile[il][cl] * scale;
    }
}

// The off-diagonal terms of row i of W = Omega S on the columns c0 .. c0 + TL - 1, added to
// w (which holds w_ii S_ic) in k_spmm_dense's order: k ascending, the diagonal skipped.
// One warp; the row's (k, w_ik) come in 32 at a time, one per lane, broadcast by
// shuffles; S[k, c] is gathered from global memory.
template <typename T, int TL>
__device__ __forceinline__ void offdiag_row(int p, const Csr<T>& om, int4 info, const T* __restrict__ S, int64_t lds,
                                            int c0, T* w) {
    constexpr int V = TL / 32;
    const int lane = threadIdx.x & 31;
    T acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = w[lane + 32 * v];
    for (int q0 = info.x; q0 < info.y; q0 += 32) {
        const int ql = q0 + lane;
        const int kl = ql < info.y ? om.ci[ql] : 0;
        const T wl = ql < info.y ? om.cv[ql] : T(0);
        const int cnt = min(32, info.y - q0);
#pragma unroll 4
        for (int t = 0; t < cnt; ++t) {
            const int k = __shfl_sync(kFull, kl, t);
            const T wk = __shfl_sync(kFull, wl, t);
            if (q0 + t == info.z) continue;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int c = c0 + lane + 32 * v;
                if (c < p) acc[v] = fmaT(wk, S[(int64_t)k * lds + c], acc[v]);
            }
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) w[lane + 32 * v] = acc[v];
}

// The support terms of G in row i on the columns c0 .. c0 + TL - 1 (one warp):
// g_ij <- fma(lambda2, w_ij, g_ij) - [i=j] / w_ii.
template <typename T, int TL>
__device__ __forceinline__ void support_terms_row(const Csr<T>& om, int i, int c0, T lam2, T* g) {
    const int lane = threadIdx.x & 31;
    for (int q = om.rp[i] + lane; q < om.rp[i + 1]; q += 32) {
        const int j = om.ci[q];
        if (j < c0 || j >= c0 + TL) continue;
        const T wv = om.cv[q];
        T v = fmaT(lam2, wv, g[j - c0]);
        if (j == i) v -= T(1) / wv;
        g[j - c0] = v;
    }
}

// 16 bytes of T for one vector store
template <typename T> struct Vec16;
template <> struct Vec16<float> {
    using type = float4;
    static __device__ __forceinline__ float4 make(const float* v) { return make_float4(v[0], v[1], v[2], v[3]); }
    static __device__ __forceinline__ void unpack(const float4& u, float* v) {
        v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
    }
};
template <> struct Vec16<double> {
    using type = double2;
    static __device__ __forceinline__ double2 make(const double* v) { return make_double2(v[0], v[1]); }
    static __device__ __forceinline__ void unpack(const double2& u, double* v) { v[0] = u.x; v[1] = u.y; }
};

// Row and column block (bi <= bj) of the t-th tile pair, pairs numbered row by row
// (row bi holds nt - bi pairs): bi from the quadratic's root in FP32, then corrected
// by exact integer steps.
__device__ __forceinline__ void pair_of(long long t, int nt, int& bi, int& bj) {
    const float b2 = 2.0f * (float)nt + 1.0f;
    int r = (int)((b2 - sqrtf(fmaxf(b2 * b2 - 8.0f * (float)t, 0.0f))) * 0.5f);
    r = max(0, min(r, nt - 1));
    auto start = [&](long long q) { return q * nt - q * (q - 1) / 2; };
    while (r > 0 && start(r) > t) --r;
    while (r + 1 < nt && start(r + 1) <= t) ++r;
    bi = r;
    bj = r + (int)(t - start(r));
}

// dL/dOmega = scale ((W + W^T)/2 + lambda2 Omega - diag(1/w_ii)), W = Omega S, on one pair
// of TL x TL tiles (I <= J) per CTA, so G is written once and never re-read:
//  0. the off-diagonal entries (k, w_ik) of the rows of I and J go into a list in shared memory,
//     row by row; the first S segments that they need are requested at once;
//  1. the tile S[I, J] is read once; it gives the diagonal terms of both W[I, J]
//     (w_ii S_ij) and W[J, I] (w_jj S_ji = w_jj S_ij: S is bitwise symmetric);
//  2. the list's terms w_ik S[k, J] are added, k ascending: a group of TL / 4 (FP64: TL / 2)
//     lanes per row, 16 bytes a lane, kAhead entries of the group's rows in flight;
//  3. G[I, J] = (W[I, J] + W[J, I]^T)/2 and its transpose, by the thread that holds both
//     entries; then the support terms, a thread per list entry, the scale, and 16-byte stores.
// The rounding sequence per element is the solver's (W in the canonical order,
// 0.5 (W_ij + W_ji), the support terms, the scale).
//
// What bounds it: memory (S[I, J], the S rows of the neighbours, both halves of G), as long as
// enough of it is asked for at once.  With a warp per row that went from the row's bounds to its
// entries to S, one row after the other, the rows with neighbours were a chain of three
// latencies each, about nine of them per warp where half of the rows have neighbours.
// Measured on GB300, p = 16384, 28 672 entries (half of the rows with neighbours): 770 -> 572 us.
// Rows with more than kGradList entries in all come in one list after another (their support terms
// a warp per row).  With a warp per row for such tile pairs, hub rows took longer: 4000 entries
// at p = 4096 4.8 ms, 3.9 now, 8000 at p = 16384 11.3, 8.4.
constexpr int kGradList = 512;
constexpr int kAhead = 4;

template <typename T, int TL>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 3)
k_dense_grad_pair(int p, Csr<T> om, const int4* __restrict__ rinfo, const T* __restrict__ rdv,
                  const T* __restrict__ S, int64_t lds, T* __restrict__ G, int64_t ldg, T lam2, T scale, int nt,
                  int vec /* bit 0: 16-byte G stores; bit 1: 16-byte S loads */) {
    __shared__ T a[TL][TL + 1];      // W[I, J], then G[I, J]
    __shared__ T b[TL][TL + 1];      // W[J, I], then G[J, I]
    __shared__ T dvs[2 * TL];        // w_ii of the rows of I, then of J
    __shared__ int off[2 * TL + 1];  // first entry of each row, all rows' entries in one sequence
    __shared__ int2 rbd[2 * TL];     // its CSR position, that of its diagonal (-1: none)
    __shared__ int lk[kGradList];    // list: column k, w_ik, the entry's row (0 .. 2 TL - 1)
    __shared__ T lw[kGradList];
    __shared__ unsigned char lr[kGradList];
    __shared__ int wsum[2 * TL / 32];
    constexpr int E = TL * TL / 256;
    static_assert(2 * TL <= 256, "a row per thread");
    int bi, bj;
    pair_of(blockIdx.x, nt, bi, bj);
    const int I0 = bi * TL, J0 = bj * TL;
    const bool dtile = bi == bj;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int VW = 16 / (int)sizeof(T), PR = TL / VW, EV = TL * PR / 256;   // 16-byte vectors
    using V16 = Vec16<T>;
    const bool full = I0 + TL <= p && J0 + TL <= p;
    const bool vload = (vec & 2) && full;
    typename V16::type tile[EV];             // S[I, J], asked for before anything else
    if (vload) {
#pragma unroll
        for (int e = 0; e < EV; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / PR, x = (idx % PR) * VW;
            tile[e] = *reinterpret_cast<const typename V16::type*>(S + (int64_t)(I0 + y) * lds + J0 + x);
        }
    }
    // 0. the list
    int4 info = make_int4(0, 0, -1, 1);
    int cnt = 0, incl = 0;
    const int row0 = (int)threadIdx.x < TL ? I0 + (int)threadIdx.x : J0 + (int)threadIdx.x - TL;
    if (threadIdx.x < 2 * TL) {
        T dv = T(0);
        if (row0 < p) {
            dv = rdv[row0];
            info = rinfo[row0];
            cnt = info.y - info.x - (info.z >= 0 ? 1 : 0);
        }
        dvs[threadIdx.x] = dv;
        rbd[threadIdx.x] = make_int2(info.x, info.z);
        incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
    }
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int w = 0; w < 2 * TL / 32; ++w) {
        if (w < warp) incl += wsum[w];
        total += wsum[w];
    }
    if (threadIdx.x < 2 * TL) {
        off[threadIdx.x] = incl - cnt;
        if (threadIdx.x == 2 * TL - 1) off[2 * TL] = total;
    }
    __syncthreads();
    // entries w0 .. of the sequence into the list, a thread each
    int w0 = 0, w1 = min(total, kGradList);
    auto fill = [&]() {
        for (int e = w0 + (int)threadIdx.x; e < w1; e += 256) {
            int lo = 0, hi = 2 * TL - 1;             // the last row that starts at or before e
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (off[mid] <= e) lo = mid; else hi = mid - 1;
            }
            int q = rbd[lo].x + e - off[lo];
            if (rbd[lo].y >= 0 && q >= rbd[lo].y) ++q;
            lk[e - w0] = om.ci[q];
            lw[e - w0] = om.cv[q];
            lr[e - w0] = (unsigned char)lo;
        }
    };
    fill();
    __syncthreads();
    // the group's cursor over the listed entries of its rows (grp, grp + 256 / PR, ..)
    const int grp = threadIdx.x / PR, gl = (threadIdx.x % PR) * VW;
    constexpr int NG = 256 / PR;
    int r = grp - NG, t = 0, end = 0;
    auto next = [&]() -> int {               // the next entry, -1 at the end
        while (t == end) {
            r += NG;
            if (r >= 2 * TL) return -1;
            t = max(off[r], w0);
            end = max(t, min(off[r + 1], w1));
        }
        return t++ - w0;
    };
    auto fetch = [&](int e) -> typename V16::type {
        const T* src = S + (int64_t)lk[e] * lds + (lr[e] < TL ? J0 : I0) + gl;
        if (vload) return *reinterpret_cast<const typename V16::type*>(src);
        T v[VW];
        const int c = (lr[e] < TL ? J0 : I0) + gl;
#pragma unroll
        for (int x = 0; x < VW; ++x) v[x] = c + x < p ? src[x] : T(0);
        return V16::make(v);
    };
    int ent[kAhead];
    typename V16::type sv4[kAhead];
    auto ahead = [&]() {
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            ent[u] = r < 2 * TL ? next() : -1;
            if (ent[u] >= 0) sv4[u] = fetch(ent[u]);
        }
    };
    ahead();
    // 1. diagonal terms of both tiles from one read of S[I, J]
    if (vload) {
#pragma unroll
        for (int e = 0; e < EV; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / PR, x = (idx % PR) * VW;
            T sv[VW];
            V16::unpack(tile[e], sv);
#pragma unroll
            for (int k = 0; k < VW; ++k) {
                a[y][x + k] = mulT(dvs[y], sv[k]);
                b[x + k][y] = mulT(dvs[TL + x + k], sv[k]);
            }
        }
    } else {
#pragma unroll 4
        for (int e = 0; e < E; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / TL, x = idx % TL;
            const T sv = (I0 + y < p && J0 + x < p) ? S[(int64_t)(I0 + y) * lds + J0 + x] : T(0);
            a[y][x] = mulT(dvs[y], sv);
            b[x][y] = mulT(dvs[TL + x], sv);
        }
    }
    __syncthreads();
    // 2. off-diagonal terms of the rows that have them, a list after another
    for (;;) {
        while (ent[0] >= 0) {
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                if (ent[u] < 0) break;
                const int row = lr[ent[u]];
                T* w = row < TL ? &a[row][gl] : &b[row - TL][gl];
                const T wk = lw[ent[u]];
                T sv[VW];
                V16::unpack(sv4[u], sv);
#pragma unroll
                for (int x = 0; x < VW; ++x) w[x] = fmaT(wk, sv[x], w[x]);
            }
            ahead();
        }
        if (w1 == total) break;
        __syncthreads();
        w0 = w1;
        w1 = min(total, w0 + kGradList);
        fill();
        __syncthreads();
        r = grp - NG;
        t = end = 0;
        ahead();
    }
    const bool listed = total <= kGradList;
    __syncthreads();
    // 3. symmetrise: G[I, J] and its transpose (a + b = b + a)
#pragma unroll 4
    for (int e = 0; e < E; ++e) {
        const int idx = threadIdx.x + 256 * e, y = idx / TL, x = idx % TL;
        const T g = T(0.5) * (a[y][x] + b[x][y]);
        a[y][x] = g;
        b[x][y] = g;
    }
    __syncthreads();
    if (dtile) {
        // the diagonal tile: every row has its diagonal entry here
        for (int y = warp; y < TL && I0 + y < p; y += kW) support_terms_row<T, TL>(om, I0 + y, I0, lam2, &a[y][0]);
    } else if (listed) {
        for (int e = threadIdx.x; e < total; e += 256) {
            const int row = lr[e], c = lk[e] - (row < TL ? J0 : I0);
            if (c < 0 || c >= TL) continue;
            T* g = row < TL ? &a[row][c] : &b[row - TL][c];
            *g = fmaT(lam2, lw[e], *g);
        }
    } else {
        for (int row = warp; row < 2 * TL; row += kW) {
            if (off[row] == off[row + 1]) continue;
            support_terms_row<T, TL>(om, row < TL ? I0 + row : J0 + row - TL, row < TL ? J0 : I0, lam2,
                                     row < TL ? &a[row][0] : &b[row - TL][0]);
        }
    }
    __syncthreads();
    const bool scaled = scale != T(1);
    if ((vec & 1) && full) {
        for (int idx = threadIdx.x; idx < TL * PR; idx += 256) {
            const int y = idx / PR, x = (idx % PR) * VW;
            T va[VW], vb[VW];
#pragma unroll
            for (int k = 0; k < VW; ++k) {
                va[k] = scaled ? a[y][x + k] * scale : a[y][x + k];
                vb[k] = scaled ? b[y][x + k] * scale : b[y][x + k];
            }
            *reinterpret_cast<typename V16::type*>(G + (int64_t)(I0 + y) * ldg + J0 + x) = V16::make(va);
            if (!dtile) *reinterpret_cast<typename V16::type*>(G + (int64_t)(J0 + y) * ldg + I0 + x) = V16::make(vb);
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / TL, x = idx % TL;
            if (I0 + y < p && J0 + x < p) {
                const T v = a[y][x];
                G[(int64_t)(I0 + y) * ldg + J0 + x] = scaled ? v * scale : v;
            }
            if (!dtile && J0 + y < p && I0 + x < p) {
                const T v = b[y][x];
                G[(int64_t)(J0 + y) * ldg + I0 + x] = scaled ? v * scale : v;
            }
        }
    }
}

// The same for wide rows: a warp per row with neighbours, without a list.  With many entries in
// every row the warps have enough of them in flight by themselves, the list's rounds only cost
// (kGradList entries are a few rows' then), and the room in shared memory is a sixth block per SM.
// The line, four neighbours per row (FP64: eight), is where a tile pair's rows fill one list.
// Measured on GB300, ms, list rounds and this: p = 16384, 20 entries a row 5.53, 5.68; p = 4096, 20 a
// row 0.45, 0.41; 200 a row 7.05, 2.69.
template <typename T, int TL>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 6 : 3)
k_dense_grad_rows(int p, Csr<T> om, const int4* __restrict__ rinfo, const T* __restrict__ rdv,
                  const T* __restrict__ S, int64_t lds, T* __restrict__ G, int64_t ldg, T lam2, T scale, int nt,
                  int vec /* bit 0: 16-byte G stores; bit 1: 16-byte S loads */) {
    __shared__ T a[TL][TL + 1];      // W[I, J], then G[I, J]
    __shared__ T b[TL][TL + 1];      // W[J, I], then G[J, I]
    __shared__ T dvs[2][TL];         // w_ii of the rows of I and of J
    __shared__ int imp[2][TL];       // rows of I and of J with off-diagonal entries
    __shared__ int nimp[2];
    constexpr int E = TL * TL / 256;
    int bi, bj;
    pair_of(blockIdx.x, nt, bi, bj);
    const int I0 = bi * TL, J0 = bj * TL;
    const bool dtile = bi == bj;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 2) nimp[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x < 2 * TL) {
        const int side = threadIdx.x / TL, yl = threadIdx.x % TL;
        const int i = (side ? J0 : I0) + yl;
        T dv = T(0);
        bool impure = false;
        if (i < p) {
            dv = rdv[i];
            impure = rinfo[i].w == 0;
        }
        dvs[side][yl] = dv;
        if (impure) imp[side][atomicAdd(&nimp[side], 1)] = yl;
    }
    __syncthreads();
    // 1. diagonal terms of both tiles from one read of S[I, J]
    constexpr int VW = 16 / (int)sizeof(T), PR = TL / VW, EV = TL * PR / 256;   // 16-byte vectors
    using V16 = Vec16<T>;
    const bool full = I0 + TL <= p && J0 + TL <= p;
    if ((vec & 2) && full) {
        typename V16::type u[EV];
#pragma unroll
        for (int e = 0; e < EV; ++e) {           // all the tile's loads in flight before any use
            const int idx = threadIdx.x + 256 * e, y = idx / PR, x = (idx % PR) * VW;
            u[e] = *reinterpret_cast<const typename V16::type*>(S + (int64_t)(I0 + y) * lds + J0 + x);
        }
#pragma unroll
        for (int e = 0; e < EV; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / PR, x = (idx % PR) * VW;
            T sv[VW];
            V16::unpack(u[e], sv);
#pragma unroll
            for (int k = 0; k < VW; ++k) {
                a[y][x + k] = mulT(dvs[0][y], sv[k]);
                b[x + k][y] = mulT(dvs[1][x + k], sv[k]);
            }
        }
    } else {
#pragma unroll 4
        for (int e = 0; e < E; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / TL, x = idx % TL;
            const T sv = (I0 + y < p && J0 + x < p) ? S[(int64_t)(I0 + y) * lds + J0 + x] : T(0);
            a[y][x] = mulT(dvs[0][y], sv);
            b[x][y] = mulT(dvs[1][x], sv);
        }
    }
    __syncthreads();
    // 2. off-diagonal terms of the rows that have them
    const int n0 = nimp[0], n1 = nimp[1];
    for (int r = warp; r < n0 + n1; r += kW) {
        const int side = r < n0 ? 0 : 1;
        const int yl = side ? imp[1][r - n0] : imp[0][r];
        const int i = (side ? J0 : I0) + yl;
        offdiag_row<T, TL>(p, om, rinfo[i], S, lds, side ? I0 : J0, side ? &b[yl][0] : &a[yl][0]);
    }
    __syncthreads();
    // 3. symmetrise: G[I, J] in place; G[J, I] is its transpose (a + b = b + a)
#pragma unroll 4
    for (int e = 0; e < E; ++e) {
        const int idx = threadIdx.x + 256 * e, y = idx / TL, x = idx % TL;
        a[y][x] = T(0.5) * (a[y][x] + b[x][y]);
    }
    __syncthreads();
    if (!dtile) {
#pragma unroll 4
        for (int e = 0; e < E; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / TL, x = idx % TL;
            b[y][x] = a[x][y];
        }
        __syncthreads();
        for (int r = warp; r < n0 + n1; r += kW) {
            const int side = r < n0 ? 0 : 1;
            const int yl = side ? imp[1][r - n0] : imp[0][r];
            support_terms_row<T, TL>(om, (side ? J0 : I0) + yl, side ? I0 : J0, lam2, side ? &b[yl][0] : &a[yl][0]);
        }
    } else {
        // the diagonal tile: every row has its diagonal entry here
        for (int y = warp; y < TL && I0 + y < p; y += kW) support_terms_row<T, TL>(om, I0 + y, I0, lam2, &a[y][0]);
    }
    __syncthreads();
    const bool scaled = scale != T(1);
    if ((vec & 1) && full) {
        for (int idx = threadIdx.x; idx < TL * PR; idx += 256) {
            const int y = idx / PR, x = (idx % PR) * VW;
            T va[VW], vb[VW];
#pragma unroll
            for (int k = 0; k < VW; ++k) {
                va[k] = scaled ? a[y][x + k] * scale : a[y][x + k];
                vb[k] = scaled ? b[y][x + k] * scale : b[y][x + k];
            }
            *reinterpret_cast<typename V16::type*>(G + (int64_t)(I0 + y) * ldg + J0 + x) = V16::make(va);
            if (!dtile) *reinterpret_cast<typename V16::type*>(G + (int64_t)(J0 + y) * ldg + I0 + x) = V16::make(vb);
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int idx = threadIdx.x + 256 * e, y = idx / TL, x = idx % TL;
            if (I0 + y < p && J0 + x < p) {
                const T v = a[y][x];
                G[(int64_t)(I0 + y) * ldg + J0 + x] = scaled ? v * scale : v;
            }
            if (!dtile && J0 + y < p && I0 + x < p) {
                const T v = b[y][x];
                G[(int64_t)(J0 + y) * ldg + I0 + x] = scaled ? v * scale : v;
            }
        }
    }
}

// out[c][r] = in[r][c] * scale, 64 x 64 shared-memory tiles held in the output type
// (an FP64 transpose stays FP64); columns rows .. rows_out - 1 of out are set to 0.
// What bounds it: memory, once enough loads are in flight: each thread has 16 of them (with
// 32 x 32 tiles it had four).  Measured on GB300, 4096 x 16384 FP32: 174 -> 79 us.
template <typename TI, typename TO>
__global__ void __launch_bounds__(256)
k_transpose(const TI* __restrict__ in, int64_t rows, int64_t cols, int64_t ldi, TO* __restrict__ out, int64_t ldo,
            int64_t rows_out, double scale) {
    __shared__ TO tile[64][65];
    const TO sc = (TO)scale;
    const int64_t r0 = (int64_t)blockIdx.y * 64, c0 = (int64_t)blockIdx.x * 64;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    TO v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        const int64_t r = r0 + ty + 8 * (u >> 1), c = c0 + tx + 32 * (u & 1);
        v[u] = (r < rows && c < cols) ? to_t<TO>(in[r * ldi + c]) : TO(0);
    }
#pragma unroll
    for (int u = 0; u < 16; ++u) tile[ty + 8 * (u >> 1)][tx + 32 * (u & 1)] = v[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        const int y = ty + 8 * (u >> 1), x = tx + 32 * (u & 1);
        const int64_t c = c0 + y, r = r0 + x;
        if (c < cols && r < rows_out) out[c * ldo + r] = tile[x][y] * sc;
    }
}

// tr[e] = position of entry (j, i) for entry e = (i, j) of a symmetric CSR (-1 if absent),
// and row[e] = i.
template <typename T>
__global__ void k_transpose_index(int p, Csr<T> om, int* __restrict__ tr, int* __restrict__ row) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kW + (threadIdx.x >> 5);
    if (i >= p) return;
    for (int e = om.rp[i] + lane; e < om.rp[i + 1]; e += 32) {
        const int j = om.ci[e];
        int lo = om.rp[j], hi = om.rp[j + 1] - 1, pos = -1;
        while (lo <= hi) {
            const int mid = (lo + hi) >> 1;
            const int c = om.ci[mid];
            if (c == i) { pos = mid; break; }
            if (c < i) lo = mid + 1; else hi = mid - 1;
        }
        tr[e] = pos;
        row[e] = i;
    }
}

// T_e = sum_{q in row i} v_q S[ci[q], j_e] for every support entry e = (i, j_e), FP64,
// diagonal term first then off-diagonals ascending.
template <typename T>
__global__ void k_support_product(int p, Csr<T> om, const int4* __restrict__ rinfo, const double* __restrict__ v,
                                  const T* __restrict__ S, int64_t lds, double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kW + (threadIdx.x >> 5);
    if (i >= p) return;
    const int4 info = rinfo[i];
    for (int e = info.x + lane; e < info.y; e += 32) {
        const int j = om.ci[e];
        double acc = info.z >= 0 ? v[info.z] * (double)S[(int64_t)i * lds + j] : 0.0;
        for (int q = info.x; q < info.y; ++q)
            if (q != info.z) acc = fma(v[q], (double)S[(int64_t)om.ci[q] * lds + j], acc);
        out[e] = acc;
    }
}

// T_e = (1/n) sum_m (Omega X^T)[i, m] X^T[j_e, m] for every support entry e = (i, j_e): the
// support-restricted (Omega S)_ij with S = X^T X / n, without S and without storing Omega X^T.
// A block per row i, kXyCols samples at a time: the row's Y = Omega X^T (k_spmm_dense's order)
// stays in registers, and the rows of X^T that made it are what its entries need next, from L1.
// 16-byte loads: ld is a multiple of 16 bytes and the columns from n to ld are 0.  Partials in T
// per thread (16 products), summed over the block and the pieces in FP64 in a fixed order.
// What bounds it: memory (the rows of X^T, 1 + the row's neighbours times).  As two kernels, Y^T
// was written and read back, and a warp per row went through its entries one after the other.
// Measured on GB300, p = 16384, n = 2048, 28 672 entries: 159 (55 + 104) -> 56 us.
constexpr int kXyT = 128;
constexpr int kXyCols = 16 * kXyT;
constexpr int kXyBatch = 16;

template <typename T>
__global__ void __launch_bounds__(kXyT)
k_support_xy(int p, Csr<T> om, const int4* __restrict__ rinfo, const T* __restrict__ rdv, const T* __restrict__ xt,
             int64_t ld, int64_t n, double* __restrict__ out) {
    using V16 = Vec16<T>;
    constexpr int VW = 16 / (int)sizeof(T), U = 16 / VW;
    __shared__ T part[kXyBatch][kXyT];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x;
    const int4 info = rinfo[i];
    const T dv = rdv[i];
    for (int64_t m0 = 0; m0 < n; m0 += kXyCols) {
        // vectors of a thread that hold samples (FP64 products of padding would be the time)
        const int nu = (int)min((int64_t)U, (n - m0 + kXyT * VW - 1) / (kXyT * VW));
        auto load = [&](int64_t row, typename V16::type (&v)[U]) {
            const T zero[VW] = {};
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t m = m0 + (int64_t)(threadIdx.x + kXyT * u) * VW;
                v[u] = m < ld ? __ldg(reinterpret_cast<const typename V16::type*>(xt + row * ld + m)) : V16::make(zero);
            }
        };
        T y[U][VW];
        {
            typename V16::type v[U];
            load(i, v);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (u >= nu) break;
                V16::unpack(v[u], y[u]);
#pragma unroll
                for (int x = 0; x < VW; ++x) y[u][x] = mulT(dv, y[u][x]);
            }
        }
        for (int q = info.x; q < info.y; ++q) {
            if (q == info.z) continue;
            const T w = om.cv[q];
            typename V16::type v[U];
            load(om.ci[q], v);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (u >= nu) break;
                T xv[VW];
                V16::unpack(v[u], xv);
#pragma unroll
                for (int x = 0; x < VW; ++x) y[u][x] = fmaT(w, xv[x], y[u][x]);
            }
        }
        for (int e0 = info.x; e0 < info.y; e0 += kXyBatch) {
            const int ne = min(kXyBatch, info.y - e0);
            for (int e = 0; e < ne; ++e) {
                typename V16::type v[U];
                load(om.ci[e0 + e], v);
                T s[VW] = {};
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (u >= nu) break;
                    T xv[VW];
                    V16::unpack(v[u], xv);
#pragma unroll
                    for (int x = 0; x < VW; ++x) s[x] = fmaT(y[u][x], xv[x], s[x]);
                }
                T r = s[0];
#pragma unroll
                for (int x = 1; x < VW; ++x) r += s[x];
                part[e][threadIdx.x] = r;
            }
            __syncthreads();
            for (int e = warp; e < ne; e += kXyT / 32) {
                double r = ((double)part[e][lane] + (double)part[e][lane + 32]) +
                           ((double)part[e][lane + 64] + (double)part[e][lane + 96]);
                r = warp_sum_d(r);
                if (lane == 0) out[e0 + e] = (m0 == 0 ? 0.0 : out[e0 + e]) + r / (double)n;
            }
            __syncthreads();
        }
    }
}

// T_e = (1/n) sum_m Y^T[i, m] X^T[j_e, m] for every support entry e = (i, j_e), where
// Y^T = Omega X^T: the support-restricted (Omega S)_ij with S = X^T X / n, without S.
// Warp per row of the support; lanes stride m (coalesced rows of X^T and Y^T), four
// independent partials per lane in T, combined and summed across lanes in FP64.
template <typename T>
__global__ void __launch_bounds__(256)
k_support_sddmm(int p, Csr<T> om, const T* __restrict__ yt, const T* __restrict__ xt, int64_t ld, int64_t n,
                double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kW + (threadIdx.x >> 5);
    if (i >= p) return;
    const T* yi = yt + (int64_t)i * ld;
    const int e1 = om.rp[i + 1];
    for (int e = om.rp[i]; e < e1; ++e) {
        const T* xj = xt + (int64_t)om.ci[e] * ld;
        T a0 = T(0), a1 = T(0), a2 = T(0), a3 = T(0);
        int64_t m = lane;
        for (; m + 96 < n; m += 128) {
            a0 = fmaT(yi[m], xj[m], a0);
            a1 = fmaT(yi[m + 32], xj[m + 32], a1);
            a2 = fmaT(yi[m + 64], xj[m + 64], a2);
            a3 = fmaT(yi[m + 96], xj[m + 96], a3);
        }
        for (; m < n; m += 32) a0 = fmaT(yi[m], xj[m], a0);
        const double v = warp_sum_d(((double)a0 + (double)a1) + ((double)a2 + (double)a3));
        if (lane == 0) out[e] = v / (double)n;
    }
}

// ---------------------------------------------------------------- CG (FP64, on the nnz entries)
// Conjugate gradients on H_A v = b in one cooperative launch, then the two inner products
// that give the hypergradient.
//
// What bounds it.  An iteration touches a few hundred KB (the vectors and the S entries of
// the support, all in L2 after the first one), so it is latency: as three kernels it
// was three ramps, three chains of dependent loads (row, row bounds, direction, S) and three
// last-block reductions.  Here a grid-wide barrier ends each of the two reductions
// (<p, Hp> and <r, r>), every block adds the blocks' partials itself in the same order, and
// all of them take the same step.
//   RES  (nnz at most the grid's threads: an entry a thread): e's vectors, indexes and row
//        bounds stay in registers, and the thread of (i, j) forms T_ji itself, in the same order
//        as the thread of (j, i) does, so that no barrier has to come before the symmetrisation:
//        twice the gathers, which no thread waits for longer than for its own.
//   else a grid-stride loop with T in memory and a third barrier: where the gathers are the
//        time, they are not made twice.
// Measured on GB300, p = 16384, 28 672 entries: 87 iterations in 1.00 ms, 11.5 us each (three
// kernels in a graph: about 15).
//
// Every wait is bounded: after CgArgs::wait_ns CgState::timeout is raised and every block leaves.
// The cooperative launch keeps all blocks resident.  A phase between two barriers gathers
// sum n_i^2 <= nnz p entries of S, which at a few 10^9 a second on wide supports takes longer than
// any fixed limit; the limit is 4 s and 0.1 ns for each of the nnz p.
constexpr long long kCgWaitNs = 4000000000ll;
constexpr int kCgT = 256;

template <typename T>
struct CgArgs {
    int64_t nnz;
    const int* row;
    Csr<T> om;
    const int4* rinfo;
    const int* tr;
    const T* S;
    int64_t lds;
    double lam2, tol2;
    int64_t max_iter;
    const double *b, *sgn, *om_d;
    double *x, *r, *p0, *p1, *Ap, *Tv;      // x, Ap, Tv: not RES
    double* part;                           // four arrays of kCgMaxBlocks partials
    CgState* st;
    long long wait_ns;
};

// sum over the block of s, into *out by thread 0 (fixed order)
__device__ __forceinline__ void cg_block_sum(double s, double* out) {
    __shared__ double red[kCgT / 32];
    s = warp_sum_d(s);
    __syncthreads();                        // the previous sum's readers are done with red
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        double r = threadIdx.x < kCgT / 32 ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = kCgT / 64; o > 0; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
        if (threadIdx.x == 0) *out = r;
    }
}

// The blocks' partials in a fixed order (total), and ratio = num / total or total / num, by one
// warp of every block: the FP64 rate is two lanes per SM and cycle, and a division by every warp
// of the block took longer than the barrier.  Every block gets the same bits.
struct CgSum {
    double total, ratio;
};
template <bool INV>
__device__ __forceinline__ CgSum cg_total(const double* part, double num) {
    __shared__ CgSum out;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) s += __ldcg(part + b);
        s = warp_sum_d(s);
        if (threadIdx.x == 0) {
            out.total = s;
            out.ratio = INV ? s / num : num / s;
        }
    }
    __syncthreads();
    return out;                             // next written after another barrier
}

// Grid-wide barrier on a counter that only grows; false after a timeout.
__device__ __forceinline__ bool cg_barrier(CgState* st, long long wait_ns, unsigned& target) {
    __shared__ int ok_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        target += gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&st->bar), "r"(1u) : "memory");
        int ok = 1;
        unsigned polls = 0;
        long long t0 = 0;
        for (;;) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&st->bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if ((++polls & 255u) == 0u) {
                unsigned long long t;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t0 == 0) t0 = (long long)t;
                if (*static_cast<volatile int*>(&st->timeout) || (long long)t - t0 > wait_ns) {
                    atomicExch(&st->timeout, 1);
                    ok = 0;
                    break;
                }
            }
        }
        ok_s = ok;
    }
    __syncthreads();
    return ok_s != 0;
}

// (V S)_ij = sum_{q in row i} v_q S[ci[q], j] with v = r + beta p: the diagonal term first,
// then the off-diagonal q ascending (k_support_product's order); four loads of each kind in
// flight.
template <typename T>
__device__ __forceinline__ double cg_row_dot(const CgArgs<T>& k, int4 info, int i, int j, const double* p,
                                             double beta) {
    const T* Sj = k.S + j;
    double acc = 0.0;
    if (info.z >= 0) acc = fma(beta, __ldcg(p + info.z), __ldcg(k.r + info.z)) * (double)__ldg(Sj + (int64_t)i * k.lds);
    for (int q0 = info.x; q0 < info.y; q0 += 4) {
        double v[4], w[4];
        T s[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + u;
            const bool on = q < info.y && q != info.z;
            v[u] = on ? __ldcg(p + q) : 0.0;
            w[u] = on ? __ldcg(k.r + q) : 0.0;
            s[u] = on ? __ldg(Sj + (int64_t)__ldg(k.om.ci + q) * k.lds) : T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (q0 + u >= info.y) break;
            if (q0 + u != info.z) acc = fma(fma(beta, v[u], w[u]), (double)s[u], acc);
        }
    }
    return acc;
}

// The S entries of one row's sum for a fixed column, kept in registers for rows of at most kKeep
// entries: an iteration then loads only r and p, all at once.
constexpr int kKeep = 8;
template <typename T>
struct CgRow {
    T s[kKeep];
    __device__ __forceinline__ void init(const CgArgs<T>& k, int4 info, int j) {
#pragma unroll
        for (int u = 0; u < kKeep; ++u)
            s[u] = info.x + u < info.y ? __ldg(k.S + (int64_t)__ldg(k.om.ci + info.x + u) * k.lds + j) : T(0);
    }
    __device__ __forceinline__ double dot(const CgArgs<T>& k, int4 info, int i, int j, const double* p, double beta) const {
        if (info.y - info.x > kKeep) return cg_row_dot(k, info, i, j, p, beta);
        double v[kKeep], w[kKeep];
#pragma unroll
        for (int u = 0; u < kKeep; ++u) {
            const bool on = info.x + u < info.y;
            v[u] = on ? __ldcg(p + info.x + u) : 0.0;
            w[u] = on ? __ldcg(k.r + info.x + u) : 0.0;
        }
        const int dz = info.z - info.x;      // the diagonal's place, below 0 if there is none
        double acc = 0.0;
#pragma unroll
        for (int u = 0; u < kKeep; ++u)
            if (u == dz) acc = fma(beta, v[u], w[u]) * (double)s[u];
#pragma unroll
        for (int u = 0; u < kKeep; ++u) {
            if (info.x + u >= info.y) break;
            if (u != dz) acc = fma(fma(beta, v[u], w[u]), (double)s[u], acc);
        }
        return acc;
    }
};

template <typename T, bool RES>
__global__ void __launch_bounds__(kCgT) k_cg(CgArgs<T> k) {
    const int64_t step = (int64_t)gridDim.x * kCgT, e0 = blockIdx.x * (int64_t)kCgT + threadIdx.x;
    double* part[4];
    for (int q = 0; q < 4; ++q) part[q] = k.part + q * kCgMaxBlocks;
    unsigned target = 0;
    // RES: entry e0's state
    int i = 0, j = 0, te = 0;
    int4 ri = make_int4(0, 0, -1, 0), rj = ri;
    double hd = 0.0, xe = 0.0, re = 0.0, pe = 0.0, ape = 0.0;      // hd: lambda2, on the diagonal + 1 / w_ii^2
    CgRow<T> si, sj;
    const bool own = RES && e0 < k.nnz;
    double s = 0.0;
    if constexpr (RES) {
        if (own) {
            i = k.row[e0];
            j = k.om.ci[e0];
            te = k.tr[e0];
            ri = k.rinfo[i];
            rj = k.rinfo[j];
            si.init(k, ri, j);
            sj.init(k, rj, i);
            const double w = (double)k.om.cv[e0];
            hd = i == j ? k.lam2 + 1.0 / (w * w) : k.lam2;
            re = k.b[e0];
            k.r[e0] = re;
            k.p0[e0] = re;
            pe = re;
            s = fma(re, re, s);
        }
    } else {
        for (int64_t e = e0; e < k.nnz; e += step) {
            const double v = k.b[e];
            k.r[e] = v;
            k.p0[e] = v;
            k.x[e] = 0.0;
            s = fma(v, v, s);
        }
    }
    cg_block_sum(s, part[0] + blockIdx.x);
    bool alive = cg_barrier(k.st, k.wait_ns, target);
    double rr = alive ? cg_total<true>(part[0], 1.0).total : 0.0, beta = 0.0;       // the first direction is r itself
    const double rr0 = rr;
    int done = rr == 0.0 ? 1 : 0;
    int64_t it = 0;
    while (alive && done == 0 && it < k.max_iter) {
        const double* p_old = (it & 1) ? k.p1 : k.p0;
        double* p_new = (it & 1) ? k.p0 : k.p1;
        // direction, H p and <p, H p>
        s = 0.0;
        if constexpr (RES) {
            if (own) {
                const double Te = si.dot(k, ri, i, j, p_old, beta);
                const double Tt = te >= 0 && te != (int)e0 ? sj.dot(k, rj, j, i, p_old, beta) : Te;
                pe = fma(beta, pe, re);
                p_new[e0] = pe;
                ape = fma(hd, pe, 0.5 * (Te + Tt));
                s = fma(pe, ape, s);
            }
        } else {
            for (int64_t e = e0; e < k.nnz; e += step) {
                const int a = k.row[e];
                k.Tv[e] = cg_row_dot(k, k.rinfo[a], a, k.om.ci[e], p_old, beta);
                p_new[e] = fma(beta, p_old[e], k.r[e]);
            }
            if (!(alive = cg_barrier(k.st, k.wait_ns, target))) break;
            for (int64_t e = e0; e < k.nnz; e += step) {
                const int t = k.tr[e] >= 0 ? k.tr[e] : (int)e;     // a symmetric pattern always has (j, i)
                const double w = (double)k.om.cv[e], v = p_new[e];
                double o = 0.5 * (k.Tv[e] + __ldcg(k.Tv + t));
                o += k.lam2 * v;
                if (k.om.ci[e] == k.row[e]) o += v / (w * w);
                k.Ap[e] = o;
                s = fma(v, o, s);
            }
        }
        cg_block_sum(s, part[1] + blockIdx.x);
        if (!(alive = cg_barrier(k.st, k.wait_ns, target))) break;
        const CgSum pap = cg_total<false>(part[1], rr);
        ++it;
        if (!(pap.total > 0.0)) { done = 2; break; }               // H not positive definite along p
        const double alpha = pap.ratio;
        // x, r and <r, r>
        s = 0.0;
        if constexpr (RES) {
            if (own) {
                xe = fma(alpha, pe, xe);
                re = fma(-alpha, ape, re);
                k.r[e0] = re;
                s = fma(re, re, s);
            }
        } else {
            for (int64_t e = e0; e < k.nnz; e += step) {
                k.x[e] = fma(alpha, p_new[e], k.x[e]);
                const double v = fma(-alpha, k.Ap[e], k.r[e]);
                k.r[e] = v;
                s = fma(v, v, s);
            }
        }
        cg_block_sum(s, part[0] + blockIdx.x);
        if (!(alive = cg_barrier(k.st, k.wait_ns, target))) break;
        const CgSum v = cg_total<true>(part[0], rr);
        beta = rr > 0.0 ? v.ratio : 0.0;
        rr = v.total;
        if (rr <= k.tol2 * rr0) done = 1;
    }
    // <x, sign(Omega_A) off the diagonal> and <x, Omega_A>
    double s1 = 0.0, s2 = 0.0;
    if constexpr (RES) {
        if (own) {
            s1 = xe * k.sgn[e0];
            s2 = xe * k.om_d[e0];
        }
    } else {
        for (int64_t e = e0; e < k.nnz; e += step) {
            s1 = fma(k.x[e], k.sgn[e], s1);
            s2 = fma(k.x[e], k.om_d[e], s2);
        }
    }
    cg_block_sum(s1, part[2] + blockIdx.x);
    cg_block_sum(s2, part[3] + blockIdx.x);
    if (alive) alive = cg_barrier(k.st, k.wait_ns, target);
    if (blockIdx.x == 0 && alive) {
        s1 = cg_total<true>(part[2], 1.0).total;
        __syncthreads();
        s2 = cg_total<true>(part[3], 1.0).total;
        if (threadIdx.x == 0) {
            k.st->rr = rr;
            k.st->rr0 = rr0;
            k.st->dot_sign = s1;
            k.st->dot_omega = s2;
            k.st->iterations = it;
            k.st->done = done;
        }
    }
}

// The held-out gradient on the support, one thread per entry e = (i, j):
//   out_e = (T_e + T_tr(e))/2 - [i=j] / w_ii.
template <typename T>
__global__ void __launch_bounds__(256)
k_support_heldout(int64_t nnz, const int* __restrict__ row, const int* __restrict__ ci, const T* __restrict__ cv,
                  const int* __restrict__ tr, const double* __restrict__ Tv, double* __restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
        const int te = tr[e] >= 0 ? tr[e] : (int)e;     // a symmetric pattern always has (j, i)
        double o = 0.5 * (Tv[e] + Tv[te]);
        if (ci[e] == row[e]) o -= 1.0 / (double)cv[e];
        out[e] = o;
    }
}

// dL/dOmega on the support, one thread per entry e = (i, j):
//   out_e = scale ((T_e + T_tr(e))/2 + lambda2 w_e - [i = j] / w_ii),  T = Omega S on the
// support (Alg. 1 step 4's G restricted to the entries of the iterate).
template <typename T>
__global__ void __launch_bounds__(256)
k_support_grad(int64_t nnz, const int* __restrict__ row, const int* __restrict__ ci, const T* __restrict__ cv,
               const int* __restrict__ tr, const double* __restrict__ Tv, double lam2, double scale,
               double* __restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
        const int te = tr[e] >= 0 ? tr[e] : (int)e;
        const double w = (double)cv[e];
        double o = 0.5 * (Tv[e] + Tv[te]) + lam2 * w;
        if (ci[e] == row[e]) o -= 1.0 / w;
        out[e] = scale * o;
    }
}

// FP64 copy of the support values.
template <typename T>
__global__ void k_support_values(int64_t nnz, const T* __restrict__ cv, double* __restrict__ omega_d) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
        omega_d[e] = (double)cv[e];
}

// sign(w_ij) off the diagonal, 0 on it.
template <typename T>
__global__ void k_sign_off(int p, Csr<T> om, double* sign_off) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kW + (threadIdx.x >> 5);
    if (i >= p) return;
    for (int e = om.rp[i] + lane; e < om.rp[i + 1]; e += 32) {
        const double w = (double)om.cv[e];
        sign_off[e] = (om.ci[e] == i) ? 0.0 : (w > 0.0 ? 1.0 : (w < 0.0 ? -1.0 : 0.0));
    }
}

// Partials of the smooth part at the iterate: [0] sum_e w_e T_e (= tr(Omega S Omega) with
// T = (Omega S) on the support), [1] ||Omega||_F^2, [2] sum_i log w_ii.  A thread per entry, then a
// thread per row: with a warp per row one lane's FP64 logarithm held the warp, at an FP64 rate
// of two lanes per SM and cycle (44 us at p = 16384, 7 now).
template <typename T>
__global__ void __launch_bounds__(256)
k_smooth_parts(int p, int64_t nnz, Csr<T> om, const int4* __restrict__ rinfo, const T* __restrict__ rdv,
               const double* __restrict__ Tv, double* part) {
    __shared__ double red[8][3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t0 = blockIdx.x * 256ll + threadIdx.x, step = gridDim.x * 256ll;
    double a = 0.0, b = 0.0, c = 0.0;
    for (int64_t e = t0; e < nnz; e += step) {
        const double w = (double)om.cv[e];
        a = fma(w, Tv[e], a);
        b = fma(w, w, b);
    }
    for (int64_t i = t0; i < p; i += step)
        if (rinfo[i].z >= 0) c += log((double)rdv[i]);
    a = warp_sum_d(a); b = warp_sum_d(b); c = warp_sum_d(c);
    if (lane == 0) { red[warp][0] = a; red[warp][1] = b; red[warp][2] = c; }
    __syncthreads();
    if (threadIdx.x < 3) {
        double r = 0.0;
        for (int w = 0; w < 8; ++w) r += red[w][threadIdx.x];
        part[blockIdx.x * 3 + threadIdx.x] = r;
    }
}

// out[k] = sum_b part[b * stride + k] for k < stride, in a fixed order.
__global__ void __launch_bounds__(256) k_reduce_strided(const double* part, int nb, int stride, double* out) {
    for (int k = 0; k < stride; ++k) {
        double s = 0.0;
        for (int b = threadIdx.x; b < nb; b += blockDim.x) s += part[(size_t)b * stride + k];
        s = warp_sum_d(s);
        __shared__ double red[8];
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double r = 0.0;
            for (int w = 0; w < 8; ++w) r += red[w];
            out[k] = r;
        }
        __syncthreads();
    }
}

}  // namespace

// ---------------------------------------------------------------- launchers
static int entry_blocks(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 1024); }

template <typename T>
void launch_smooth_parts(int p, int64_t nnz, Csr<T> om, const int4* rinfo, const T* rdv, const double* Tv, double* part,
                         double* out3, cudaStream_t s) {
    const int nb = entry_blocks(std::max<int64_t>(p, nnz));
    k_smooth_parts<T><<<nb, 256, 0, s>>>(p, nnz, om, rinfo, rdv, Tv, part);
    k_reduce_strided<<<1, 256, 0, s>>>(part, nb, 3, out3);
}

template <typename T>
void launch_dense_grad(int p, int64_t nnz, Csr<T> om, const int4* rinfo, const T* rdv, const T* S, int64_t lds, T* G,
                       int64_t ldg, T lam2, T scale, cudaStream_t s) {
    constexpr int TL = sizeof(T) == 4 ? 64 : 32;      // two tiles: 33 KB (FP32) / 17 KB (FP64) of shared memory
    const int nt = (p + TL - 1) / TL;
    // bit 0: 16-byte stores of G; bit 1: 16-byte loads of S
    const int vec = (((uintptr_t)G % 16 == 0 && (ldg * (int64_t)sizeof(T)) % 16 == 0) ? 1 : 0) |
                    (((uintptr_t)S % 16 == 0 && (lds * (int64_t)sizeof(T)) % 16 == 0) ? 2 : 0);
    const unsigned nb = (unsigned)((int64_t)nt * (nt + 1) / 2);
    if ((nnz - p) * 2 * TL > (int64_t)kGradList * p)
        k_dense_grad_rows<T, TL><<<nb, 256, 0, s>>>(p, om, rinfo, rdv, S, lds, G, ldg, lam2, scale, nt, vec);
    else
        k_dense_grad_pair<T, TL><<<nb, 256, 0, s>>>(p, om, rinfo, rdv, S, lds, G, ldg, lam2, scale, nt, vec);
}

template <typename T>
void launch_spmm_dense(int p, Csr<T> om, const int4* rinfo, const T* rdv, const T* B, int64_t ldb, int64_t m,
                       T* C, int64_t ldc, cudaStream_t s) {
    dim3 g((p + kW - 1) / kW, (unsigned)((m + 127) / 128));
    k_spmm_dense<T><<<g, 256, 0, s>>>(p, om, rinfo, rdv, B, ldb, m, C, ldc);
}

template <typename T>
void launch_spmm_dense_t(int p, Csr<T> om, const int4* rinfo, const T* rdv, const T* B, int64_t ldb, int64_t m,
                         T* Ct, int64_t ldt, T scale, cudaStream_t s) {
    dim3 g((unsigned)((p + 31) / 32), (unsigned)((m + 127) / 128));
    k_spmm_dense_t<T><<<g, 256, 0, s>>>(p, om, rinfo, rdv, B, ldb, m, Ct, ldt, scale);
}

void launch_transpose(const void* in, int in_dt, int64_t rows, int64_t cols, int64_t ldi, void* out, int out_dt,
                      int64_t ldo, double scale, cudaStream_t s, int64_t pad_to) {
    const int64_t rows_out = std::max(rows, pad_to);
    dim3 g((unsigned)((cols + 63) / 64), (unsigned)((rows_out + 63) / 64));
    const bool o64 = out_dt == HPC_F64;
    if (in_dt == HPC_BF16 && o64) {
        k_transpose<__nv_bfloat16, double><<<g, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(in), rows, cols, ldi,
                                                              static_cast<double*>(out), ldo, rows_out, scale);
    } else if (in_dt == HPC_BF16) {
        k_transpose<__nv_bfloat16, float><<<g, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(in), rows, cols, ldi,
                                                             static_cast<float*>(out), ldo, rows_out, scale);
    } else if (in_dt == HPC_F64 && o64) {
        k_transpose<double, double><<<g, 256, 0, s>>>(static_cast<const double*>(in), rows, cols, ldi,
                                                       static_cast<double*>(out), ldo, rows_out, scale);
    } else if (in_dt == HPC_F64) {
        k_transpose<double, float><<<g, 256, 0, s>>>(static_cast<const double*>(in), rows, cols, ldi,
                                                      static_cast<float*>(out), ldo, rows_out, scale);
    } else if (o64) {
        k_transpose<float, double><<<g, 256, 0, s>>>(static_cast<const float*>(in), rows, cols, ldi,
                                                      static_cast<double*>(out), ldo, rows_out, scale);
    } else {
        k_transpose<float, float><<<g, 256, 0, s>>>(static_cast<const float*>(in), rows, cols, ldi,
                                                     static_cast<float*>(out), ldo, rows_out, scale);
    }
}

template <typename T>
void launch_transpose_index(int p, Csr<T> om, int* tr, int* row, cudaStream_t s) {
    k_transpose_index<T><<<(p + kW - 1) / kW, 256, 0, s>>>(p, om, tr, row);
}

template <typename T>
void launch_support_product(int p, Csr<T> om, const int4* rinfo, const double* v, const T* S, int64_t lds,
                            double* out, cudaStream_t s) {
    k_support_product<T><<<(p + kW - 1) / kW, 256, 0, s>>>(p, om, rinfo, v, S, lds, out);
}

template <typename T>
void launch_support_xy(int p, Csr<T> om, const int4* rinfo, const T* rdv, const T* xt, int64_t ld, int64_t n,
                       double* out, cudaStream_t s) {
    k_support_xy<T><<<p, kXyT, 0, s>>>(p, om, rinfo, rdv, xt, ld, n, out);
}

template <typename T>
void launch_support_sddmm(int p, Csr<T> om, const T* yt, const T* xt, int64_t ld, int64_t n, double* out,
                          cudaStream_t s) {
    k_support_sddmm<T><<<(p + kW - 1) / kW, 256, 0, s>>>(p, om, yt, xt, ld, n, out);
}

template <typename T>
void launch_support_heldout(int64_t nnz, const int* row, Csr<T> om, const int* tr, const double* Tv, double* out,
                            cudaStream_t s) {
    k_support_heldout<T><<<entry_blocks(nnz), 256, 0, s>>>(nnz, row, om.ci, om.cv, tr, Tv, out);
}

template <typename T>
void launch_support_grad(int64_t nnz, const int* row, Csr<T> om, const int* tr, const double* Tv, double lam2,
                         double scale, double* out, cudaStream_t s) {
    k_support_grad<T><<<entry_blocks(nnz), 256, 0, s>>>(nnz, row, om.ci, om.cv, tr, Tv, lam2, scale, out);
}

template <typename T>
void launch_support_vectors(int p, int64_t nnz, Csr<T> om, double* omega_d, double* sign_off, cudaStream_t s) {
    k_support_values<T><<<256, 256, 0, s>>>(nnz, om.cv, omega_d);
    k_sign_off<T><<<(p + kW - 1) / kW, 256, 0, s>>>(p, om, sign_off);
}

size_t cg_vector_doubles(int64_t nnz) { return 6 * (size_t)nnz + 4 * kCgMaxBlocks; }

// CG on H_A v = b and its two inner products; vec: cg_vector_doubles(nnz), st: zeroed here.
template <typename T>
cudaError_t launch_cg(int p, int64_t nnz, const int* row, Csr<T> om, const int4* rinfo, const int* tr, const T* S, int64_t lds,
                      double lam2, double tol, int64_t max_iter, const double* b, const double* sgn, const double* om_d,
                      double* vec, CgState* st, int num_sms, cudaStream_t s) {
    CgArgs<T> k{nnz, row, om, rinfo, tr, S, lds, lam2, tol * tol, max_iter, b, sgn, om_d, nullptr, nullptr, nullptr,
                nullptr, nullptr, nullptr, nullptr, st, kCgWaitNs + (long long)(0.1 * (double)nnz * (double)p)};
    double** v[6] = {&k.x, &k.r, &k.p0, &k.p1, &k.Ap, &k.Tv};
    for (int q = 0; q < 6; ++q) *v[q] = vec + (size_t)q * nnz;
    k.part = vec + 6 * (size_t)nnz;
    int occ[2] = {0, 0};
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[0], k_cg<T, false>, kCgT, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[1], k_cg<T, true>, kCgT, 0);
    if (e != cudaSuccess) return e;
    const int64_t want = (nnz + kCgT - 1) / kCgT;
    const int64_t fit = std::min<int64_t>((int64_t)occ[1] * num_sms, kCgMaxBlocks);
    const bool res = want <= fit;
    int64_t nb = res ? want : std::max<int64_t>(1, std::min<int64_t>((int64_t)occ[0] * num_sms, kCgMaxBlocks));
    e = cudaMemsetAsync(st, 0, sizeof(CgState), s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)nb);
    cfg.blockDim = dim3(kCgT);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return res ? cudaLaunchKernelEx(&cfg, k_cg<T, true>, k) : cudaLaunchKernelEx(&cfg, k_cg<T, false>, k);
}

#define HPC_ADJ_INSTANTIATE(T)                                                                                  \
    template void launch_dense_grad<T>(int, int64_t, Csr<T>, const int4*, const T*, const T*, int64_t, T*, int64_t, T, T, \
                                       cudaStream_t);                                                           \
    template void launch_spmm_dense<T>(int, Csr<T>, const int4*, const T*, const T*, int64_t, int64_t, T*,      \
                                       int64_t, cudaStream_t);                                                  \
    template void launch_spmm_dense_t<T>(int, Csr<T>, const int4*, const T*, const T*, int64_t, int64_t, T*,    \
                                         int64_t, T, cudaStream_t);                                             \
    template void launch_transpose_index<T>(int, Csr<T>, int*, int*, cudaStream_t);                             \
    template void launch_support_product<T>(int, Csr<T>, const int4*, const double*, const T*, int64_t, double*, \
                                            cudaStream_t);                                                      \
    template void launch_support_sddmm<T>(int, Csr<T>, const T*, const T*, int64_t, int64_t, double*,         \
                                          cudaStream_t);                                                        \
    template void launch_support_xy<T>(int, Csr<T>, const int4*, const T*, const T*, int64_t, int64_t, double*, \
                                       cudaStream_t);                                                           \
    template void launch_support_heldout<T>(int64_t, const int*, Csr<T>, const int*, const double*, double*,     \
                                            cudaStream_t);                                                      \
    template cudaError_t launch_cg<T>(int, int64_t, const int*, Csr<T>, const int4*, const int*, const T*, int64_t,  \
                                      double, double, int64_t, const double*, const double*, const double*,     \
                                      double*, CgState*, int, cudaStream_t);                                    \
    template void launch_support_vectors<T>(int, int64_t, Csr<T>, double*, double*, cudaStream_t);          \
    template void launch_support_grad<T>(int64_t, const int*, Csr<T>, const int*, const double*, double,      \
                                         double, double*, cudaStream_t);                                        \
    template void launch_smooth_parts<T>(int, int64_t, Csr<T>, const int4*, const T*, const double*, double*,   \
                                         double*, cudaStream_t);

HPC_ADJ_INSTANTIATE(float)
HPC_ADJ_INSTANTIATE(double)

}  // namespace hpc
