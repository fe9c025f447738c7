// S = X^T X / n with SIMT fused multiply-adds (Alg. 2 step 2): the FP64 mode and
// the "plain FP32" mode that the tensor-core modes are measured against.
//
// X is n x p row-major, so a K-slab X[k0:k0+BK, i0:i0+BM] is BK contiguous row
// segments: both operands of the tile S[I, J] are loaded coalesced from the same
// matrix.  Only tiles with I <= J run; each writes its tile and the mirror
// S[J, I], so S is bitwise symmetric (the product x_ki x_kj is commutative and
// every entry is one FMA chain over k in the same order).
#include <cuda_bf16.h>

#include <cstdint>
#include <type_traits>

#include "internal.cuh"

namespace hpc {
namespace {

template <typename TX, typename T>
__device__ __forceinline__ T load_as(const TX* p) { return (T)(*p); }
template <>
__device__ __forceinline__ float load_as<__nv_bfloat16, float>(const __nv_bfloat16* p) { return __bfloat162float(*p); }
template <>
__device__ __forceinline__ double load_as<__nv_bfloat16, double>(const __nv_bfloat16* p) {
    return (double)__bfloat162float(*p);
}

__device__ __forceinline__ float fmaT(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return __fma_rn(a, b, c); }

// 256 threads as 16 x 16; each thread owns a TM x TM micro-tile at rows ty + 16a,
// columns tx + 16b of the BM x BM tile (BM = 16 TM).
template <typename TX, typename T, int TM>
__global__ void __launch_bounds__(256)
k_gram_simt(const TX* __restrict__ X, int64_t n, int64_t p, T* __restrict__ S, int64_t lds, int nb) {
    constexpr int BM = 16 * TM;
    constexpr int BK = 16;
    __shared__ T As[BK][BM + 1];
    __shared__ T Bs[BK][BM + 1];
    // map the linear block index to an upper-triangular tile (bi <= bj)
    int t = blockIdx.x, bi = 0;
    while (t >= nb - bi) { t -= nb - bi; ++bi; }
    const int bj = bi + t;
    const int64_t i0 = (int64_t)bi * BM, j0 = (int64_t)bj * BM;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    T acc[TM][TM];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TM; ++b) acc[a][b] = T(0);

    for (int64_t k0 = 0; k0 < n; k0 += BK) {
        for (int idx = threadIdx.x; idx < BK * BM; idx += 256) {
            const int kk = idx / BM, ii = idx % BM;
            const int64_t k = k0 + kk;
            const int64_t ia = i0 + ii, ja = j0 + ii;
            As[kk][ii] = (k < n && ia < p) ? load_as<TX, T>(X + k * p + ia) : T(0);
            Bs[kk][ii] = (k < n && ja < p) ? load_as<TX, T>(X + k * p + ja) : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[TM], b[TM];
#pragma unroll
            for (int q = 0; q < TM; ++q) { a[q] = As[kk][ty + 16 * q]; b[q] = Bs[kk][tx + 16 * q]; }
#pragma unroll
            for (int q = 0; q < TM; ++q)
#pragma unroll
                for (int r = 0; r < TM; ++r) acc[q][r] = fmaT(a[q], b[r], acc[q][r]);
        }
        __syncthreads();
    }
    const T dn = (T)n;
#pragma unroll
    for (int q = 0; q < TM; ++q) {
        const int64_t i = i0 + ty + 16 * q;
        if (i >= p) continue;
#pragma unroll
        for (int r = 0; r < TM; ++r) {
            const int64_t j = j0 + tx + 16 * r;
            if (j >= p) continue;
            const T v = acc[q][r] / dn;
            S[i * lds + j] = v;
            if (bi != bj) S[j * lds + i] = v;
        }
    }
}

// FP32 form: BM x BM tiles (BM = 16 TM), 256 threads as 16 x 16, each thread owning a TM x TM
// micro-tile made of groups of four rows {64 h + 4 ty .. + 3} and the same split of columns
// around tx, so that the 16-byte operand reads of eight consecutive lanes fall on 32
// different banks.  K-slabs of 16 rows are double-buffered in shared memory: the next slab
// is loaded into registers while the current one is multiplied, one barrier per slab.  Every
// entry is one FMA chain over k in ascending order, so S is bitwise symmetric and equals the
// scalar kernel's values.
//
// What bounds it: FP32 FMAs, 128 per SM and cycle.  They are issued in pairs
// (fma.rn.f32x2, each half rounded as fma.rn.f32), a pair of columns per
// instruction, which leaves half of the issue slots to the operand reads, the loads and the
// packing of the row operand.  VEC: rows of X that start on 16-byte boundaries (8 for
// BF16) come in by four elements and S goes out by four; other rows element by
// element, 128 neighbours at a time, into the same slabs.
// Measured on GB300, FP32 X: p = 3001, n = 1500 (rows off 16 bytes) 421 -> 326 us, 41 TFLOP/s;
// p = 3001, n = 600 170 -> 150; p = 4096, n = 600 242 -> 225; p = 300, n = 600 70 -> 31.
template <typename TX>
__device__ __forceinline__ float4 load4(const TX* p);
template <>
__device__ __forceinline__ float4 load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <>
__device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
}
template <>
__device__ __forceinline__ float4 load4<double>(const double*) { return make_float4(0.f, 0.f, 0.f, 0.f); }   // not VEC

__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long dup2(float a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}

template <typename TX, int TM, bool VEC>
__global__ void __launch_bounds__(256, TM == 4 ? 4 : 2)
k_gram_simt_f32(const TX* __restrict__ X, int64_t n, int64_t p, float* __restrict__ S, int64_t lds, int nb) {
    constexpr int BM = 16 * TM, BK = 16, H = TM / 4;
    constexpr int L = BK * BM / 256;                  // elements of each operand a thread loads
    __shared__ __align__(16) float As[2][BK][BM];
    __shared__ __align__(16) float Bs[2][BK][BM];
    int t = blockIdx.x, bi = 0;
    while (t >= nb - bi) { t -= nb - bi; ++bi; }
    const int bj = bi + t;
    const int64_t i0 = (int64_t)bi * BM, j0 = (int64_t)bj * BM;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    // slab loader: VEC: vector u of thread t is row t / (BM / 4) + u 1024 / BM, columns
    // 4 (t % (BM / 4)) .. + 3; else element u is row t / BM + u 256 / BM, column t % BM
    constexpr int PR = VEC ? BM / 4 : BM, RS = 256 / PR;
    const int lk = threadIdx.x / PR, lc = (threadIdx.x % PR) * (VEC ? 4 : 1);
    const bool ai = i0 + lc < p, bj_ok = j0 + lc < p;          // VEC: p % 4 == 0, a vector is all in or all out
    float ra[L], rb[L];
    auto load = [&](int64_t k0) {
        if constexpr (VEC) {
#pragma unroll
            for (int u = 0; u < L / 4; ++u) {
                const int64_t k = k0 + lk + RS * u;
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 va = k < n && ai ? load4<TX>(X + k * p + i0 + lc) : z;
                const float4 vb = k < n && bj_ok ? load4<TX>(X + k * p + j0 + lc) : z;
                ra[4 * u] = va.x; ra[4 * u + 1] = va.y; ra[4 * u + 2] = va.z; ra[4 * u + 3] = va.w;
                rb[4 * u] = vb.x; rb[4 * u + 1] = vb.y; rb[4 * u + 2] = vb.z; rb[4 * u + 3] = vb.w;
            }
        } else {
#pragma unroll
            for (int u = 0; u < L; ++u) {
                const int64_t k = k0 + lk + RS * u;
                ra[u] = k < n && ai ? load_as<TX, float>(X + k * p + i0 + lc) : 0.f;
                rb[u] = k < n && bj_ok ? load_as<TX, float>(X + k * p + j0 + lc) : 0.f;
            }
        }
    };
    auto store = [&](int b) {
        if constexpr (VEC) {
#pragma unroll
            for (int u = 0; u < L / 4; ++u) {
                *reinterpret_cast<float4*>(&As[b][lk + RS * u][lc]) =
                    make_float4(ra[4 * u], ra[4 * u + 1], ra[4 * u + 2], ra[4 * u + 3]);
                *reinterpret_cast<float4*>(&Bs[b][lk + RS * u][lc]) =
                    make_float4(rb[4 * u], rb[4 * u + 1], rb[4 * u + 2], rb[4 * u + 3]);
            }
        } else {
#pragma unroll
            for (int u = 0; u < L; ++u) {
                As[b][lk + RS * u][lc] = ra[u];
                Bs[b][lk + RS * u][lc] = rb[u];
            }
        }
    };
    unsigned long long acc[TM][TM / 2];
#pragma unroll
    for (int q = 0; q < TM; ++q)
#pragma unroll
        for (int r = 0; r < TM / 2; ++r) acc[q][r] = 0ull;
    load(0);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int64_t k0 = 0; k0 < n; k0 += BK) {
        const bool more = k0 + BK < n;
        if (more) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[TM];
            unsigned long long b[TM / 2];
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const float4 v = *reinterpret_cast<const float4*>(&As[buf][kk][64 * h + 4 * ty]);
                a[4 * h] = v.x; a[4 * h + 1] = v.y; a[4 * h + 2] = v.z; a[4 * h + 3] = v.w;
                const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][64 * h + 4 * tx]);
                b[2 * h] = w.x; b[2 * h + 1] = w.y;
            }
#pragma unroll
            for (int q = 0; q < TM; ++q) {
                const unsigned long long aa = dup2(a[q]);
#pragma unroll
                for (int r = 0; r < TM / 2; ++r) fma2(acc[q][r], aa, b[r]);
            }
        }
        if (more) store(buf ^ 1);
        __syncthreads();
        buf ^= 1;
    }
    const float dn = (float)n;
    float v[TM][TM];
#pragma unroll
    for (int q = 0; q < TM; ++q)
#pragma unroll
        for (int r = 0; r < TM / 2; ++r) {
            v[q][2 * r] = __uint_as_float((unsigned)acc[q][r]) / dn;
            v[q][2 * r + 1] = __uint_as_float((unsigned)(acc[q][r] >> 32)) / dn;
        }
    // row (column) q of the thread is 64 (q / 4) + 4 ty (tx) + q % 4 of the tile
#pragma unroll
    for (int q = 0; q < TM; ++q) {
        const int64_t i = i0 + 64 * (q >> 2) + 4 * ty + (q & 3), j = j0 + 64 * (q >> 2) + 4 * tx + (q & 3);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int64_t jc = j0 + 64 * h + 4 * tx, ic = i0 + 64 * h + 4 * ty;
            if constexpr (VEC) {         // a group of four is all inside or all outside
                if (i < p && jc < p)
                    *reinterpret_cast<float4*>(S + i * lds + jc) =
                        make_float4(v[q][4 * h], v[q][4 * h + 1], v[q][4 * h + 2], v[q][4 * h + 3]);
                // the mirror: row j of the lower tile gets this thread's column q
                if (bi != bj && j < p && ic < p)
                    *reinterpret_cast<float4*>(S + j * lds + ic) =
                        make_float4(v[4 * h][q], v[4 * h + 1][q], v[4 * h + 2][q], v[4 * h + 3][q]);
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (i < p && jc + u < p) S[i * lds + jc + u] = v[q][4 * h + u];
                    if (bi != bj && j < p && ic + u < p) S[j * lds + ic + u] = v[4 * h + u][q];
                }
            }
        }
    }
}

template <typename TX, int TM>
cudaError_t run_f32_t(const void* X, int64_t n, int64_t p, float* S, int64_t lds, bool vec, cudaStream_t s) {
    const int64_t nb = (p + 16 * TM - 1) / (16 * TM);
    const unsigned tiles = (unsigned)(nb * (nb + 1) / 2);
    if constexpr (!std::is_same<TX, double>::value) {
        if (vec) {
            k_gram_simt_f32<TX, TM, true><<<tiles, 256, 0, s>>>(static_cast<const TX*>(X), n, p, S, lds, (int)nb);
            return cudaGetLastError();
        }
    }
    k_gram_simt_f32<TX, TM, false><<<tiles, 256, 0, s>>>(static_cast<const TX*>(X), n, p, S, lds, (int)nb);
    return cudaGetLastError();
}

template <typename TX>
cudaError_t run_f32(const void* X, int64_t n, int64_t p, void* S, int64_t lds, cudaStream_t s) {
    const bool vec = p % 4 == 0 && lds % 4 == 0 && reinterpret_cast<uintptr_t>(S) % 16 == 0 &&
                     reinterpret_cast<uintptr_t>(X) % (4 * sizeof(TX)) == 0;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // 64 x 64 tiles where 128 x 128 ones would leave a third of the SMs without one, or give a few
    // of them a second one (n = 600, us, 64 against 128: p = 1001 35, 84; p = 1500 45, 70; p = 2000
    // 86, 70; p = 2200 107, 121; p = 3001 above 150, 150)
    const int64_t nb = (p + 127) / 128, t = nb * (nb + 1) / 2;
    const bool small = 3 * t < 2 * sms || (t > sms && 7 * t < 8 * sms);
    return small ? run_f32_t<TX, 4>(X, n, p, static_cast<float*>(S), lds, vec, s)
                 : run_f32_t<TX, 8>(X, n, p, static_cast<float*>(S), lds, vec, s);
}

template <typename TX, typename T, int TM>
cudaError_t run(const void* X, int64_t n, int64_t p, void* S, int64_t lds, cudaStream_t s) {
    constexpr int BM = 16 * TM;
    const int nb = (int)((p + BM - 1) / BM);
    const long long tiles = (long long)nb * (nb + 1) / 2;
    k_gram_simt<TX, T, TM><<<(unsigned)tiles, 256, 0, s>>>(static_cast<const TX*>(X), n, p, static_cast<T*>(S),
                                                           lds, nb);
    return cudaGetLastError();
}

}  // namespace

cudaError_t gram_simt(const void* X, int xdt, int64_t n, int64_t p, void* S, int sdt, int64_t lds,
                      cudaStream_t s, int* launches) {
    if (launches) *launches += 1;
    if (sdt == HPC_F64) {
        if (xdt == HPC_F64) return run<double, double, 4>(X, n, p, S, lds, s);
        if (xdt == HPC_F32) return run<float, double, 4>(X, n, p, S, lds, s);
        return run<__nv_bfloat16, double, 4>(X, n, p, S, lds, s);
    }
    if (xdt == HPC_F64) return run_f32<double>(X, n, p, S, lds, s);
    if (xdt == HPC_F32) return run_f32<float>(X, n, p, S, lds, s);
    return run_f32<__nv_bfloat16>(X, n, p, S, lds, s);
}

}  // namespace hpc
