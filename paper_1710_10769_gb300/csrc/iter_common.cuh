// Device helpers shared by the iteration's translation units: exact-rounding
// arithmetic of both value types, compensated FP32 sums, the prox of eq. (2), BF16
// upper bounds, and the acquire/release primitives of the grid-wide barriers.
#pragma once

#include "internal.cuh"

namespace hpc {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;

__device__ __forceinline__ float fmaT(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return __fma_rn(a, b, c); }

__device__ __forceinline__ void vload(float (&a)[4], const float* p) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w;
}
__device__ __forceinline__ void vload(double (&a)[2], const double* p) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    a[0] = v.x; a[1] = v.y;
}

__device__ __forceinline__ int warp_incl_scan(int x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// Compensated FP32 accumulator for sums that would otherwise need FP64, whose
// rate on this GPU is a small fraction of FP32: every addition is Knuth's
// TwoSum, the rounding errors collect in lo, and the pair carries ~44 bits.
// FP64 appears only in the final cross-block reductions.
struct F2 {
    float hi = 0.f, lo = 0.f;
};
__device__ __forceinline__ void acc_add(F2& a, float b) {
    const float s = __fadd_rn(a.hi, b);
    const float bp = __fsub_rn(s, a.hi);
    const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bp)), __fsub_rn(b, bp));
    a.hi = s;
    a.lo = __fadd_rn(a.lo, err);
}
__device__ __forceinline__ void acc_add(double& a, double b) { a += b; }
__device__ __forceinline__ double acc_value(const F2& a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double acc_value(double a) { return a; }
__device__ __forceinline__ F2 warp_sum(F2 a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h = __shfl_xor_sync(kFull, a.hi, o);
        const float l = __shfl_xor_sync(kFull, a.lo, o);
        acc_add(a, h);
        a.lo = __fadd_rn(a.lo, l);
    }
    return a;
}
template <typename T> struct AccOf { using type = F2; };
template <> struct AccOf<double> { using type = double; };

__device__ __forceinline__ float mulT(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulT(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float logT(float a) { return logf(a); }
__device__ __forceinline__ double logT(double a) { return log(a); }

// phi(x) = x - log(1 + x) for x > -1.  FP32: for |x| < 1/8 the Taylor series
// sum_{k>=0} (-1)^k x^(k+2) / (k+2), truncated after x^10 (relative error
// < 2e-9), avoids the cancellation of x - log1p(x); otherwise x - log1pf(x).
__device__ __forceinline__ float phiT(float x) {
    if (fabsf(x) < 0.125f) {
        float r = 1.0f / 10.0f;
        r = fmaf(x, r, -1.0f / 9.0f);
        r = fmaf(x, r, 1.0f / 8.0f);
        r = fmaf(x, r, -1.0f / 7.0f);
        r = fmaf(x, r, 1.0f / 6.0f);
        r = fmaf(x, r, -1.0f / 5.0f);
        r = fmaf(x, r, 1.0f / 4.0f);
        r = fmaf(x, r, -1.0f / 3.0f);
        r = fmaf(x, r, 1.0f / 2.0f);
        return x * x * r;
    }
    return x - log1pf(x);
}
__device__ __forceinline__ double phiT(double x) { return x - log1p(x); }

// Prox of eq. (2) for one candidate entry at step tau (tau and tau*lambda1 are
// exact: tau is a power of two).  The diagonal is not thresholded.
template <typename T>
__device__ __forceinline__ T prox_entry(T om, T g, T tau, T tl1, bool diag) {
    const T z = om - tau * g;
    if (diag) return z;
    if (z > tl1) return z - tl1;
    if (z < -tl1) return z + tl1;
    return T(0);
}

// NaN-propagating maximum of two non-negative values.
template <typename T>
__device__ __forceinline__ T max_nan(T a, T b) { return (a != a || b != b) ? T(NAN) : (a > b ? a : b); }

// Non-negative value rounded up to BF16 (an upper bound: 8 bits of mantissa kept,
// the rest carried upwards), and its float value.
__device__ __forceinline__ unsigned short bf16_up(float x) {
    if (!(x == x)) return 0x7fc0;
    unsigned u = __float_as_uint(x);
    if (u & 0xffffu) u += 0x10000u;
    return (unsigned short)(u >> 16);
}
__device__ __forceinline__ unsigned short bf16_up(double x) { return bf16_up(__double2float_ru(x)); }
__device__ __forceinline__ float bf16_val(unsigned short b) { return __uint_as_float((unsigned)b << 16); }

// Eight BF16 block maxima from one 16-byte load (element 0 in the low half of x).
__device__ __forceinline__ void bf16x8(const uint4 v, float (&f)[8]) {
    f[0] = __uint_as_float(v.x << 16);
    f[1] = __uint_as_float(v.x & 0xffff0000u);
    f[2] = __uint_as_float(v.y << 16);
    f[3] = __uint_as_float(v.y & 0xffff0000u);
    f[4] = __uint_as_float(v.z << 16);
    f[5] = __uint_as_float(v.z & 0xffff0000u);
    f[6] = __uint_as_float(v.w << 16);
    f[7] = __uint_as_float(v.w & 0xffff0000u);
}

template <typename T>
__device__ __forceinline__ float abs_up(T x) {
    if constexpr (sizeof(T) == 4) return fabsf(x);
    else return __double2float_ru(fabs(x));
}

template <typename T>
__device__ __forceinline__ bool bound_keeps(float g1, float B, bool long_chain, T lam1) {
    const float bound = __fmul_ru(g1, B);
    bool below;
    if constexpr (sizeof(T) == 4) below = bound <= lam1;
    else below = (double)bound <= lam1;
    return long_chain || !below;
}

// tau = 2^-h in T, exactly (what ldexp(1, -h) rounds to, denormals and 0 included).
template <typename T> __device__ __forceinline__ T tau_pow2(int h);
template <> __device__ __forceinline__ float tau_pow2<float>(int h) {
    return h <= 126 ? __int_as_float((127 - h) << 23) : (h <= 149 ? __int_as_float(1 << (149 - h)) : 0.f);
}
template <> __device__ __forceinline__ double tau_pow2<double>(int h) {
    return h <= 1022 ? __longlong_as_double((long long)(1023 - h) << 52)
                     : (h <= 1074 ? __longlong_as_double(1ll << (1074 - h)) : 0.0);
}

__device__ __forceinline__ F2 to_acc(float x) { F2 a; a.hi = x; return a; }
__device__ __forceinline__ double to_acc(double x) { return x; }
__device__ __forceinline__ void acc_merge(F2& a, const F2& b) { acc_add(a, b.hi); a.lo = __fadd_rn(a.lo, b.lo); }
__device__ __forceinline__ void acc_merge(double& a, double b) { a += b; }

__device__ __forceinline__ long long tail_clock_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return (long long)t;
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned atom_add_acq_rel_gpu(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ int ld_volatile_int(const int* p) { return *static_cast<const volatile int*>(p); }

constexpr long long kBarrierWaitNs = 4000000000ll;   // 4 s

}  // namespace
}  // namespace hpc
