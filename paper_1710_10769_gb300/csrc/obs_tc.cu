// Obs variant (Alg. 3): the products that replace S.
//
//   Y^T = Omega X^T (p x n)            row-split SpMM (adjoint.cu), canonical order
//   Z   = Y X / n = Y^T (X^T)^T / n    this file: tcgen05 GEMM on K-major panels
//
// Z equals W = Omega S, so the screening rule of the Cov pass applies: an entry
// can enter a prox step only if it is in the support or |G_ij| > lambda1, and
// |G_ij| > lambda1 needs max(|Z_ij|, |Z_ji|) > lambda1.  Persistent CTAs walk the
// tile pairs Z[I, J] and Z[J, I] (I <= J, 128 x 128 tiles), each into one of two
// TMEM accumulator pairs; the epilogue warps transpose the second tile through
// shared memory and emit both (i, j) and (j, i) -- flagged as paired, so no
// partner request follows -- for every pair in the support or above the
// threshold (Alg. 3 steps 4-6 with the transpose done inside the CTA), while the
// next pair accumulates.  Z is never stored.
//
// Operands are BF16 hi/lo panels (BF16X3: hi*hi + hi*lo + lo*hi) or TF32
// panels, K-major, zero padded; loaded by TMA (128-byte swizzle) through an
// mbarrier ring; every wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <vector>

#include "internal.cuh"
#include "ptx.cuh"

namespace hpc {
namespace {

constexpr int kT = 128;                    // tile edge (UMMA M = N = 128)
constexpr int kRowB = 128;                 // bytes per swizzle row
constexpr int kPanelTile = kT * kRowB;     // 16 KB
constexpr int kObsBand = 8;                // row blocks per band of the pair list
constexpr uint32_t kTmemCols = 256;        // one accumulator pair: two 128-column FP32 accumulators
constexpr long long kWaitLimit = 1ll << 22;     // polls of at most 1 us each

enum : int { kObsBf16x3 = 0, kObsTf32 = 1 };

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ptx::smem_u32(dst)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void ptx_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(ptx::smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <int MODE>
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    if constexpr (MODE == kObsTf32) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
            : "memory");
    }
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     ptx::smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// K-major, 128-byte swizzle, 8-row groups 1024 bytes apart, descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

template <int MODE>
__host__ __device__ constexpr uint32_t instr_desc() {
    return (1u << 4) | ((MODE == kObsTf32 ? 2u : 1u) << 7) | ((MODE == kObsTf32 ? 2u : 1u) << 10) |
           ((uint32_t)(kT >> 3) << 17) | ((uint32_t)(kT >> 4) << 24);
}

template <int MODE>
struct ObsCfg {
    static constexpr int kPieces = MODE == kObsBf16x3 ? 2 : 1;
    static constexpr int kTerms = MODE == kObsBf16x3 ? 3 : 1;
    static constexpr int kElem = MODE == kObsTf32 ? 4 : 2;
    static constexpr int kBK = kRowB / kElem;
    static constexpr int kMmaK = 32 / kElem;
    static constexpr int kStageBytes = kPieces * 2 * kPanelTile;    // A and B tiles, each piece
    static constexpr int kStages = MODE == kObsBf16x3 ? 3 : 5;
    static constexpr int kRing = 8;                                  // pair slots between the roles
    static constexpr int kLook = 4;                                  // pairs published ahead of the loads
    static constexpr int kSupBytes = kRing * kT * (16 + 4);          // support masks (uint4) and CSR starts
    static constexpr int kCtlBytes = 512;                            // barriers, pair slots, TMEM address
    static constexpr int kSmem = kStages * kStageBytes + kSupBytes + kCtlBytes + 1024;
};

constexpr int kEpiWarps = 8;
constexpr int kObsThreads = 128 + 32 * kEpiWarps;     // warpgroup 0: roles; warpgroups 1-2: epilogue
constexpr int kHelpThreads = 64;                      // warps 2-3: support masks
// Registers per thread after setmaxnreg (warpgroup 0 down, the epilogue warpgroups up);
// the host checks that the launch's pool covers both (kMinLaunchRegs) before launching.
constexpr int kRegsSmall = 56;
constexpr int kRegsEpi = 216;
constexpr int kMinLaunchRegs = (128 * kRegsSmall + 32 * kEpiWarps * kRegsEpi + kObsThreads - 1) / kObsThreads;


// 32 TMEM lanes x 16 consecutive 32-bit columns: thread t gets lane (base + t).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

// v[O + b] for a run-time b in 0..31 without indexing registers dynamically: a
// five-level tree of selects on the bits of b.
template <int O>
__device__ __forceinline__ float pick32(const float (&v)[64], int b) {
    float t16[16], t8[8], t4[4], t2[2];
#pragma unroll
    for (int i = 0; i < 16; ++i) t16[i] = (b & 16) ? v[O + 16 + i] : v[O + i];
#pragma unroll
    for (int i = 0; i < 8; ++i) t8[i] = (b & 8) ? t16[8 + i] : t16[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) t4[i] = (b & 4) ? t8[4 + i] : t8[i];
#pragma unroll
    for (int i = 0; i < 2; ++i) t2[i] = (b & 2) ? t4[2 + i] : t4[i];
    return (b & 1) ? t2[1] : t2[0];
}

// Support of row g in the columns j0 .. j0 + 127: a 128-bit mask and the CSR position
// of the row's first entry at or after column j0 (columns ascend, so the k-th set bit
// of the mask is entry qs + k).  A binary search narrows long rows; the entries are
// then read eight at a time with independent loads.
__device__ __forceinline__ void row_tile_support(const int* __restrict__ rp, const int* __restrict__ ci, int g, int j0,
                                                 uint4& mask, int& qs) {
    uint32_t m0 = 0u, m1 = 0u, m2 = 0u, m3 = 0u;
    int lo = rp[g];
    const int e = rp[g + 1];
    int hi = e;
    while (hi - lo > 8) {
        const int mid = (lo + hi) >> 1;
        if (ci[mid] < j0) lo = mid + 1;
        else hi = mid;
    }
    // lower_bound lies in [lo, hi]; entries before lo are < j0
    int q = lo;
    bool more = true;
    int first = -1;
    while (more) {
        int v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = q + u < e ? ci[q + u] : 0x7fffffff;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int c = v[u] - j0;
            if (first < 0 && v[u] >= j0) first = q + u;
            const uint32_t bit = (c >= 0 && c < kT) ? 1u << (c & 31) : 0u;
            const int w = c >> 5;
            m0 |= w == 0 ? bit : 0u;
            m1 |= w == 1 ? bit : 0u;
            m2 |= w == 2 ? bit : 0u;
            m3 |= w == 3 ? bit : 0u;
        }
        more = q + 8 < e && v[7] < j0 + kT;
        q += 8;
    }
    qs = first < 0 ? e : first;
    mask = make_uint4(m0, m1, m2, m3);
}

// Persistent pair kernel: one CTA per SM takes block pairs (I <= J) from a shared
// counter, in the pair list's order (bands of row blocks, so the pairs in flight
// across the GPU share their panels in L2).  For pair (I, J) it forms, in TMEM,
//   phase 0:  Y^T[I] X^T[J]^T = n Z[I, J]          (row r, column c: n Z_{I0+r, J0+c})
//   phase 1:  X^T[I] Y^T[J]^T = n Z[J, I]^T        (row r, column c: n Z_{J0+c, I0+r})
// so that the thread holding row r of the tile has both n Z_ij and n Z_ji of every
// pair (i, j) = (I0 + r, J0 + c) in its registers: the transpose of Alg. 3 step 6
// costs nothing, and the screening test and the emission of both (i, j) and (j, i)
// happen in one thread.
//
// Chunked accumulation, as in the Gram: the K loop of a pair is cut into chunks
// (chunk_start), each chunk accumulates both tiles from zero into one TMEM
// accumulator pair, and the epilogue adds the chunk sums in FP32 round-to-nearest in
// registers, so the bias of the tensor core's truncating accumulation scales with
// the chunk, not with n.
//
// Roles:
//   warp 0      thread 0: takes the CTA's next pair from the counter, publishes it in
//               a ring of kRing pair slots, and streams per chunk the stages of
//               (Y^T[I], X^T[J]), then of (X^T[I], Y^T[J]) through TMA;
//   warp 1      MMA issuer (thread 32) and TMEM owner: chunk c of the CTA's sequence
//               into accumulator pair c & 1 (columns 256 (c & 1) + {0, 128});
//   warps 2-3   the support of the pair's rows in its columns (row_tile_support),
//               into the slot's masks, ahead of the epilogue;
//   warps 4-11  running sums (warp w: TMEM lanes 32 (w % 4) .. + 31, one row per
//               thread; warps 4-7 columns 0-63, warps 8-11 columns 64-127 of both
//               tiles), then the screening test and the emission.
// pair_full / pair_empty hand the pair slots around, sup_full the masks, acc_full /
// acc_empty the accumulator pairs.  Every wait is bounded; after an abort every
// role stops, the loads in flight drain and TMEM is freed.
//
// Only the pairs of ob.sel are taken (see k_obs_list); each leaves the largest |n Z_ij|
// and |n Z_ji| that it found in ob.b.  The K steps whose 16 (TF32: 8) elements are all padding
// are left out: at n = 100 one step in eight.  Every stage holds samples (k_tiles counts no
// stage of padding alone), so that a chunk's first step, which resets its accumulator, runs.
template <int MODE>
__global__ void __launch_bounds__(kObsThreads, 1)
k_obs_pair(const __grid_constant__ CUtensorMap ya, const __grid_constant__ CUtensorMap yb,
           const __grid_constant__ CUtensorMap xa, const __grid_constant__ CUtensorMap xb, const int2* __restrict__ pairs,
           const ObsBounds ob, float eps, int k_tiles, int p, int64_t n, const int* __restrict__ rp, const int* __restrict__ ci,
           const float* __restrict__ cv, Emit<float> em, Ctrl* __restrict__ ctrl, int chunk_kt, int lead_kt) {
    using C = ObsCfg<MODE>;
    constexpr int R = C::kRing;
    const float lam1 = (float)ctrl->lam1;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint4* s_mask = reinterpret_cast<uint4*>(smem + C::kStages * C::kStageBytes);           // [R][kT]
    int* s_qs = reinterpret_cast<int*>(s_mask + R * kT);                                   // [R][kT]
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kStages * C::kStageBytes + C::kSupBytes);
    uint64_t* empty = full + C::kStages;
    uint64_t* acc_full = empty + C::kStages;     // [2]
    uint64_t* acc_empty = acc_full + 2;          // [2]
    uint64_t* pair_full = acc_empty + 2;         // [R]
    uint64_t* pair_empty = pair_full + R;        // [R]
    uint64_t* sup_full = pair_empty + R;         // [R]
    int2* s_pair = reinterpret_cast<int2*>(sup_full + R);                                  // [R]
    int* s_id = reinterpret_cast<int*>(s_pair + R);                                        // [R]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_id + R);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    static_assert(8 * (2 * C::kStages + 4 + 3 * R) + 12 * R + 8 <= C::kCtlBytes, "control area");
    static_assert(C::kSmem <= 232448, "shared memory per block");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (chunk_kt < 1) chunk_kt = 1;
    if (lead_kt < chunk_kt) lead_kt = chunk_kt;
    const int nch = num_chunks(k_tiles, chunk_kt, lead_kt);
    // without bounds (ob.b null) every pair is taken
    const bool bounded = ob.b != nullptr;
    const int npairs = bounded ? __ldcg(ob.count) : ob.npairs;

    // this pass's norms and eps become the last pass's, and the maxima start at 0 again
    if (bounded && blockIdx.x == 0 && threadIdx.x == 0) *ob.eps_prev = eps;
    for (int t = blockIdx.x * kObsThreads + threadIdx.x; bounded && t < ob.nb; t += gridDim.x * kObsThreads) {
        ob.yprev[t] = ob.y[t];
        ob.s[t] = ob.r[t] = ob.y[t] = 0u;
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; ++s) { ptx::mbar_init(&full[s], 1); ptx::mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { ptx::mbar_init(&acc_full[b], 1); ptx::mbar_init(&acc_empty[b], kEpiWarps); }
        for (int s = 0; s < R; ++s) {
            ptx::mbar_init(&pair_full[s], 1);
            ptx::mbar_init(&pair_empty[s], 1 + 2 + kEpiWarps);      // MMA issuer, helper warps, epilogue warps
            ptx::mbar_init(&sup_full[s], kHelpThreads);
        }
        *abort_flag = 0;
        ptx::mbar_init_fence();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 2 * kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    long long issued = 0;
    if (warp < 4) {
        // producer, MMA issuer and the helpers: one warpgroup that gives registers away
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsSmall));
        if (threadIdx.x == 0) {
            // ---------------- scheduler and producer
            // Pairs are published kLook ahead of the loads, so that the counter's and the
            // pair list's latency, and the helpers' mask work, stay off the MMA's path.
            long long g = 0;
            bool ok = true, pub_done = false;
            int pub = 0;
            int nxt = atomicAdd(&ctrl->obs_next, 1);
            auto publish = [&]() -> bool {
                const int slot = pub % R;
                if (!ptx::mbar_wait_bounded(&pair_empty[slot], ((uint32_t)(pub / R) & 1u) ^ 1u, abort_flag,
                                            kWaitLimit))
                    return false;
                const int idx = nxt;
                const int id = idx >= npairs ? -1 : bounded ? ob.sel[idx] : idx;
                const int2 pr = id >= 0 ? pairs[id] : make_int2(-1, -1);
                if (idx < npairs) nxt = atomicAdd(&ctrl->obs_next, 1);
                s_pair[slot] = pr;
                s_id[slot] = id;
                ptx::mbar_arrive(&pair_full[slot]);
                ++pub;
                pub_done = pr.x < 0;
                return true;
            };
            for (int q = 0; q < C::kLook && ok && !pub_done; ++q) ok = publish();
            for (int t = 0; ok && t < pub; ++t) {
                const int2 pr = s_pair[t % R];
                if (pr.x < 0) break;
                if (!pub_done && !publish()) break;            // pair t + kLook
                const int I0 = pr.x * kT, J0 = pr.y * kT;
                for (int c = 0; c < nch && ok; ++c) {
                    const int kt0 = chunk_start(c, k_tiles, chunk_kt, lead_kt);
                    const int kt1 = chunk_start(c + 1, k_tiles, chunk_kt, lead_kt);
                    for (int phase = 0; phase < 2 && ok; ++phase) {
                        // phase 0: A = Y^T[I], B = X^T[J]; phase 1: A = X^T[I], B = Y^T[J]
                        const CUtensorMap* ma = phase == 0 ? &ya : &xa;
                        const CUtensorMap* mb = phase == 0 ? &xa : &ya;
                        const CUtensorMap* la = phase == 0 ? &yb : &xb;
                        const CUtensorMap* lb = phase == 0 ? &xb : &yb;
                        for (int kt = kt0; kt < kt1; ++kt, ++g) {
                            const int s = (int)(g % C::kStages);
                            const uint32_t ph = (uint32_t)(g / C::kStages) & 1u;
                            if (!ptx::mbar_wait_bounded(&empty[s], ph ^ 1u, abort_flag, kWaitLimit)) {
                                ok = false;
                                break;
                            }
                            uint8_t* st = smem + s * C::kStageBytes;
                            ptx::mbar_expect_tx(&full[s], C::kStageBytes);
                            const int kc = kt * C::kBK;
                            ptx::tma_load_2d(st, ma, &full[s], kc, I0);
                            ptx::tma_load_2d(st + kPanelTile, mb, &full[s], kc, J0);
                            if (C::kPieces > 1) {
                                ptx::tma_load_2d(st + 2 * kPanelTile, la, &full[s], kc, I0);
                                ptx::tma_load_2d(st + 3 * kPanelTile, lb, &full[s], kc, J0);
                            }
                            ++issued;
                        }
                    }
                }
            }
        } else if (threadIdx.x == 32) {
            // ---------------- MMA issuer
            constexpr uint32_t idesc = instr_desc<MODE>();
            long long g = 0, gc = 0;
            bool ok = true;
            for (int t = 0; ok; ++t) {
                const int slot = t % R;
                if (!ptx::mbar_wait_bounded(&pair_full[slot], (uint32_t)(t / R) & 1u, abort_flag, kWaitLimit)) break;
                const int2 pr = s_pair[slot];
                ptx::mbar_arrive(&pair_empty[slot]);
                if (pr.x < 0) break;
                for (int c = 0; c < nch && ok; ++c, ++gc) {
                    const int b = (int)(gc & 1);
                    if (!ptx::mbar_wait_bounded(&acc_empty[b], ((uint32_t)(gc >> 1) & 1u) ^ 1u, abort_flag,
                                                kWaitLimit)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const int kt0 = chunk_start(c, k_tiles, chunk_kt, lead_kt);
                    const int kt1 = chunk_start(c + 1, k_tiles, chunk_kt, lead_kt);
                    for (int phase = 0; phase < 2 && ok; ++phase) {
                        const uint32_t d = tmem + (uint32_t)(b * 2 * kT + phase * kT);
                        for (int kt = kt0; kt < kt1; ++kt, ++g) {
                            const int s = (int)(g % C::kStages);
                            const uint32_t ph = (uint32_t)(g / C::kStages) & 1u;
                            if (!ptx::mbar_wait_bounded(&full[s], ph, abort_flag, kWaitLimit)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const uint32_t st = ptx::smem_u32(smem + s * C::kStageBytes);
                            const uint32_t a_hi = st, b_hi = st + kPanelTile, a_lo = st + 2 * kPanelTile,
                                           b_lo = st + 3 * kPanelTile;
                            const int steps = (int)min((int64_t)(C::kBK / C::kMmaK),
                                                       (n - (int64_t)kt * C::kBK + C::kMmaK - 1) / C::kMmaK);
#pragma unroll
                            for (int kk = 0; kk < C::kBK / C::kMmaK; ++kk) {
                                if (kk >= steps) break;
                                const uint32_t off = kk * 32;
                                const uint32_t acc0 = (kt > kt0 || kk > 0) ? 1u : 0u;
                                umma<MODE>(d, smem_desc_sw128(a_hi + off), smem_desc_sw128(b_hi + off), idesc, acc0);
                                if constexpr (C::kTerms == 3) {
                                    umma<MODE>(d, smem_desc_sw128(a_hi + off), smem_desc_sw128(b_lo + off), idesc, 1u);
                                    umma<MODE>(d, smem_desc_sw128(a_lo + off), smem_desc_sw128(b_hi + off), idesc, 1u);
                                }
                            }
                            umma_commit(&empty[s]);
                        }
                    }
                    if (ok) umma_commit(&acc_full[b]);
                }
            }
        } else if (warp >= 2) {
            // ---------------- support masks of the pair's rows (two rows per thread)
            const int ht = threadIdx.x - 64;
            for (int t = 0;; ++t) {
                const int slot = t % R;
                if (!ptx::mbar_wait_bounded(&pair_full[slot], (uint32_t)(t / R) & 1u, abort_flag, kWaitLimit)) break;
                const int2 pr = s_pair[slot];
                if (pr.x < 0) break;
                const int I0 = pr.x * kT, J0 = pr.y * kT;
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2) {
                    const int rr = ht + kHelpThreads * h2;
                    const int g = I0 + rr;
                    uint4 m = make_uint4(0u, 0u, 0u, 0u);
                    int qs = 0;
                    if (g < p) row_tile_support(rp, ci, g, J0, m, qs);
                    s_mask[slot * kT + rr] = m;
                    s_qs[slot * kT + rr] = qs;
                }
                ptx::mbar_arrive(&sup_full[slot]);
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&pair_empty[slot]);
            }
        }
    } else {
        // the epilogue warpgroups take them: 2 x 64 running sums live in registers
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
        // ---------------- epilogue
        // Thread (q4, lane) of warp w owns row r = 32 q4 + lane of the tile (g = I0 + r)
        // and the columns c0 .. c0 + 63 (c0 = 64 half).  For each column it holds
        // a = n Z_ij and b = n Z_ji (j = J0 + c).  The pair {(i, j), (j, i)} is emitted
        // when it is in the support, on the diagonal, or when |a| or |b| exceeds lambda1 n;
        // (i, j) carries a / n and (j, i) carries b / n, both flagged as paired (each is the
        // other's partner) and both with w_ij (the iterate is symmetric).  In a diagonal
        // pair (I = J) each thread emits only its own row's entry: (j, i) is the row of
        // another thread of the same tile.
        const int q4 = warp & 3;
        const int half = (warp - 4) >> 2;
        const int r = q4 * 32 + lane;
        const int c0 = half * 64;
        const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0;
        // Z = (Y X) / n: the sums are tested against lambda1 n and only the emitted entries
        // are scaled.  The threshold is lowered by 2^-20 relative, so that the entries
        // emitted include every one whose scaled value exceeds lambda1 in FP32; an extra
        // entry at the threshold is harmless (its prox step leaves it at zero).
        const float inv_n = 1.0f / (float)n;
        const float thr = (float)((double)lam1 * (double)n * (1.0 - 0x1p-20));
        long long gc = 0;
        for (int t = 0;; ++t) {
            const int slot = t % R;
            const uint32_t rph = (uint32_t)(t / R) & 1u;
            bool got = !*abort_flag && ptx::mbar_wait_bounded(&pair_full[slot], rph, abort_flag, kWaitLimit);
            got = __all_sync(kFull, got);
            if (!got) break;
            const int2 pr = s_pair[slot];
            if (pr.x < 0) break;
            const int I0 = pr.x * kT, J0 = pr.y * kT;
            const bool diag_pair = pr.x == pr.y;
            const int g = I0 + r;
            float za[64], zb[64];
            bool have = true;
            for (int c = 0; c < nch; ++c, ++gc) {
                const int b = (int)(gc & 1);
                bool ok = have && !*abort_flag &&
                          ptx::mbar_wait_bounded(&acc_full[b], (uint32_t)(gc >> 1) & 1u, abort_flag, kWaitLimit);
                ok = __all_sync(kFull, ok);
                if (!ok) { have = false; continue; }
                tc_fence_after();
#pragma unroll
                for (int s4 = 0; s4 < 4; ++s4) {
                    uint32_t va[16], vb[16];
                    tmem_ld16(lane_base + (uint32_t)(b * 2 * kT + s4 * 16), va);
                    tmem_ld16(lane_base + (uint32_t)(b * 2 * kT + kT + s4 * 16), vb);
                    tmem_ld_wait();
                    if (c == 0) {
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            za[s4 * 16 + q] = __uint_as_float(va[q]);
                            zb[s4 * 16 + q] = __uint_as_float(vb[q]);
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            za[s4 * 16 + q] += __uint_as_float(va[q]);
                            zb[s4 * 16 + q] += __uint_as_float(vb[q]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx_arrive(&acc_empty[b]);
            }
            if (!have) break;
            bool sok = ptx::mbar_wait_bounded(&sup_full[slot], rph, abort_flag, kWaitLimit);
            sok = __all_sync(kFull, sok);
            if (!sok) break;
            const uint4 m4 = s_mask[slot * kT + r];
            const int qs = s_qs[slot * kT + r];
            const uint32_t sm[2] = {half ? m4.z : m4.x, half ? m4.w : m4.y};
            const int before0 = half ? __popc(m4.x) + __popc(m4.y) : 0;
            const bool mine = g < p;
            // the pair's largest |n Z| as integers, which order non-negative floats and put NaN last
            if (bounded) {
                uint32_t mx = 0u;
#pragma unroll
                for (int q = 0; q < 64; ++q)
                    mx = max(mx, max(__float_as_uint(za[q]) & 0x7fffffffu, __float_as_uint(zb[q]) & 0x7fffffffu));
                mx = __reduce_max_sync(kFull, mx);
                if (lane == 0) atomicMax(reinterpret_cast<unsigned*>(ob.b) + s_id[slot], mx);
            }
            uint32_t eb[2];
            int cnt = 0;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                uint32_t w = 0u;
#pragma unroll
                for (int q = 0; q < 32; ++q) {
                    const bool big = !(fabsf(za[32 * k + q]) <= thr) || !(fabsf(zb[32 * k + q]) <= thr);
                    w |= (uint32_t)big << q;
                }
                w |= sm[k];
                const int lim = p - (J0 + c0 + 32 * k);                 // columns J0 + c0 + 32 k + q < p
                if (lim < 32) w &= lim > 0 ? (1u << lim) - 1u : 0u;
                if (diag_pair && (r >> 5) == 2 * half + k) w |= 1u << (r & 31);      // the diagonal
                eb[k] = mine ? w : 0u;
                cnt += __popc(eb[k]);
            }
            if (!diag_pair) cnt *= 2;
            // one atomic per warp: an inclusive scan of the lanes' counts, the last lane takes
            // the warp's total from the emission counter and every lane writes from its offset
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += v;
            }
            int base = 0;
            if (lane == 31 && incl > 0) base = atomicAdd(&ctrl->em_count, incl);
            base = __shfl_sync(kFull, base, 31);
            int pos = base + incl - cnt;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                uint32_t bits = eb[k];
                const uint32_t sw = sm[k];
                const int before = before0 + (k ? __popc(sm[0]) : 0);
                while (bits) {
                    const int q = __ffs(bits) - 1;
                    bits &= bits - 1u;
                    const int j = J0 + c0 + 32 * k + q;
                    const bool sup = (sw >> q) & 1u;
                    const float om = sup ? cv[qs + before + __popc(sw & ((1u << q) - 1u))] : 0.f;
                    const unsigned fl = 0x40000000u | (sup ? 0x80000000u : 0u);
                    if (pos < em.cap) {
                        em.row[pos] = g;
                        em.col[pos] = (int)((unsigned)j | fl);
                        em.w[pos] = __fmul_rn(k ? pick32<32>(za, q) : pick32<0>(za, q), inv_n);
                        em.om[pos] = om;
                    }
                    ++pos;
                    if (!diag_pair) {
                        if (pos < em.cap) {
                            em.row[pos] = j;
                            em.col[pos] = (int)((unsigned)g | fl);
                            em.w[pos] = __fmul_rn(k ? pick32<32>(zb, q) : pick32<0>(zb, q), inv_n);
                            em.om[pos] = om;
                        }
                        ++pos;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&pair_empty[slot]);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) {
            atomicOr(&ctrl->flags, kFlagTimeout);
            if (bounded) *ob.poison = 1;
            for (long long g = issued > C::kStages ? issued - C::kStages : 0; g < issued; ++g) {
                const int s = (int)(g % C::kStages);
                const uint32_t ph = (uint32_t)(g / C::kStages) & 1u;
                for (long long it = 0; it < (1ll << 22) && !ptx::mbar_try_wait(&full[s], ph); ++it) __nanosleep(64);
            }
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 2 * kTmemCols);
    }
}

// ---------------------------------------------------------------- which block pairs a pass needs
// A pass over all block pairs is 2 p^2 n products (times three in BF16X3) however little Omega
// has moved: about 1 ms at p = 40000, n = 100, every iteration.  But a pair emits nothing unless
// it holds support or a |Z_ij| above lambda1, and near the estimate Z hardly moves.  So each
// pair keeps a certified bound of the largest |n Z_ij|, |n Z_ji| in it, and a pass takes only
// the pairs on the diagonal, with an off-diagonal support entry, or whose bound exceeds the
// threshold: the emitted entries are those of a full pass.
//
// With y_i the stored FP32 rows of Y^T and n z_ij = <y_i, x_j> exactly:
//   y_i = s_i y_i(last pass) + d_i with s_i = w_ii / w_ii(last pass), so that a row with the
//   diagonal alone has d_i = 0 up to rounding, and |n z_ij| <= |s_i| |n z_ij(last)| + |d_i| |x_j|;
//   the tensor product differs from n z_ij by at most eps |y_i| |x_j| (obs_eps).
// Per 128-row block the largest |s_i|, |d_i|, |y_i| and |x_j| stand for all rows; every operation
// rounds up (the norms carry 1% for their FP32 sums).  NaN and infinities make a bound that no
// comparison passes: such pairs are taken.
// Measured on GB300, solves in ms, without and with bounds: p = 24000, n = 100, lambda1 = 0.55
// 16.4 -> 12.0; p = 24000, n = 130, lambda1 = 0.46 21.6 -> 16.1; p = 12000, n = 100 8.3 -> 7.9
// (7.2, 10.8 and 4.8 with the line search's later form);
// p = 40000, n = 100, lambda1 = 0.46, where nearly every pair holds an entry to emit, the same.

// position of block pair (I, J), I <= J, in obs_pair_list's order
__host__ __device__ __forceinline__ long long obs_pair_index(int I, int J, int nb) {
    const int b0 = I / kObsBand * kObsBand, hb = nb - b0 < kObsBand ? nb - b0 : kObsBand, c = J - b0;
    const long long before = (long long)b0 * nb - (long long)b0 * (b0 - 1) / 2;
    return before + (c <= hb ? (long long)c * (c + 1) / 2 : hb * (hb + 1) / 2 + (long long)(c - hb) * hb) + (I - b0);
}

__device__ __forceinline__ float warp_sum_up(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

template <int MODE>
__device__ __forceinline__ void split_store(float x, void* hi, void* lo, int64_t t) {
    if constexpr (MODE == kObsTf32) {
        uint32_t u;
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
        static_cast<float*>(hi)[t] = __uint_as_float(u);
    } else {
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        static_cast<__nv_bfloat16*>(hi)[t] = h;
        static_cast<__nv_bfloat16*>(lo)[t] = __float2bfloat16_rn(x - __bfloat162float(h));
    }
}

// Y^T = Omega X^T in k_spmm_dense's order (w_ii x_i first, then the neighbours ascending), its
// panels, and the bounds' |s_i|, |d_i|, |y_i| per block of rows.  Warp per row; ld = n padded
// to 64, the padding of X^T is zero.  Four neighbours' rows are in flight: the passes of a dense
// iterate, up to 1500 neighbours a row, took 0.46 ms with one, 0.24 with four (p = 40000).
template <int MODE>
__global__ void __launch_bounds__(256)
k_obs_rows(int p, int64_t rows_pad, Csr<float> om, const int4* __restrict__ rinfo, const float* __restrict__ rdv,
           const float* __restrict__ xt, int64_t ld, float* __restrict__ yt, void* hi, void* lo, const ObsBounds ob) {
    __shared__ unsigned m[3];
    const int lane = threadIdx.x & 31;
    const int64_t i = blockIdx.x * 8ll + (threadIdx.x >> 5);
    if (threadIdx.x < 3) m[threadIdx.x] = 0u;
    __syncthreads();
    if (i < p) {
        const int4 info = rinfo[i];
        const float dv = rdv[i], s = __fdiv_rn(dv, ob.dold[i]);
        float d2 = 0.f, y2 = 0.f;
        for (int64_t c0 = lane; c0 < ld; c0 += 128) {
            float acc[4], old[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int64_t c = c0 + 32 * v;
                acc[v] = c < ld ? __fmul_rn(dv, xt[i * ld + c]) : 0.f;
                old[v] = c < ld ? yt[i * ld + c] : 0.f;
            }
            for (int q0 = info.x; q0 < info.y; q0 += 4) {       // four neighbours' rows in flight
                float w[4], x[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int q = q0 + u;
                    const bool on = q < info.y && q != info.z;
                    const int64_t k = on ? om.ci[q] : 0;
                    w[u] = on ? om.cv[q] : 0.f;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int64_t c = c0 + 32 * v;
                        x[u][v] = on && c < ld ? xt[k * ld + c] : 0.f;
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (q0 + u >= info.y || q0 + u == info.z) continue;
#pragma unroll
                    for (int v = 0; v < 4; ++v) acc[v] = __fmaf_rn(w[u], x[u][v], acc[v]);
                }
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int64_t c = c0 + 32 * v;
                if (c < ld) {
                    yt[i * ld + c] = acc[v];
                    split_store<MODE>(acc[v], hi, lo, i * ld + c);
                    const float d = __fmaf_rn(-s, old[v], acc[v]);
                    d2 = __fmaf_rn(d, d, d2);
                    y2 = __fmaf_rn(acc[v], acc[v], y2);
                }
            }
        }
        d2 = warp_sum_up(d2);
        y2 = warp_sum_up(y2);
        if (lane == 0) {
            ob.dold[i] = dv;
            // 1e-18: squares below the smallest float
            atomicMax(&m[0], __float_as_uint(fabsf(s)));
            atomicMax(&m[1], __float_as_uint(__fmaf_ru(sqrtf(d2), 1.01f, 1e-18f)));
            atomicMax(&m[2], __float_as_uint(__fmaf_ru(sqrtf(y2), 1.01f, 1e-18f)));
        }
    } else if (i < rows_pad) {
        for (int64_t c = lane; c < ld; c += 32) split_store<MODE>(0.f, hi, lo, i * ld + c);
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        unsigned* out = threadIdx.x == 0 ? ob.s : threadIdx.x == 1 ? ob.r : ob.y;
        const unsigned v = m[threadIdx.x] & 0x7fffffffu;
        if (v) atomicMax(out + blockIdx.x * 8 / kT, v);
    }
}

// the largest |x_j| of each 128-row block of X^T
__global__ void __launch_bounds__(256) k_obs_norms(int p, const float* __restrict__ xt, int64_t ld, unsigned* nx) {
    const int lane = threadIdx.x & 31;
    const int64_t i = blockIdx.x * 8ll + (threadIdx.x >> 5);
    if (i >= p) return;
    float x2 = 0.f;
    for (int64_t c = lane; c < ld; c += 32) x2 = __fmaf_rn(xt[i * ld + c], xt[i * ld + c], x2);
    x2 = warp_sum_up(x2);
    if (lane == 0) atomicMax(nx + i / kT, __float_as_uint(__fmaf_ru(sqrtf(x2), 1.01f, 1e-18f)) & 0x7fffffffu);
}

// the block pairs with an off-diagonal support entry; warp per row
__global__ void __launch_bounds__(256) k_obs_mark(int p, const int* __restrict__ rp, const int* __restrict__ ci,
                                                  const ObsBounds ob) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *ob.count = 0;
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= p) return;
    const int I = i / kT;
    for (int q = rp[i] + lane; q < rp[i + 1]; q += 32) {
        const int J = ci[q] / kT;
        if (J > I) ob.mark[obs_pair_index(I, J, ob.nb)] = 1;
    }
}

// The pairs to take, a thread per pair.
__global__ void __launch_bounds__(256) k_obs_list(const int2* __restrict__ pairs, int npairs, int64_t n, float eps,
                                                  const ObsBounds ob, const Ctrl* __restrict__ ctrl) {
    const float thr = (float)((double)(float)ctrl->lam1 * (double)n * (1.0 - 0x1p-20));     // k_obs_pair's
    const int lane = threadIdx.x & 31;
    const bool all = *ob.poison != 0;
    const float eps_prev = *ob.eps_prev;
    for (int64_t t0 = blockIdx.x * 256ll; t0 < npairs; t0 += gridDim.x * 256ll) {
        const int64_t t = t0 + threadIdx.x;
        bool take = false;
        if (t < npairs) {
            const int2 pr = pairs[t];
            const int I = pr.x, J = pr.y;
            const float nxi = __uint_as_float(ob.nx[I]), nxj = __uint_as_float(ob.nx[J]);
            // the larger of a[I] |x|_J and a[J] |x|_I, NaN kept
            auto cross = [&](const unsigned* a) {
                const float u = __fmul_ru(__uint_as_float(a[I]), nxj), v = __fmul_ru(__uint_as_float(a[J]), nxi);
                return __uint_as_float(max(__float_as_uint(u) & 0x7fffffffu, __float_as_uint(v) & 0x7fffffffu));
            };
            float b = ob.b[t];
            if (ob.fresh[t]) b = __fmaf_ru(eps_prev, cross(ob.yprev), b);
            b = __fmaf_ru(__uint_as_float(max(ob.s[I], ob.s[J])), b, cross(ob.r));
            take = all || I == J || ob.mark[t] || !(__fmaf_ru(eps, cross(ob.y), b) <= thr);
            ob.mark[t] = 0;
            ob.fresh[t] = take;
            ob.b[t] = take ? 0.f : b;
        }
        const unsigned vote = __ballot_sync(kFull, take);
        int at = 0;
        if (lane == 0 && vote) at = atomicAdd(ob.count, __popc(vote));
        at = __shfl_sync(kFull, at, 0);
        if (take) ob.sel[at + __popc(vote & ((1u << lane) - 1u))] = (int)t;
    }
}

// FP32 rows (rows x ldi, K contiguous) -> K-major panels (rows_pad x n_pad) of the MMA input type.
template <int MODE>
__global__ void k_obs_split(const float* __restrict__ in, int64_t rows, int64_t cols, int64_t ldi, void* hi, void* lo,
                            int64_t rows_pad, int64_t n_pad) {
    const int64_t total = rows_pad * n_pad;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / n_pad, k = t % n_pad;
        const float x = (r < rows && k < cols) ? in[r * ldi + k] : 0.f;
        split_store<MODE>(x, hi, lo, t);
    }
}

}  // namespace

// ---------------------------------------------------------------- host side
size_t obs_panel_bytes(int precision, int64_t n, int64_t p) {
    const int64_t p_pad = (p + kT - 1) / kT * kT, n_pad = (n + 63) / 64 * 64;
    const int es = precision == HPC_PREC_TF32 ? 4 : 2;
    return ((size_t)p_pad * n_pad * es + 1023) / 1024 * 1024;
}

int obs_pieces(int precision) { return precision == HPC_PREC_TF32 ? 1 : 2; }

int64_t obs_npairs(int64_t p) {
    const int64_t nb = (p + kT - 1) / kT;
    return nb * (nb + 1) / 2;
}

void obs_pair_list(int64_t p, std::vector<int2>& out) {
    const int64_t nb = (p + kT - 1) / kT;
    out.clear();
    // bands of kObsBand row blocks, columns left to right: pairs in flight share panels in L2
    for (int64_t b0 = 0; b0 < nb; b0 += kObsBand)
        for (int64_t bj = 0; bj < nb; ++bj)
            for (int64_t bi = b0; bi < std::min<int64_t>(b0 + kObsBand, nb); ++bi)
                if (bi <= bj) out.push_back(make_int2((int)bi, (int)bj));
}

void launch_obs_split(int precision, const float* in, int64_t rows, int64_t cols, int64_t ldi, void* hi, void* lo,
                      int64_t n, int64_t p, cudaStream_t s) {
    const int64_t rows_pad = (p + kT - 1) / kT * kT, n_pad = (n + 63) / 64 * 64;
    if (precision == HPC_PREC_TF32)
        k_obs_split<kObsTf32><<<2048, 256, 0, s>>>(in, rows, cols, ldi, hi, lo, rows_pad, n_pad);
    else
        k_obs_split<kObsBf16x3><<<2048, 256, 0, s>>>(in, rows, cols, ldi, hi, lo, rows_pad, n_pad);
}

bool obs_make_maps(int precision, const void* y_hi, const void* y_lo, const void* x_hi, const void* x_lo, int64_t n,
                   int64_t p, CUtensorMap* maps /*4: ya, yb, xa, xb*/) {
    const int64_t p_pad = (p + kT - 1) / kT * kT, n_pad = (n + 63) / 64 * 64;
    const int es = precision == HPC_PREC_TF32 ? 4 : 2;
    const void* bases[4] = {y_hi, precision == HPC_PREC_TF32 ? y_hi : y_lo, x_hi,
                            precision == HPC_PREC_TF32 ? x_hi : x_lo};
    for (int t = 0; t < 4; ++t)
        if (!encode_tensor_map_2d_sw128(&maps[t], bases[t], es, (uint64_t)n_pad, (uint64_t)p_pad,
                                        (uint64_t)n_pad * es, (uint32_t)(kRowB / es), (uint32_t)kT))
            return false;
    return true;
}

// Stages of kbk elements that hold samples (the panels are padded to 64, two stages of TF32).
static int k_stages(int64_t n, int kbk) { return (int)((n + kbk - 1) / kbk); }
// K elements -> whole stages of kbk elements, at least one.
static int kt_of(int64_t k, int kbk) { return (int)std::max<int64_t>(1, std::min<int64_t>(k / kbk, 1 << 30)); }

// The tensor product's error over |y_i| |x_j|: the operands' rounding (BF16 hi + lo: 2^-18 each
// and lo lo left out, together below 2^-15; TF32: 2^-11 each, below 2^-9), and 2^-19 per
// accumulation step of the longest chunk (16 elements and up to three products; 17 terms, each
// cut at the largest one's last bit) and per chunk sum.
static float obs_eps(bool tf32, int64_t ldx, int64_t chunk_k, int64_t lead_k) {
    if (chunk_k <= 0) chunk_k = 256;
    if (lead_k <= 0) lead_k = 4 * chunk_k;
    const double k = (double)std::min<int64_t>(std::max(chunk_k, lead_k) + 64, ldx);
    const double steps = (tf32 ? k / 8 : 3 * k / 16) + (double)ldx / (double)chunk_k + 2;
    return (float)((tf32 ? 0x1p-9 : 0x1p-15) + steps * 0x1p-19);
}

// Bounds are kept from kObsBoundPairs block pairs on (p about 11500): below, a pass over all pairs
// takes less than the kernels that choose among them cost (p = 2000: 3.0 ms without, 3.2 with
// bounds; p = 6000 4.6, 4.6; p = 12000 8.3, 7.9).
constexpr int64_t kObsBoundPairs = 4096;
size_t obs_bounds_bytes(int64_t p) {
    if (obs_npairs(p) < kObsBoundPairs) return 0;
    const size_t nb = (size_t)(p + kT - 1) / kT, np = (size_t)obs_npairs(p);
    return (3 + 5 * nb + (size_t)p + 2 * np) * 4 + 2 * np;
}

ObsBounds obs_bounds(void* buf, int64_t p) {
    const size_t nb = (size_t)(p + kT - 1) / kT, np = (size_t)obs_npairs(p);
    ObsBounds ob{};
    unsigned* q = static_cast<unsigned*>(buf);
    auto take = [&](size_t k) { unsigned* r = q; q += k; return r; };
    ob.nb = (int)nb;
    ob.count = reinterpret_cast<int*>(take(1));
    ob.poison = reinterpret_cast<int*>(take(1));
    ob.eps_prev = reinterpret_cast<float*>(take(1));
    ob.nx = take(nb);
    ob.s = take(nb);
    ob.r = take(nb);
    ob.y = take(nb);
    ob.yprev = take(nb);
    ob.dold = reinterpret_cast<float*>(take((size_t)p));
    ob.b = reinterpret_cast<float*>(take(np));
    ob.sel = reinterpret_cast<int*>(take(np));
    ob.mark = reinterpret_cast<unsigned char*>(q);
    ob.fresh = ob.mark + np;
    return ob;
}

// After a load: |x_j|, and bounds that no comparison passes (NaN), so that the next pass takes
// every pair.
cudaError_t launch_obs_reset(void* buf, int64_t p, const float* xt, int64_t ldx, cudaStream_t s) {
    const ObsBounds ob = obs_bounds(buf, p);
    cudaError_t e = cudaMemsetAsync(buf, 0, obs_bounds_bytes(p), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(ob.b, 0xff, (size_t)obs_npairs(p) * sizeof(float), s);
    if (e != cudaSuccess) return e;
    k_obs_norms<<<(unsigned)((p + 7) / 8), 256, 0, s>>>((int)p, xt, ldx, ob.nx);
    return cudaGetLastError();
}

// Y^T, its panels, and the list of block pairs of this pass.
cudaError_t launch_obs_rows(int precision, int64_t n, int64_t p, Csr<float> om, const int4* rinfo, const float* rdv,
                            const float* xt, int64_t ldx, float* yt, void* hi, void* lo, void* bounds,
                            const int2* pairs, int64_t npairs, const Ctrl* ctrl, cudaStream_t s, int64_t chunk_k,
                            int64_t lead_k) {
    const ObsBounds ob = obs_bounds(bounds, p);
    const int64_t rows_pad = (p + kT - 1) / kT * kT;
    const unsigned nb = (unsigned)(rows_pad / 8);
    const bool tf32 = precision == HPC_PREC_TF32;
    if (tf32) k_obs_rows<kObsTf32><<<nb, 256, 0, s>>>((int)p, rows_pad, om, rinfo, rdv, xt, ldx, yt, hi, lo, ob);
    else k_obs_rows<kObsBf16x3><<<nb, 256, 0, s>>>((int)p, rows_pad, om, rinfo, rdv, xt, ldx, yt, hi, lo, ob);
    k_obs_mark<<<(unsigned)((p + 7) / 8), 256, 0, s>>>((int)p, om.rp, om.ci, ob);
    const float eps = obs_eps(tf32, ldx, chunk_k, lead_k);
    const unsigned lb = (unsigned)std::min<int64_t>((npairs + 255) / 256, 4096);
    k_obs_list<<<lb, 256, 0, s>>>(pairs, (int)npairs, n, eps, ob, ctrl);
    return cudaGetLastError();
}

cudaError_t launch_obs_pairs(int precision, const CUtensorMap* maps, const int2* pairs, int64_t npairs, void* bounds,
                             int64_t n,
                             int p, const int* rp, const int* ci, const float* cv, Emit<float> em,
                             Ctrl* ctrl, cudaStream_t s, int64_t chunk_k, int64_t lead_k) {
    const int64_t n_pad = (n + 63) / 64 * 64;
    ObsBounds ob{};
    if (bounds) ob = obs_bounds(bounds, p);
    ob.npairs = (int)npairs;
    const float eps = obs_eps(precision == HPC_PREC_TF32, n_pad, chunk_k, lead_k);
    // K elements per accumulation chunk (the Gram's BF16X3 / TF32 default when none is given)
    if (chunk_k <= 0) chunk_k = 256;
    if (lead_k <= 0) lead_k = 4 * chunk_k;
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                      cudaSuccess || sms < 1)
            sms = 1;
    }
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(npairs, sms));   // one CTA per SM
    // setmaxnreg moves registers between the warpgroups of a block: the kernel must have
    // been built with enough registers per thread for both shares (else it would wait)
    static int regs[2] = {-1, -1};
    const int mi = precision == HPC_PREC_TF32 ? 1 : 0;
    if (regs[mi] < 0) {
        cudaFuncAttributes fa;
        const cudaError_t e = cudaFuncGetAttributes(
            &fa, mi ? (const void*)k_obs_pair<kObsTf32> : (const void*)k_obs_pair<kObsBf16x3>);
        if (e != cudaSuccess) return e;
        regs[mi] = fa.numRegs;
    }
    if (regs[mi] < kMinLaunchRegs) return cudaErrorNotSupported;
    if (precision == HPC_PREC_TF32) {
        using C = ObsCfg<kObsTf32>;
        cudaError_t e = set_smem_once((const void*)k_obs_pair<kObsTf32>, C::kSmem, kSmemSlotObsTf32);
        if (e != cudaSuccess) return e;
        k_obs_pair<kObsTf32><<<grid, kObsThreads, C::kSmem, s>>>(maps[0], maps[1], maps[2], maps[3], pairs,
                                                                 ob, eps, k_stages(n, C::kBK), p, n, rp, ci,
                                                                 cv, em, ctrl, kt_of(chunk_k, C::kBK),
                                                                 kt_of(lead_k, C::kBK));
    } else {
        using C = ObsCfg<kObsBf16x3>;
        cudaError_t e = set_smem_once((const void*)k_obs_pair<kObsBf16x3>, C::kSmem, kSmemSlotObsBf16x3);
        if (e != cudaSuccess) return e;
        k_obs_pair<kObsBf16x3><<<grid, kObsThreads, C::kSmem, s>>>(maps[0], maps[1], maps[2], maps[3], pairs,
                                                                   ob, eps, k_stages(n, C::kBK), p, n, rp, ci,
                                                                   cv, em, ctrl, kt_of(chunk_k, C::kBK),
                                                                   kt_of(lead_k, C::kBK));
    }
    return cudaGetLastError();
}


}  // namespace hpc
