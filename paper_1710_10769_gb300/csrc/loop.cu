// The Cov iteration loop as one cooperative kernel (Alg. 1 with Alg. 2 steps 5-12):
// every outer iteration of a solve runs inside one launch, with three grid-wide
// barriers per iteration instead of about twenty dependent kernels.
//
// What bounds it.  At the iterates the estimator meets (a few entries per row) an
// iteration moves a few MB, so it is a chain of latencies: the kernels of the chain
// each cost 4-6 us of ramp, dependent loads and drain, and its candidate structure is
// built by seven of them (count, two scans, scatter, sort, partner fill, gradient).
// Here rows are owned: block b of the grid holds rows b R .. b R + R - 1 for the whole
// launch, and the steps are arranged so that a row's owner needs nothing from the
// other owners between barriers:
//
//   screen   support entries: W_ij and W_ji by gathers, a thread each.  Everything else: a
//            list of (row, column block) tasks, the blocks of 128 columns that can hold a
//            |W_ij| > lambda1 off the support: for a row with the diagonal alone, where
//            |w_ii| max|S_ij| over the block exceeds lambda1 (the block maxima are exact to
//            their BF16 rounding up); for a row with neighbours, where its certified bound
//            does.
//            Where |W_ij| > lambda1 off the support, the warp that met it also gathers
//            W_ji -- in the canonical order (diagonal term first, then the neighbours
//            ascending), so with the bits row j's own screening has -- and G_ij from the
//            two.  Only the entries a prox step can touch (the support, |G_ij| > lambda1)
//            go on, straight into the buckets of rows i and j (kSlots slots, then pages
//            of a pool; a cursor per row): no emission list, count, scan, scatter or
//            partner fill.  Of two rows that both meet the pair the lower one emits it.
//   -- barrier --
//   build    the owner sorts its rows' slots by column.
//   search   kWin step sizes of the line search on the owned rows (prox of eq. (2),
//            the partials of Alg. 1 step 9 in the expanded form, and the entries each
//            step size would keep).  Two windows at once when the last accepted step
//            needed more than one.  Partials per block.
//   -- barrier --
//   decide   every block reduces all blocks' partials in the same fixed order and
//            takes the same decision; the kept-entry counts of the blocks before it
//            give the block's first CSR position.
//   accept   the owner writes its rows of Omega+ (CSR), their set-up for the next
//            screening pass, the column maxima, the bounds of its rows with neighbours and
//            the tasks they leave.
//   -- barrier --
//
// The certified bounds.  bnd[i][jb] >= |W_ij| for every column j of block jb that is
// neither i nor in row i's support, for the exact product of the current iterate.  A row
// that gains its first neighbour starts from sum_t |w_t| m1[k_t][jb] (m1: block maxima,
// column k_t itself left out of row k_t's).  A step that changes the row by D adds
// sum_t |D_t| m1[k_t][jb]; a column that leaves the support sets its block's bound to
// infinity.  Screening a block replaces its bound by the largest |W_ij| found plus a
// rounding term.  The computed W differs from the exact one by at most
// gamma_m sum_t |w_t| max|S| (m terms, gamma_m = m u / (1 - m u)), which is added where a
// bound is set and again where it is tested; every operation rounds up.  So a block
// that is left out has no |fl(W_ij)| > lambda1: the emitted set is that of a full pass,
// while near convergence, where D is small, a pass reads little more than the support.
// (The bounds without this memory keep nearly every block once lambda1 is near the noise
// of S: at p = 8192, lambda1 = 0.05 a pass then reads 1.7 GB of S.)
//
// A row that collects more than kMaxE - 2 candidates, or more pages than the pool has, or a pass
// that the chain does faster (dense iterates and hub rows, see in_debt) ends the launch with
// Ctrl::loop_full set and the iterate unchanged; the chain of kernels then runs the next
// iterations (one at first, twice as many after every further end of this kind) before the loop
// tries again.  An iterate that is not symmetric (hpc_set_omega takes any) is the chain's
// altogether: a column could come twice into a row's bucket, and the chain removes such duplicates.
// No phase of a launch is long, then, which the bounded waits need.
//
// Measured on GB300 (us per iteration, the chain of kernels -> this loop): 140 -> 46 at
// p = 65536 (n = 32768), 120 -> 41 at p = 16384, 98 -> 29 at p = 1001, 220 -> 47 in FP64 at
// p = 500; the 32-point path at p = 8192 from 163 to 52 ms.  Of the 41 us at p = 16384 the screening
// takes 10, the build 4, the search with its decision 16, the accept 11; at the path's
// smallest lambda1 the screening takes 200 of 310.  What is left is the latency of the steps'
// dependent loads and of the three barriers (about 2 us each).
//
// Every wait is bounded (kBarrierWaitNs), after which kFlagTimeout is raised and every
// block leaves.  The cooperative launch keeps all blocks resident (one per SM).
#include <algorithm>
#include <type_traits>
#include <vector>

#include "iter_common.cuh"

namespace hpc {
namespace {

constexpr int kLW = 16;                  // warps per block
constexpr int kLT = kLW * 32;            // threads per block
constexpr int kSlots = 128;              // slots of a row's bucket, and of a page
constexpr int kPages = 16;               // pages per row, the bucket itself among them
constexpr int kMaxE = kPages * kSlots;
constexpr int kWin = 4;                  // step sizes per line-search window
constexpr int kItemCap = 4096;           // owned support entries kept in shared memory
constexpr int kHitCap = 64;              // entries waiting for their W_ji, per warp
constexpr int kMaxR = 2048;              // rows per block
constexpr int kHeavyTerms = 32;          // rows with more terms are screened by four warps a block
constexpr int kQA = 3 * kWin;            // accumulated partials per window: quadratic form, ||D||^2, phi
constexpr int kQI = 2 * kWin;            // counted partials per window: w+_ii <= 0, entries kept
constexpr int kNA = 2 * kQA + 1;         // and ||Omega||^2
constexpr int kNI = 2 * kQI + 5;         // and entries emitted, NaN / Inf, full rows, LoopSmem::halves, off

constexpr unsigned kColMask = 0x0fffffffu;
constexpr unsigned kFSupp = 0x80000000u;

// One candidate of a row: (column | support flag), w_ij, G_ij, W_ij.
template <typename T> struct alignas(sizeof(T) == 4 ? 16 : 32) Ent {
    unsigned cf;
    T om, g, w;
};

__device__ __forceinline__ Ent<float> ld_slot(const Ent<float>* q) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(q));
    return Ent<float>{v.x, __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w)};
}
__device__ __forceinline__ Ent<double> ld_slot(const Ent<double>* q) {
    const double2 a = __ldcg(reinterpret_cast<const double2*>(q));
    const double2 b = __ldcg(reinterpret_cast<const double2*>(q) + 1);
    return Ent<double>{(unsigned)__double_as_longlong(a.x), a.y, b.x, b.y};
}
__device__ __forceinline__ Ent<float> ld_ent(const Ent<float>* q) {
    const uint4 v = *reinterpret_cast<const uint4*>(q);
    return Ent<float>{v.x, __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w)};
}
__device__ __forceinline__ Ent<double> ld_ent(const Ent<double>* q) {
    const double2 a = reinterpret_cast<const double2*>(q)[0], b = reinterpret_cast<const double2*>(q)[1];
    return Ent<double>{(unsigned)__double_as_longlong(a.x), a.y, b.x, b.y};
}
__device__ __forceinline__ void st_ent(Ent<float>* q, unsigned cf, float om, float g, float w) {
    *reinterpret_cast<uint4*>(q) = make_uint4(cf, __float_as_uint(om), __float_as_uint(g), __float_as_uint(w));
}
__device__ __forceinline__ void st_ent(Ent<double>* q, unsigned cf, double om, double g, double w) {
    reinterpret_cast<double2*>(q)[0] = make_double2(__longlong_as_double((long long)cf), om);
    reinterpret_cast<double2*>(q)[1] = make_double2(g, w);
}

enum : int { kFullPool = 1, kFullDense = 2 };      // bits of kCtrFull
enum : int { kCtrPage, kCtrBig, kCtrFull, kCtrStart, kCtrCount };

template <typename T>
struct LoopK {
    const T* S;
    int64_t ld;
    int p, R;
    Csr<T> cur, next;
    int csr_cap, em_cap;
    Ent<T>* slots;       // p x kSlots: the buckets, in any order
    Ent<T>* ents;        // p x kSlots: sorted by column
    int* cnt;            // p: slot cursors
    int* len;            // p: candidates per row (0: only the diagonal, in ents[i kSlots])
    int4* rinfo;         // p: CSR bounds, diagonal position, pure flag
    T* rds;              // ld: w_jj, negated for the rows with neighbours
    int* pages;          // p x kPages: page numbers (from 1) of rows with more than kSlots slots
    Ent<T>* pool;        // npool x kSlots: the pages
    Ent<T>* big;         // as many entries: sorted candidates of those rows
    int npool;
    int* eoff;           // p: at the end, the row's place in `big` (-1: in ents)
    int* tasks;          // 2 x ntask_cap: row * nbm + block of the blocks to screen; from the
                         // back those of rows with more than 32 terms
    int ntask_cap;
    float* bnd;          // p x nbp: the certified bounds
    float* slack;        // p: the rounding term of the row
    int nbp;
    unsigned* mg;        // bits of max |S_ij|, i != j (rounded up)
    ulonglong2* todo;    // 2: tasks in the list, and of long rows: their number, and from bit 32 on their
                         // terms in units of 64
    int* ctr;            // counters: pages, entries of big, full rows (kCtrFull's bits), and whether the first
                         // pass is too dense (a word of its own: without bounds no barrier lies between
                         // the blocks' reads of it and the first pass's votes)
    double* part_a;      // 2 x kNA x grid
    int* part_i;         // 2 x kNI x grid
    unsigned* bar;
    Ctrl* ctrl;
    double eps;
    int max_halvings;
    const unsigned short* m1;    // block maxima (null: no bounds)
    const unsigned short* m1g;   // group maxima (null: none)
    int nbm, ngl;
    const unsigned long long* symmetric;     // 0: the iterate is not
    int use_cond;
    cudaGraphConditionalHandle chain_cond;   // set to 1 where the chain has to run next
    cudaGraphConditionalHandle outer_cond;   // the loop over both: ends here unless the chain runs
};

// Shared memory of a block, laid out by the host's sizes.
template <typename T>
struct LoopSmem {
    unsigned key[kLW][kSlots];          // a row's slots by column
    unsigned heavy[2][kLW];             // a quarter block's largest |W_ij|, per warp
    int hit_i[kLW][kHitCap];            // entries (i, j) waiting for W_ji
    int hit_j[kLW][kHitCap];
    T hit_w[kLW][kHitCap];
    T del[kLW][kWin][32];
    unsigned jf[kLW][32];
    double red_a[kLW][kNA];
    int red_i[kLW][kNI];
    double sum_a[kNA];
    int sum_i[kNI], pre_i[kNI];
    int items[kItemCap];                // owned support entries of rows with neighbours; keys of a long sort
    short item_r[kItemCap];             // their rows
    int ni, npl, nlong, nhuge, ok, e0, e1, pool_full;
    int wsum[kLW], wbig[kLW];
    int sup;                            // sum of n_i^2 / 64 over the owned rows of n_i entries
    unsigned debt, sup_debt;            // in_debt's; one thread's
    int leave[2];                       // outcomes of leave_support and leave_tasks
    int halves;                         // pairs of rows with the diagonal alone that have one entry above lambda1
    int off;                            // owned rows with neighbours
    int units;                          // pairs of 32-entry chunks of the rows with more than 32 candidates
    // the decision, the same in every block
    int flags, accept, nnz, nnz_pre, more, converged, full;
    double n2;
};

template <typename T>
__host__ __device__ constexpr size_t loop_smem_bytes(int R) {
    return (sizeof(LoopSmem<T>) + 15) / 16 * 16 + (size_t)R * (5 * sizeof(T) + 7 * sizeof(int)) + 16;
}

__device__ __forceinline__ double shfl_xor_acc(double x, int o) { return __shfl_xor_sync(kFull, x, o); }
__device__ __forceinline__ F2 shfl_xor_acc(const F2& x, int o) {
    F2 r;
    r.hi = __shfl_xor_sync(kFull, x.hi, o);
    r.lo = __shfl_xor_sync(kFull, x.lo, o);
    return r;
}

// Quantity t summed over the block's warps, a fixed tree: FP64 from here on, as the chain's sums
// (a thread's and a warp's sums are compensated FP32 pairs).
__device__ __forceinline__ double warps_sum(const double (*red)[kNA], int t) {
    double a[kLW];
#pragma unroll
    for (int w = 0; w < kLW; ++w) a[w] = red[w][t];
#pragma unroll
    for (int n = kLW / 2; n >= 1; n >>= 1)
#pragma unroll
        for (int w = 0; w < n; ++w) a[w] += a[w + n];
    return a[0];
}

// Grid-wide barrier on a counter that only grows: one release add per block, then
// acquire polls until every block of this barrier has added.  false after a timeout.
__device__ __forceinline__ bool loop_barrier(unsigned* bar, unsigned& target, Ctrl* ctrl, int* s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        target += gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(1u) : "memory");
        int ok = 1;
        unsigned polls = 0;
        long long t0 = 0;
        while ((int)(ld_acquire_gpu(bar) - target) < 0) {
            if ((++polls & 255u) == 0u) {
                const long long t = tail_clock_ns();
                if (t0 == 0) t0 = t;
                if ((ld_volatile_int(&ctrl->flags) & kFlagTimeout) || t - t0 > kBarrierWaitNs) {
                    atomicOr(&ctrl->flags, kFlagTimeout);
                    ok = 0;
                    break;
                }
            }
        }
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// W_ab = (Omega S)_ab in the canonical order, by gathers.
template <typename T>
__device__ __forceinline__ T gather_w(const LoopK<T>& k, const Csr<T>& om, int a, int b) {
    const int4 ri = __ldcg(k.rinfo + a);
    const T* Sb = k.S + b;
    T acc = mulT((T)fabs(__ldcg(k.rds + a)), __ldg(Sb + (int64_t)a * k.ld));
    for (int q0 = ri.x; q0 < ri.y; q0 += 8) {
        T w[8], s[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = q0 + u;
            const bool use = q < ri.y && q != ri.z;
            const int c = use ? __ldcg(om.ci + q) : 0;
            w[u] = use ? __ldcg(om.cv + q) : T(0);
            s[u] = use ? __ldg(Sb + (int64_t)c * k.ld) : T(0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (q0 + u < ri.y && q0 + u != ri.z) acc = fmaT(w[u], s[u], acc);
    }
    return acc;
}

// Slot s of a row: in its bucket, then in pages of the pool.  The page numbers of a row
// are taken as needed: of threads that race for one, the first to write it wins (the
// others' pages stay unused until the counter is reset).
template <typename T>
__device__ __forceinline__ Ent<T>* slot_at(const LoopK<T>& k, int row, int s) {
    if (s < kSlots) return k.slots + (size_t)row * kSlots + s;
    const int id = __ldcg(k.pages + (size_t)row * kPages + s / kSlots);
    return k.pool + (size_t)(id - 1) * kSlots + s % kSlots;
}
template <typename T>
__device__ __forceinline__ void put_slot(const LoopK<T>& k, int row, unsigned cf, T om, T g, T w) {
    const int s = atomicAdd(k.cnt + row, 1);
    if (s < kSlots) {
        st_ent(k.slots + (size_t)row * kSlots + s, cf, om, g, w);
        return;
    }
    if (s >= kMaxE) return;                        // the row's owner sees the count
    int* pt = k.pages + (size_t)row * kPages + s / kSlots;
    int id = __ldcg(pt);
    if (id == 0) {
        const int n = 1 + atomicAdd(k.ctr + kCtrPage, 1);
        if (n > k.npool) { atomicOr(k.ctr + kCtrFull, kFullPool); return; }
        const int old = atomicCAS(pt, 0, n);
        id = old ? old : n;
    }
    st_ent(k.pool + (size_t)(id - 1) * kSlots + s % kSlots, cf, om, g, w);
}

// G_ij = (W_ij + W_ji)/2 + lambda2 w_ij - [i=j]/w_ii, one fixed rounding sequence.
template <typename T>
__device__ __forceinline__ T gradient_of(T w, T wt, T om, T lam2, bool diag) {
    T g = fmaT(lam2, om, T(0.5) * (w + wt));
    if (diag) g -= T(1) / om;
    return g;
}

// The warp's queue of entries (i, j) with their W_ij: where W_ji has to be gathered --
// three dependent loads -- 32 entries go through it together, a lane each.
template <typename T>
struct Hits {
    int* i;
    int* j;
    T* w;
    int n;        // the same in every lane
    int emitted;  // per lane: entries with |W_ij| > lambda1 or in the support
    int* halves;  // LoopSmem's

    __device__ __forceinline__ void flush(const LoopK<T>& k, const Csr<T>& csr, T lam1, T lam2, int lane) {
        __syncwarp();
        const int first = max(0, n - 32);
        if (first + lane < n) {
            const int row = i[first + lane];
            const int col = j[first + lane];
            const T wij = w[first + lane];
            const T wji = gather_w(k, csr, col, row);
            // row col's own screening meets the pair too where |W_ji| > lambda1
            const bool first_meets = row < col || fabs(wji) <= lam1;
            const bool both = __ldcg(k.rds + row) > T(0) && __ldcg(k.rds + col) > T(0);
            const bool other = !(fabs(wji) <= lam1);
            emitted += both ? (first_meets ? 1 + other : 0) : 1;
            if (both && first_meets && !other) atomicAdd(halves, 1);
            if (first_meets) {
                const T g = gradient_of(wij, wji, T(0), lam2, false);
                if (!(fabs(g) <= lam1)) {
                    put_slot(k, row, (unsigned)col, T(0), g, wij);
                    put_slot(k, col, (unsigned)row, T(0), g, wji);
                }
            }
        }
        n = first;
        __syncwarp();
    }
    // one entry of each lane with `hit`
    __device__ __forceinline__ void push(const LoopK<T>& k, const Csr<T>& csr, T lam1, T lam2, bool hit, int row,
                                         int col, T wij, int lane) {
        const unsigned bal = __ballot_sync(kFull, hit);
        if (!bal) return;
        if (hit) {
            const int q = n + __popc(bal & ((1u << lane) - 1u));
            i[q] = row;
            j[q] = col;
            w[q] = wij;
        }
        n += __popc(bal);
        if (n >= 32) flush(k, csr, lam1, lam2, lane);
    }
};

// A row's block after its W is known (acc: this lane's V columns; mb: the support among
// them, the row's own column too): the bound of the rest (slack < 0: none is kept), and
// the entries with |W_ij| > lambda1 among them.
template <typename T, int V>
__device__ __forceinline__ void screen_emit(const LoopK<T>& k, const Csr<T>& csr, Hits<T>& hits, int i, int jb,
                                            const T (&acc)[V], unsigned mb, float slack, T lam1, T lam2, int lane) {
    constexpr int BJ = 32 * V;
    unsigned mx = 0;                     // bits of non-negative floats order as the floats; NaN above all
    bool big = false;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if ((mb >> v) & 1u) continue;
        mx = max(mx, __float_as_uint(abs_up(acc[v])) & 0x7fffffffu);
        big |= !(fabs(acc[v]) <= lam1);
    }
    if (k.bnd && slack >= 0.0f) {
        mx = __reduce_max_sync(kFull, mx);
        if (lane == 0) k.bnd[(size_t)i * k.nbp + jb] = __fadd_ru(__uint_as_float(mx), slack);
    }
    if (!__any_sync(kFull, big)) return;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int j = jb * BJ + lane * V + v;
        hits.push(k, csr, lam1, lam2, j < k.p && !((mb >> v) & 1u) && !(fabs(acc[v]) <= lam1), i, j, acc[v], lane);
    }
}

// Screening of the G column blocks jb[] (-1: none) of row i; lane t of the warp holds
// (tk, tw) of term t, the diagonal first, then the neighbours ascending; nt <= 32.
template <typename T, int G>
__device__ __forceinline__ void screen_blocks(const LoopK<T>& k, const Csr<T>& csr, Hits<T>& hits, int i, int tk, T tw,
                                              int nt, const int (&jb)[G], float slack, T lam1, T lam2, int lane) {
    constexpr int V = 16 / (int)sizeof(T), BJ = 32 * V, U = 8 / G;
    T acc[G][V];
    for (int t0 = 0; t0 < nt; t0 += U) {
        T sv[U][G][V], w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int kk = __shfl_sync(kFull, tk, (t0 + u) & 31);
            w[u] = __shfl_sync(kFull, tw, (t0 + u) & 31);
            if (t0 + u < nt) {
#pragma unroll
                for (int g = 0; g < G; ++g)
                    if (jb[g] >= 0) vload(sv[u][g], k.S + (int64_t)kk * k.ld + jb[g] * BJ + lane * V);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (t0 + u < nt) {
#pragma unroll
                for (int g = 0; g < G; ++g) {
#pragma unroll
                    for (int v = 0; v < V; ++v)
                        acc[g][v] = (t0 + u == 0) ? mulT(w[u], sv[u][g][v]) : fmaT(w[u], sv[u][g][v], acc[g][v]);
                }
            }
        }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
        if (jb[g] < 0) continue;
        const int j0 = jb[g] * BJ;
        unsigned sup = __ballot_sync(kFull, lane < nt && tk >= j0 && tk < j0 + BJ);
        unsigned mb = 0;
        while (sup) {
            const int o = __shfl_sync(kFull, tk, __ffs(sup) - 1) - j0;
            sup &= sup - 1;
            if (lane == o / V) mb |= 1u << (o % V);
        }
        screen_emit<T, V>(k, csr, hits, i, jb[g], acc[g], mb, slack, lam1, lam2, lane);
    }
}

// The same for one block of a row with more than 32 terms, which come 32 at a time.
template <typename T>
__device__ __forceinline__ void screen_block_long(const LoopK<T>& k, const Csr<T>& csr, Hits<T>& hits, int i, int4 ri,
                                                  T dv, int jb, float slack, T lam1, T lam2, int lane) {
    constexpr int V = 16 / (int)sizeof(T), BJ = 32 * V, U = 8;
    const int j0 = jb * BJ;
    T acc[V], s0[V];
    vload(s0, k.S + (int64_t)i * k.ld + j0 + lane * V);
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = mulT(dv, s0[v]);
    unsigned mb = 0;
    for (int q0 = ri.x; q0 < ri.y; q0 += 32) {
        const int q = q0 + lane;
        const int kq = q < ri.y ? __ldcg(csr.ci + q) : -1;
        const T wq = q < ri.y ? __ldcg(csr.cv + q) : T(0);
        unsigned sup = __ballot_sync(kFull, kq >= j0 && kq < j0 + BJ);
        while (sup) {
            const int o = __shfl_sync(kFull, kq, __ffs(sup) - 1) - j0;
            sup &= sup - 1;
            if (lane == o / V) mb |= 1u << (o % V);
        }
        const int nt = min(32, ri.y - q0);
        for (int t0 = 0; t0 < nt; t0 += U) {
            T sv[U][V], w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int kk = __shfl_sync(kFull, kq, (t0 + u) & 31);
                w[u] = __shfl_sync(kFull, wq, (t0 + u) & 31);
                if (t0 + u < nt) vload(sv[u], k.S + (int64_t)kk * k.ld + j0 + lane * V);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (t0 + u < nt && q0 + t0 + u != ri.z) {
#pragma unroll
                    for (int v = 0; v < V; ++v) acc[v] = fmaT(w[u], sv[u][v], acc[v]);
                }
            }
        }
    }
    screen_emit<T, V>(k, csr, hits, i, jb, acc, mb, slack, lam1, lam2, lane);
}

// The tasks lo .. hi - 1 of the list (all: of every block of every row, tested here),
// one warp; the blocks of a row come together.
template <typename T>
__device__ __forceinline__ void screen_tasks(const LoopK<T>& k, const Csr<T>& csr, Hits<T>& hits, const int* list,
                                             bool all, long long lo, long long hi, T lam1, T lam2, int lane) {
    int row = -1, nt = 0, tk = 0;
    T tw = T(0), dv = T(0);
    float slack = 0.0f;
    int4 ri = make_int4(0, 0, -1, 0);
    for (long long t0 = lo; t0 < hi; t0 += 32) {
        int tr = -1, tb = -1;
        if (t0 + lane < hi) {
            if (all) {
                const long long t = t0 + lane;
                tr = (int)(t / k.nbm);
                tb = (int)(t % k.nbm);
                if (k.m1) {
                    const T d = __ldcg(k.rds + tr);
                    bool below;
                    if (d > T(0)) {
                        below = mulT(d, (T)bf16_val(__ldg(k.m1 + (int64_t)tr * k.nbm + tb))) <= lam1;
                    } else {
                        const float b = __fadd_ru(__ldcg(k.bnd + (size_t)tr * k.nbp + tb), __ldcg(k.slack + tr));
                        if constexpr (sizeof(T) == 4) below = b <= lam1;
                        else below = (double)b <= lam1;
                    }
                    if (below) tr = -1;
                }
            } else {
                const int c = __ldcg(list + t0 + lane);
                tr = c / k.nbm;
                tb = c - tr * k.nbm;
            }
        }
        const int cnt = (int)min(32ll, hi - t0);
        for (int u = 0; u < cnt;) {
            const int r = __shfl_sync(kFull, tr, u);
            if (r != row && r >= 0) {
                row = r;
                ri = __ldcg(k.rinfo + row);
                dv = (T)fabs(__ldcg(k.rds + row));
                nt = (ri.y - ri.x) + (ri.z >= 0 ? 0 : 1);
                slack = k.bnd && nt > 1 ? __ldcg(k.slack + row) : -1.0f;
                tk = row;
                tw = dv;
                if (lane > 0 && lane < nt) {
                    int q = ri.x + lane - 1;
                    if (ri.z >= 0 && q >= ri.z) ++q;
                    tk = __ldcg(csr.ci + q);
                    tw = __ldcg(csr.cv + q);
                }
            }
            // the run of this row's tasks from u on
            const unsigned same = __ballot_sync(kFull, lane >= u && lane < cnt && tr == r) >> u;
            const int run = same == 0xffffffffu ? 32 : __ffs(~same) - 1;
            if (r < 0) {
            } else if (nt > 32) {
                for (int g = 0; g < run; ++g)
                    screen_block_long(k, csr, hits, row, ri, dv, __shfl_sync(kFull, tb, u + g), slack, lam1, lam2, lane);
            } else if (nt <= 2) {
                for (int g0 = 0; g0 < run; g0 += 4) {
                    int jb[4];
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const int b = __shfl_sync(kFull, tb, (u + g0 + g) & 31);
                        jb[g] = g0 + g < run ? b : -1;
                    }
                    screen_blocks<T, 4>(k, csr, hits, row, tk, tw, nt, jb, slack, lam1, lam2, lane);
                }
            } else if (nt <= 4) {
                for (int g0 = 0; g0 < run; g0 += 2) {
                    int jb[2];
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        const int b = __shfl_sync(kFull, tb, (u + g0 + g) & 31);
                        jb[g] = g0 + g < run ? b : -1;
                    }
                    screen_blocks<T, 2>(k, csr, hits, row, tk, tw, nt, jb, slack, lam1, lam2, lane);
                }
            } else {
                for (int g = 0; g < run; ++g) {
                    const int jb[1] = {__shfl_sync(kFull, tb, u + g)};
                    screen_blocks<T, 1>(k, csr, hits, row, tk, tw, nt, jb, slack, lam1, lam2, lane);
                }
            }
            u += run;
        }
    }
}

// A block of a row with more than 32 terms by four warps, 32 columns each (a lane per
// column), so that 16 loads are in flight per lane of a chain that is long.  red: the
// four warps' maxima, two buffers; bar: their named barrier.
template <typename T>
__device__ __forceinline__ void screen_heavy(const LoopK<T>& k, const Csr<T>& csr, Hits<T>& hits, int i, int jb,
                                             T lam1, T lam2, unsigned* red, int buf, int quarter, int bar, int lane) {
    constexpr int BJ = 32 * (16 / (int)sizeof(T)), NS = BJ / 32, U = 16;
    const int4 ri = __ldcg(k.rinfo + i);
    const T dv = (T)fabs(__ldcg(k.rds + i));
    const float slack = __ldcg(k.slack + i);
    const int j = jb * BJ + 32 * quarter + lane;
    unsigned mx = 0;
    bool hit = false;
    T acc = T(0);
    if (quarter < NS) {
        acc = mulT(dv, __ldg(k.S + (int64_t)i * k.ld + j));
        bool sup = j == i;
        for (int q0 = ri.x; q0 < ri.y; q0 += 32) {
            const int q = q0 + lane;
            const int kq = q < ri.y ? __ldcg(csr.ci + q) : 0;
            const T wq = q < ri.y ? __ldcg(csr.cv + q) : T(0);
            const int nt = min(32, ri.y - q0);
            for (int t0 = 0; t0 < nt; t0 += U) {
                T sv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int kk = __shfl_sync(kFull, kq, (t0 + u) & 31);
                    sup |= t0 + u < nt && kk == j;
                    sv[u] = t0 + u < nt ? __ldg(k.S + (int64_t)kk * k.ld + j) : T(0);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const T w = __shfl_sync(kFull, wq, (t0 + u) & 31);
                    if (t0 + u < nt && q0 + t0 + u != ri.z) acc = fmaT(w, sv[u], acc);
                }
            }
        }
        if (!sup) {
            mx = __float_as_uint(abs_up(acc)) & 0x7fffffffu;
            hit = j < k.p && !(fabs(acc) <= lam1);
        }
        mx = __reduce_max_sync(kFull, mx);
    }
    if (lane == 0) red[buf * kLW + quarter] = mx;
    asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
    if (quarter == 0 && lane == 0) {
        unsigned m = 0;
        for (int q = 0; q < 4; ++q) m = max(m, red[buf * kLW + q]);
        k.bnd[(size_t)i * k.nbp + jb] = __fadd_ru(__uint_as_float(m), slack);
    }
    hits.push(k, csr, lam1, lam2, hit, i, j, acc, lane);
}

// The support entries of the block's own rows with neighbours: n listed ones (items: CSR
// position, item_r: row), or, where the list was too long for it, all entries e0 .. e1 - 1
// (start: the rows' first positions).  Two threads per entry, one for W_ij and one for W_ji.
template <typename T>
__device__ __forceinline__ void screen_support(const LoopK<T>& k, const Csr<T>& csr, int i0, int nr, const int* items,
                                               const short* item_r, int n, const int* start, const int* s_rc, int e0,
                                               int e1, T lam2, int& emitted) {
    const int side = threadIdx.x & 1;
    const bool listed = n <= kItemCap;
    const int b0 = listed ? 0 : e0, b1 = listed ? n : e1;
    for (int b = b0; b < b1; b += kLT / 2) {
        int q = b + (threadIdx.x >> 1);
        int r = 0, j = 0;
        bool in = q < b1;
        if (in && listed) {
            r = item_r[q];
            q = items[q];
        } else if (in) {
            int lo = 0, hi = nr - 1;                 // last row with start <= q
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (start[mid] <= q) lo = mid; else hi = mid - 1;
            }
            r = lo;
            in = s_rc[r] >= 0;
        }
        T w = T(0);
        if (in) {
            j = __ldcg(csr.ci + q);
            w = side ? gather_w(k, csr, j, i0 + r) : gather_w(k, csr, i0 + r, j);
        }
        const T wt = __shfl_xor_sync(kFull, w, 1);
        if (in && !side) {
            const T o = __ldcg(csr.cv + q);
            put_slot(k, i0 + r, (unsigned)j | kFSupp, o, gradient_of(w, wt, o, lam2, j == i0 + r), w);
            ++emitted;
        }
    }
}

// The warp's blocks 8 oc .. 8 oc + 7 of row i with their bit in `bits` onto the task list
// (heavy: from the back of it); terms: the row's.
template <typename T>
__device__ __forceinline__ void push_tasks(const LoopK<T>& k, int par, bool heavy, int terms, int i, int oc,
                                           unsigned bits, int lane) {
    const int c = __popc(bits);
    const int incl = warp_incl_scan(c, lane);
    const int total = __shfl_sync(kFull, incl, 31);
    if (!total) return;
    int base = 0;
    if (lane == 0) {
        const unsigned long long work = ((unsigned long long)total * terms + 32) >> 6;
        base = (int)atomicAdd(heavy ? &k.todo[par].y : &k.todo[par].x, work << 32 | (unsigned)total);
    }
    int pos = __shfl_sync(kFull, base, 0) + incl - c;
    while (bits) {
        const int v = __ffs(bits) - 1;
        bits &= bits - 1;
        if (pos < k.ntask_cap)
            k.tasks[(size_t)par * k.ntask_cap + (heavy ? k.ntask_cap - 1 - pos : pos)] = i * k.nbm + 8 * oc + v;
        ++pos;
    }
}

// The tasks of a row with the diagonal alone (one warp): fl(|w_ii| m1[i][jb]) > lambda1.
template <typename T>
__device__ __forceinline__ void pure_row_tasks(const LoopK<T>& k, int i, T d, T lam1, int par, int lane) {
    const int noct = (k.nbm + 7) / 8;
    for (int o0 = 0; o0 < noct; o0 += 32) {
        const int oc = o0 + lane;
        unsigned bits = 0;
        if (oc < noct) {
            if (k.m1g) {
                if (!(mulT(d, (T)bf16_val(__ldg(k.m1g + (int64_t)i * k.ngl + oc))) <= lam1)) {
                    float f[8];
                    bf16x8(__ldg(reinterpret_cast<const uint4*>(k.m1 + (int64_t)i * k.nbm + 8 * oc)), f);
#pragma unroll
                    for (int v = 0; v < 8; ++v)
                        if (!(mulT(d, (T)f[v]) <= lam1)) bits |= 1u << v;
                }
            } else {
#pragma unroll
                for (int v = 0; v < 8; ++v)
                    if (8 * oc + v < k.nbm &&
                        !(mulT(d, (T)bf16_val(__ldg(k.m1 + (int64_t)i * k.nbm + 8 * oc + v))) <= lam1))
                        bits |= 1u << v;
            }
        }
        push_tasks(k, par, false, 1, i, oc, bits, lane);
    }
}

// The certified bounds of row i after a change of its weights, and the tasks they leave
// (one warp).  term(e): column, |change| rounded up, and whether the column left the
// support, for e < n; init: the bounds start here.  terms, slack: the row's length, its rounding
// term.
template <typename T, typename F>
__device__ __forceinline__ void bound_row(const LoopK<T>& k, int i, int n, bool init, int terms, float slack, T lam1,
                                          int par, int lane, F&& term) {
    constexpr int V = 16 / (int)sizeof(T), BJ = 32 * V;
    const bool vec = (k.nbm & 7) == 0;
    const int noct = (k.nbm + 7) / 8;
    // lanes: octets of blocks, and where a row has few octets also the terms
    const int groups = noct <= 4 ? 8 : noct <= 8 ? 4 : noct <= 16 ? 2 : 1;
    const int gl = 32 / groups, grp = lane / gl, ol = lane % gl;
    for (int c0 = 0; c0 < noct; c0 += gl) {
        const int oc = c0 + ol;
        const bool act = oc < noct;
        float B[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) B[v] = 0.0f;
        float4* m = reinterpret_cast<float4*>(k.bnd + (size_t)i * k.nbp + 8 * oc);
        float4 m_lo = make_float4(0.f, 0.f, 0.f, 0.f), m_hi = m_lo;
        if (!init && act && grp == 0) {
            m_lo = __ldcg(m);
            m_hi = __ldcg(m + 1);
        }
        unsigned inf = 0;
        for (int a = 0; a < n; a += 32) {
            int tk = 0;
            float tw = 0.0f;
            bool left = false;
            if (a + lane < n) term(a + lane, tk, tw, left);
            unsigned lb = __ballot_sync(kFull, left);
            while (lb) {
                const int kb = __shfl_sync(kFull, tk, __ffs(lb) - 1) / BJ;
                lb &= lb - 1;
                if (act && kb / 8 == oc) inf |= 1u << (kb & 7);
            }
            const int nt = min(32, n - a);
            for (int t0 = 0; t0 < nt; t0 += 4 * groups) {
                uint4 mv[4];
                float w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int t = t0 + q * groups + grp;
                    const int kk = __shfl_sync(kFull, tk, t & 31);
                    w[q] = __shfl_sync(kFull, tw, t & 31);
                    mv[q] = make_uint4(0, 0, 0, 0);
                    if (t >= nt || w[q] == 0.0f) { w[q] = 0.0f; continue; }
                    if (!act) continue;
                    const unsigned short* src = k.m1 + (int64_t)kk * k.nbm + 8 * oc;
                    if (vec) {
                        mv[q] = __ldg(reinterpret_cast<const uint4*>(src));
                    } else {
                        unsigned e[8];
#pragma unroll
                        for (int v = 0; v < 8; ++v) e[v] = 8 * oc + v < k.nbm ? __ldg(src + v) : 0;
                        mv[q] = make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16), e[4] | (e[5] << 16),
                                           e[6] | (e[7] << 16));
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float f[8];
                    bf16x8(mv[q], f);
#pragma unroll
                    for (int v = 0; v < 8; ++v) B[v] = __fadd_ru(B[v], __fmul_ru(w[q], f[v]));
                }
            }
        }
        for (int o = gl; o < 32; o <<= 1) {
#pragma unroll
            for (int v = 0; v < 8; ++v) B[v] = __fadd_ru(B[v], __shfl_xor_sync(kFull, B[v], o));
        }
        unsigned bits = 0;
        if (act && grp == 0) {
            const float old[8] = {m_lo.x, m_lo.y, m_lo.z, m_lo.w, m_hi.x, m_hi.y, m_hi.z, m_hi.w};
            if (!init) {
#pragma unroll
                for (int v = 0; v < 8; ++v) B[v] = __fadd_ru(B[v], old[v]);
            }
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                if ((inf >> v) & 1u) B[v] = __int_as_float(0x7f800000);
                const float t = __fadd_ru(B[v], slack);
                bool below;
                if constexpr (sizeof(T) == 4) below = t <= lam1;
                else below = (double)t <= lam1;
                if (8 * oc + v < k.nbm && !below) bits |= 1u << v;
            }
            m[0] = make_float4(B[0], B[1], B[2], B[3]);
            m[1] = make_float4(B[4], B[5], B[6], B[7]);
        }
        push_tasks(k, par, terms > kHeavyTerms, terms, i, oc, bits, lane);
    }
}

// The rounding term of a row of m terms with sum |w| = sumw: gamma_m sumw max|S|, every
// operation rounded up (gamma_m <= m u (1 + 2^-9) while m u <= 2^-10; longer rows are
// always screened).
template <typename T>
__device__ __forceinline__ float slack_of(int m, float sumw, float mg) {
    const float mu = (float)m * (sizeof(T) == 4 ? 0x1p-24f : 0x1p-53f);
    if (mu > 0x1p-10f) return __int_as_float(0x7f800000);
    return __fmul_ru(__fmul_ru(__fmul_ru(mu, 1.001953125f), sumw), mg);
}
__device__ __forceinline__ float warp_sum_up(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = __fadd_ru(x, __shfl_xor_sync(kFull, x, o));
    return x;
}

// Which passes the chain of kernels does faster.  The loop keeps 16 warps per SM and a row with
// its block, where the chain spreads a row over the grid and keeps more loads in flight; the chain
// pays 70 to 100 us for its launches and has no memory in its bounds.  Measured on GB300:
//   screening  the loop 0.18 to 0.3 us per 1000 terms (a term: 128 FP32 columns of one neighbour's
//              row of S), the chain 0.1 us per 1000 terms of all blocks of the neighbours,
//              nbm (nnz - p), where the iterate is dense: level at half of them;
//   support    W_ij and W_ji by gathers, up to 1.3 us per 1000 of sum n_i^2 over the rows of
//              the block that has most, as 6 terms each: a quarter of the chain's terms, at most
//              0.9 ms (a band of 2000 entries a row takes seconds: its blocks are few for the chain);
//   search     1 us per pair of 32-entry chunks of a block's rows: level at about 500.
// A pass that loses may be worth it (bounds that start anew keep more blocks than they do a pass
// later, if the rows are short), so the losses add up to a debt, and the loop leaves when that
// passes what a pass over all blocks loses.  Without bounds there is nothing to wait for.
// us of the chain and of the loop per iteration, without the rule: p = 8192, n = 1000, lambda1 = 0.07
// (130 entries a row) 8200, 18300; p = 2000, 90 entries a row 640, 1080; a hub row of 700
// entries at p = 700 430, 710.
// Terms are counted by 1024 here.
constexpr unsigned kWorkEven = 512, kWorkBlind = 1370, kSupEven = 340, kSupMost = 4096;
constexpr unsigned kDebtLeast = 256, kDebtMost = 1u << 16;
constexpr int kShortMean = 32;
constexpr int kUnitsMax = 512;
constexpr int kTasksFew = 1 << 16, kHeavyFew = 256, kSupFew = 900;
__device__ __forceinline__ int row_units(int entries) {
    const int c = (entries + 31) >> 5;
    return c * (c + 1) / 2;
}
__device__ __forceinline__ int row_sup(int entries) { return min(entries, 1 << 11) * min(entries, 1 << 11) >> 6; }
__device__ __forceinline__ unsigned chain_terms(int nnz, int nbm, int p) {
    return (unsigned)((unsigned long long)nbm * (unsigned)max(0, nnz - p) >> 10);
}
// One more pass that does `work` where both forms are level at `even`; whether to leave before it.
__device__ __forceinline__ bool in_debt(unsigned& debt, unsigned work, unsigned even, unsigned credit) {
    debt = work > even ? debt + (work - even) : debt - min(debt, even - work);
    return debt > min(kDebtLeast + credit, kDebtMost);
}
__device__ __forceinline__ bool support_debt(unsigned& debt, int sup, int nnz, int nbm, int p) {
    return in_debt(debt, 3u * (unsigned)sup >> 3, min(kSupEven + chain_terms(nnz, nbm, p) / 4, kSupMost), 0u);
}
// Whether to leave before a pass of many tasks (the same answer in the whole grid), and whether
// this block leaves its support entries out, which ends the launch after the screening barrier.
// Block-wide calls.  Passes with few do not come here, and the calls are not inlined: with the
// arithmetic in line every pass took 2 us longer (47.8 -> 50.5 us at p = 400).
template <typename T>
__device__ __noinline__ bool leave_tasks(LoopSmem<T>& sm, unsigned long long terms64, int nnz, int nbm, int p) {
    const unsigned chain = chain_terms(nnz, nbm, p), all = chain_terms(nnz, nbm, 0);
    if (threadIdx.x == 0)
        sm.leave[1] = in_debt(sm.debt, (unsigned)(terms64 >> 4), kWorkEven + chain / 2,
                              nnz / kShortMean < p ? all - chain / 2 : 0u);
    __syncthreads();
    return sm.leave[1] != 0;
}
template <typename T>
__device__ __noinline__ bool leave_support(LoopSmem<T>& sm, int* full, int nnz, int nbm, int p) {
    if (threadIdx.x == 0) {
        sm.leave[0] = support_debt(sm.sup_debt, sm.sup, nnz, nbm, p);
        if (sm.leave[0]) atomicOr(full, kFullDense);
    }
    __syncthreads();
    return sm.leave[0] != 0;
}

// After a timeout: no further pass of either graph loop.
template <typename T>
__device__ __forceinline__ void end_loops(const LoopK<T>& k) {
    if (!k.use_cond) return;
    cudaGraphSetConditional(k.chain_cond, 0u);
    cudaGraphSetConditional(k.outer_cond, 0u);
}

// 512 threads of up to 128 registers: one block per SM.
template <typename T>
__global__ void __launch_bounds__(kLT, 1) k_loop(LoopK<T> k) {
    using A = typename AccOf<T>::type;
    extern __shared__ __align__(16) unsigned char raw[];
    LoopSmem<T>& sm = *reinterpret_cast<LoopSmem<T>*>(raw);
    const int R = k.R;
    T* s_dv = reinterpret_cast<T*>(raw + (sizeof(LoopSmem<T>) + 15) / 16 * 16);   // w_ii of the owned rows
    T* s_g = s_dv + R;                 // G_ii
    T* s_om = s_g + R;                 // w_ii at the last gradient pass
    T* s_sd = s_om + R;                // S_ii
    T* s_w = s_sd + R;                 // W_ii
    // per owned row: pure -1 - (slots), else the slots; in the accept step its entries
    int* s_rc = reinterpret_cast<int*>(s_w + R);
    int* s_list = s_rc + R;            // rows: from the front up to 32 candidates, from the back more
    float* s_m1 = reinterpret_cast<float*>(s_list + R);         // max of the row's block maxima
    int* s_eo = reinterpret_cast<int*>(s_m1 + R);               // place in `big` of its candidates (-1: in ents)
    int* s_mv = s_eo + R;              // the row's bounds are set
    int* s_rb = s_mv + R;              // CSR position of its first entry
    int* s_pl = s_rb + R;              // rows of the diagonal alone that have tasks

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bid = blockIdx.x, nb = gridDim.x;
    const int i0 = bid * R, nr = max(0, min(R, k.p - i0));
    Ctrl* ctrl = k.ctrl;
    const T lam1 = (T)ctrl->lam1, lam2 = (T)ctrl->lam2;
    const double lam2d = ctrl->lam2;
    const int iter_limit = ctrl->iter_limit, use_stop = ctrl->use_stop;
    const int ng = k.m1g ? k.nbm / 8 : 0;
    unsigned target = 0;
    int iter = ctrl->iter;
    long long trials = 0;
    long long screen_ns = 0;
    int attempts = 0;
    int nnz_now = ctrl->nnz_cur;       // entries of the current iterate
    int par = 0;                       // parity of the lists and column maxima
    int pbuf = 0;                      // partial buffer
    int buf = 0;                       // CSR buffer of the current iterate: 0 cur, 1 next
    int last_h = 0;
    if (tid == 0) { sm.flags = 0; sm.full = 0; sm.accept = -1; sm.converged = 0; sm.n2 = 0.0; sm.nlong = 0; sm.nhuge = 0; sm.ni = 0; sm.npl = 0; sm.sup = 0; sm.units = 0; sm.halves = 0; sm.off = 0; }
    __syncthreads();

    if (*k.symmetric == 0ull) {
        // all of the solve is the chain's
        if (bid == 0 && tid == 0) {
            ctrl->loop_launches += 1;
            ctrl->loop_full = 1;
            ctrl->chain_left = 0x7fffffff;
            if (k.use_cond) {
                cudaGraphSetConditional(k.chain_cond, 1u);
                cudaGraphSetConditional(k.outer_cond, 1u);
            }
        }
        return;
    }

    // ---------------- set-up of the owned rows from the current iterate
    for (int r = tid; r < nr; r += kLT) {
        const int i = i0 + r;
        const int rb = k.cur.rp[i], re = k.cur.rp[i + 1];
        int lo = rb, hi = re;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (k.cur.ci[mid] < i) lo = mid + 1; else hi = mid;
        }
        const int pd = (lo < re && k.cur.ci[lo] == i) ? lo : -1;
        const T dv = pd >= 0 ? k.cur.cv[pd] : T(0);
        const bool pure = re - rb == 1 && pd >= 0;
        k.rinfo[i] = make_int4(rb, re, pd, pure ? 1 : 0);
        k.rds[i] = pure ? dv : -dv;
        s_dv[r] = dv;
        s_sd[r] = __ldg(k.S + (int64_t)i * k.ld + i);
        s_rc[r] = pure ? -1 : 0;
        s_rb[r] = rb;
        s_eo[r] = -1;
        s_mv[r] = 0;
        if (!pure) {
            s_list[atomicAdd(&sm.nlong, 1)] = r;
            atomicAdd(&sm.off, 1);
            atomicAdd(&sm.sup, row_sup(re - rb));
            const int at = atomicAdd(&sm.ni, re - rb);
            for (int q = rb; q < re; ++q)
                if (at + q - rb < kItemCap) { sm.items[at + q - rb] = q; sm.item_r[at + q - rb] = (short)r; }
        }
        if (r == 0) sm.e0 = rb;
        if (r == nr - 1) sm.e1 = re;
        float m = 0.0f;
        if (k.m1g) {
            // rows of m1g are 16-byte aligned; the entries past ng are not written
            const unsigned short* gm = k.m1g + (int64_t)i * k.ngl;
            int g = 0;
            for (; g + 8 <= ng; g += 8) {
                float f[8];
                bf16x8(__ldg(reinterpret_cast<const uint4*>(gm + g)), f);
#pragma unroll
                for (int v = 0; v < 8; ++v) m = max_nan(m, f[v]);
            }
            for (; g < ng; ++g) m = max_nan(m, bf16_val(__ldg(gm + g)));
        } else if (k.m1) {
            for (int b = 0; b < k.nbm; ++b) m = max_nan(m, bf16_val(__ldg(k.m1 + (int64_t)i * k.nbm + b)));
        }
        s_m1[r] = m;
        if (k.m1) atomicMax(k.mg, __float_as_uint(m) & 0x7fffffffu);
        if (pure && k.m1 && !(mulT(dv, (T)m) <= lam1)) s_pl[atomicAdd(&sm.npl, 1)] = r;
    }
    __syncthreads();
    if (tid == 0) {
        unsigned d = 0u;
        sm.debt = ctrl->loop_debt;
        sm.sup_debt = 0u;
        if (support_debt(d, sm.sup, nnz_now, k.nbm, k.p)) atomicOr(k.ctr + kCtrStart, 1);
    }
    bool alive = loop_barrier(k.bar, target, ctrl, &sm.ok);
    const float mg = __uint_as_float(__ldcg(k.mg));
    bool dense = alive && __ldcg(k.ctr + kCtrStart) != 0;
    if (alive && k.bnd && !dense) {
        // the tasks of the rows of the diagonal alone; the bounds of the others, from their
        // weights
        for (int li = warp; li < sm.npl; li += kLW) pure_row_tasks(k, i0 + s_pl[li], s_dv[s_pl[li]], lam1, par, lane);
        for (int li = warp; li < sm.nlong; li += kLW) {
            const int r = s_list[li], i = i0 + r;
            const int4 ri = k.rinfo[i];
            float sw = 0.0f;
            for (int q = ri.x + lane; q < ri.y; q += 32) sw = __fadd_ru(sw, abs_up(k.cur.cv[q]));
            const float slack = slack_of<T>(ri.y - ri.x + 1, warp_sum_up(sw), mg);
            bound_row(k, i, ri.y - ri.x, true, ri.y - ri.x, slack, lam1, par, lane, [&](int e, int& c, float& w, bool&) {
                c = k.cur.ci[ri.x + e];
                w = abs_up(k.cur.cv[ri.x + e]);
            });
            if (lane == 0) { k.slack[i] = slack; s_mv[r] = 1; }
        }
        alive = loop_barrier(k.bar, target, ctrl, &sm.ok);
    }
    if (alive && k.bnd && !dense) {
        const ulonglong2 todo = __ldcg(k.todo + par);
        if ((int)todo.x > kTasksFew || (int)todo.y > kHeavyFew)
            dense = leave_tasks(sm, (todo.x >> 32) + (todo.y >> 32), nnz_now, k.nbm, k.p);
    }
    bool run = alive && iter < iter_limit;

    while (run) {
        if (!k.bnd) dense |= ((unsigned long long)k.nbm * (unsigned)nnz_now >> 10) > kWorkBlind;
        if (dense) break;
        const Csr<T> om = buf ? k.next : k.cur;
        const Csr<T> out = buf ? k.cur : k.next;
        const long long t_scr = tid == 0 && bid == 0 ? tail_clock_ns() : 0;
        // ---------------- screen
        if (bid == 0 && tid == 0) k.ctr[kCtrBig] = 0;
        Hits<T> hits{sm.hit_i[warp], sm.hit_j[warp], sm.hit_w[warp], 0, 0, &sm.halves};
        // the owned rows' support entries, then a share of the (row, block) tasks
        if (sm.sup < kSupFew || !leave_support(sm, k.ctr + kCtrFull, nnz_now, k.nbm, k.p))
            screen_support(k, om, i0, nr, sm.items, sm.item_r, sm.ni, s_rb, s_rc, sm.e0, sm.e1, lam2, hits.emitted);
        {
            const ulonglong2 todo = k.bnd ? __ldcg(k.todo + par) : make_ulonglong2(0, 0);
            const int nt = (int)todo.x, nh = (int)todo.y;
            // the same in every block: the pass is left to the chain before its tasks
            if (attempts > 0 && (nt > kTasksFew || nh > kHeavyFew))
                dense = leave_tasks(sm, (todo.x >> 32) + (todo.y >> 32), nnz_now, k.nbm, k.p);
            if (dense) break;
            const bool all = !k.bnd || nt > k.ntask_cap - nh || nt < 0 || nh < 0;
            const int* list = k.tasks + (size_t)par * k.ntask_cap;
            if (!all) {
                // rows of many terms: four warps on a block, the blocks dealt over the grid
                int buf2 = 0;
                for (int t = (warp >> 2) * nb + bid; t < nh; t += (kLW / 4) * nb, buf2 ^= 1) {
                    const int c = __ldcg(list + k.ntask_cap - 1 - t), i = c / k.nbm;
                    screen_heavy(k, om, hits, i, c - i * k.nbm, lam1, lam2, &sm.heavy[0][warp & ~3], buf2, warp & 3,
                                 1 + (warp >> 2), lane);
                }
            }
            const long long total = all ? (long long)k.p * k.nbm : nt;
            const long long nw = (long long)kLW * nb, gw = (long long)bid * kLW + warp;
            screen_tasks(k, om, hits, list, all, total * gw / nw, total * (gw + 1) / nw, lam1, lam2, lane);
        }
        if (hits.n) hits.flush(k, om, lam1, lam2, lane);
        alive = loop_barrier(k.bar, target, ctrl, &sm.ok);
        if (!alive) break;
        if (tid == 0 && bid == 0) screen_ns += tail_clock_ns() - t_scr;

        // ---------------- build
        // this parity's list was read by every block before the barrier: empty it for the
        // accept step of the next iteration
        if (bid == nb - 1 && tid == 0) k.todo[par] = make_ulonglong2(0, 0);
        if (tid == 0) { sm.nlong = 0; sm.nhuge = 0; sm.units = 0; sm.pool_full = __ldcg(k.ctr + kCtrFull); }
        __syncthreads();
        dense = (sm.pool_full & kFullDense) != 0;      // a block has left its support out
        if (dense) break;
        ++attempts;
        const bool pool_full = sm.pool_full != 0;
        int em = hits.emitted, bad = 0, full = 0;
        A o2{};
        // the rows with candidates beside the diagonal, in row order (the sums below follow it)
        for (int r0 = 0; r0 < nr; r0 += kLT) {
            const int r = r0 + tid, i = i0 + r;
            int kind = 0;                        // 1: up to 32 candidates, 2: more
            if (r < nr) {
                const int c = __ldcg(k.cnt + i);
                const bool pure = s_rc[r] < 0;
                const T dv = s_dv[r];
                s_om[r] = dv;
                if (pure) ++em;
                if (c) k.cnt[i] = 0;
                if (c > kMaxE - 2 || (pool_full && c > kSlots)) {
                    ++full;
                } else if (c == 0 && pure) {
                    const T w = mulT(dv, s_sd[r]);
                    const T g = gradient_of(w, w, dv, lam2, true);
                    if (!(g == g) || isinf((double)g)) ++bad;
                    s_g[r] = g;
                    s_w[r] = w;
                    acc_add(o2, mulT(dv, dv));
                    k.len[i] = 0;
                } else {
                    s_rc[r] = pure ? -1 - c : c;
                    kind = c + (pure ? 1 : 0) <= 32 ? 1 : 2;
                    if (kind == 2) atomicAdd(&sm.units, row_units(c + (pure ? 1 : 0)));
                }
            }
            const unsigned b1 = __ballot_sync(kFull, kind == 1), b2 = __ballot_sync(kFull, kind == 2);
            if (lane == 0) { sm.wsum[warp] = __popc(b1); sm.wbig[warp] = __popc(b2); }
            __syncthreads();
            int p1 = sm.nlong, p2 = sm.nhuge;
            for (int w = 0; w < warp; ++w) { p1 += sm.wsum[w]; p2 += sm.wbig[w]; }
            const unsigned below = (1u << lane) - 1u;
            if (kind == 1) s_list[p1 + __popc(b1 & below)] = r;
            if (kind == 2) s_list[R - 1 - (p2 + __popc(b2 & below))] = r;
            __syncthreads();
            if (tid == kLT - 1) { sm.nlong = p1 + __popc(b1); sm.nhuge = p2 + __popc(b2); }
            __syncthreads();
        }
        // too much for one block: as a full bucket
        const bool many = sm.units > kUnitsMax;
        if (many && tid == 0) ++full;
        const int nsmall = many ? 0 : sm.nlong, nlong = many ? 0 : nsmall + sm.nhuge;
        auto row_at = [&](int li) { return li < nsmall ? s_list[li] : s_list[R - 1 - (li - nsmall)]; };
        auto ents_of = [&](int r) { return s_eo[r] < 0 ? k.ents + (size_t)(i0 + r) * kSlots : k.big + s_eo[r]; };
        // rows of more than kSlots candidates: the whole block on one, keys in shared memory
        for (int li = nsmall; li < nlong; ++li) {
            const int r = row_at(li), i = i0 + r;
            const bool pure = s_rc[r] < 0;
            const int c = pure ? -1 - s_rc[r] : s_rc[r];
            const int E = c + (pure ? 1 : 0);
            if (E <= kSlots) continue;
            if (tid == 0) {
                const int at = atomicAdd(k.ctr + kCtrBig, E);
                s_eo[r] = at + E <= 2 * k.npool * kSlots ? at : -2;
            }
            __syncthreads();
            if (s_eo[r] == -2) {          // no room: as a full bucket
                __syncthreads();
                if (tid == 0) {
                    s_eo[r] = -1;
                    k.len[i] = 0;
                    ++full;
                }
                continue;
            }
            Ent<T> sl[kMaxE / kLT];
            int rank[kMaxE / kLT];
#pragma unroll
            for (int q = 0; q < kMaxE / kLT; ++q) {
                const int e = tid + kLT * q;
                rank[q] = 0;
                if (e < c) {
                    sl[q] = ld_slot(slot_at(k, i, e));
                } else if (e < E) {
                    const T w = mulT(s_dv[r], s_sd[r]);
                    sl[q] = Ent<T>{(unsigned)i | kFSupp, s_dv[r], gradient_of(w, w, s_dv[r], lam2, true), w};
                }
                if (e < E) sm.items[e] = (int)(sl[q].cf & kColMask);
            }
            __syncthreads();
            for (int t = 0; t < E; ++t) {
                const int kt = sm.items[t];
#pragma unroll
                for (int q = 0; q < kMaxE / kLT; ++q)
                    rank[q] += tid + kLT * q < E && kt < (int)(sl[q].cf & kColMask) ? 1 : 0;
            }
            Ent<T>* dst = ents_of(r);
#pragma unroll
            for (int q = 0; q < kMaxE / kLT; ++q) {
                if (tid + kLT * q < E) {
                    const Ent<T> x = sl[q];
                    if (!(x.g == x.g) || isinf((double)x.g)) ++bad;
                    if ((int)(x.cf & kColMask) == i) { s_g[r] = x.g; s_w[r] = x.w; }
                    st_ent(dst + rank[q], x.cf, x.om, x.g, x.w);
                }
            }
            // the row's pages are read: free for the next pass
            if (tid >= 1 && tid < kPages) k.pages[(size_t)i * kPages + tid] = 0;
            if (tid == 0) k.len[i] = E;
            __syncthreads();
        }
        for (int li = warp; li < nlong; li += kLW) {
            const int r = row_at(li), i = i0 + r;
            const bool pure = s_rc[r] < 0;
            const int c = pure ? -1 - s_rc[r] : s_rc[r];
            const int E = c + (pure ? 1 : 0);
            if (E > kSlots) continue;
            if (lane == 0) s_eo[r] = -1;
            Ent<T> sl[kSlots / 32];
            unsigned key[kSlots / 32];
            int rank[kSlots / 32];
#pragma unroll
            for (int q = 0; q < kSlots / 32; ++q) {
                const int e = lane + 32 * q;
                key[q] = 0xffffffffu;
                rank[q] = 0;
                if (e < c) {
                    sl[q] = ld_slot(k.slots + (size_t)i * kSlots + e);
                } else if (e < E) {
                    const T w = mulT(s_dv[r], s_sd[r]);       // a pure row's diagonal
                    sl[q] = Ent<T>{(unsigned)i | kFSupp, s_dv[r], gradient_of(w, w, s_dv[r], lam2, true), w};
                }
                if (e < E) {
                    key[q] = sl[q].cf & kColMask;
                    sm.key[warp][e] = key[q];
                }
            }
            __syncwarp();
            // the columns of a row are distinct: the rank is the place in column order
            for (int t = 0; t < E; ++t) {
                const unsigned kt = sm.key[warp][t];
#pragma unroll
                for (int q = 0; q < kSlots / 32; ++q) rank[q] += kt < key[q] ? 1 : 0;
            }
#pragma unroll
            for (int q = 0; q < kSlots / 32; ++q) {
                if (lane + 32 * q < E) {
                    const Ent<T> x = sl[q];
                    if (!(x.g == x.g) || isinf((double)x.g)) ++bad;
                    if ((int)key[q] == i) { s_g[r] = x.g; s_w[r] = x.w; }
                    st_ent(k.ents + (size_t)i * kSlots + rank[q], x.cf, x.om, x.g, x.w);
                }
            }
            if (lane == 0) k.len[i] = E;
            __syncwarp();
        }
        __syncthreads();

        // ---------------- search
        int h_base = 0;
        bool first = true;
        for (;;) {
            const int nwin = first && last_h >= kWin - 1 ? 2 : 1;
            for (int wn = 0; wn < nwin; ++wn) {
                const int hb = h_base + wn * kWin;
                A q[kWin]{}, n2[kWin]{}, ph[kWin]{};
                int ib[kWin], iz[kWin];
#pragma unroll
                for (int m = 0; m < kWin; ++m) ib[m] = iz[m] = 0;
                // diagonal terms of every owned row; rows with nothing else are complete here
                for (int r = tid; r < nr; r += kLT) {
                    const T o = s_om[r], g = s_g[r];
                    const bool alone = s_rc[r] == -1;
                    const T sd = s_sd[r];
#pragma unroll
                    for (int m = 0; m < kWin; ++m) {
                        const T tau = tau_pow2<T>(hb + m);
                        const T np = prox_entry(o, g, tau, tau * lam1, true);
                        const T d = np - o;
                        if (!(np > T(0))) ++ib[m];
                        else acc_add(ph[m], phiT(d / o));
                        acc_add(n2[m], mulT(d, d));
                        if (alone) {
                            acc_add(q[m], mulT(mulT(d, d), sd));
                            ++iz[m];
                        }
                    }
                }
                // the other rows, in units: the pair (a, b) of 32-entry chunks of a row, a <= b
                auto unit = [&](int i, const Ent<T>* re, int L, int a, int b) {
                    const int e = a + lane;
                    Ent<T> x{0u, T(0), T(0), T(0)};
                    T de[kWin];
                    bool act = false;
                    if (e < L) x = ld_ent(re + e);
                    const int je = (int)(x.cf & kColMask);
                    const bool diag = e < L && je == i;
#pragma unroll
                    for (int m = 0; m < kWin; ++m) {
                        const T tau = tau_pow2<T>(hb + m);
                        const T np = prox_entry(x.om, x.g, tau, tau * lam1, diag);
                        de[m] = e < L ? np - x.om : T(0);
                        act |= de[m] != T(0);
                        if (a == b) {
                            if (e < L && (diag || np != T(0))) ++iz[m];
                            if (!diag) acc_add(n2[m], mulT(de[m], de[m]));
                        }
                    }
                    if (first && wn == 0 && a == b && (x.cf & kFSupp)) acc_add(o2, mulT(x.om, x.om));
                    T df[kWin];
                    int jf = je;
                    bool af = act;
                    if (b == a) {
#pragma unroll
                        for (int m = 0; m < kWin; ++m) df[m] = de[m];
                    } else {
                        const int f = b + lane;
                        Ent<T> y{0u, T(0), T(0), T(0)};
                        if (f < L) y = ld_ent(re + f);
                        jf = (int)(y.cf & kColMask);
                        af = false;
#pragma unroll
                        for (int m = 0; m < kWin; ++m) {
                            const T tau = tau_pow2<T>(hb + m);
                            const T np = prox_entry(y.om, y.g, tau, tau * lam1, f < L && jf == i);
                            df[m] = f < L ? np - y.om : T(0);
                            af |= df[m] != T(0);
                        }
                    }
                    unsigned bits = __ballot_sync(kFull, af);
                    sm.jf[warp][lane] = (unsigned)jf;
#pragma unroll
                    for (int m = 0; m < kWin; ++m) sm.del[warp][m][lane] = df[m];
                    __syncwarp();
                    if (act) {
                        T qf[kWin];
#pragma unroll
                        for (int m = 0; m < kWin; ++m) qf[m] = T(0);
                        const T* srow = k.S + (int64_t)je * k.ld;
                        while (bits) {
                            int t[4];
                            T sv[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                t[u] = bits ? __ffs(bits) - 1 : -1;
                                bits &= bits - 1;           // 0 stays 0
                                const bool use = t[u] >= 0 && (a != b || t[u] >= lane);
                                sv[u] = use ? __ldg(srow + sm.jf[warp][t[u] & 31]) : T(0);
                                // a pair of different entries counts twice (exact)
                                if (!(a == b && t[u] == lane)) sv[u] = sv[u] + sv[u];
                            }
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (t[u] >= 0) {
#pragma unroll
                                    for (int m = 0; m < kWin; ++m)
                                        qf[m] = fmaT(mulT(de[m], sm.del[warp][m][t[u]]), sv[u], qf[m]);
                                }
                            }
                        }
#pragma unroll
                        for (int m = 0; m < kWin; ++m) acc_add(q[m], qf[m]);
                    }
                    __syncwarp();
                };
                // a row of one chunk per warp; the units of longer rows dealt to the warps
                for (int li = warp; li < nsmall; li += kLW) {
                    const int r = s_list[li];
                    unit(i0 + r, ents_of(r), k.len[i0 + r], 0, 0);
                }
                for (int li = nsmall, u0 = 0; li < nlong; ++li) {
                    const int r = row_at(li), L = k.len[i0 + r], nc = (L + 31) / 32;
                    const Ent<T>* re = ents_of(r);
                    for (int a = 0; a < nc; ++a)
                        for (int b = a; b < nc; ++b, ++u0)
                            if (u0 % kLW == warp) unit(i0 + r, re, L, 32 * a, 32 * b);
                }
                // block sums of the window: the warp, then the warps in order.  The warp's sums of
                // sixteen quantities together: at every step half of them go to each half of the
                // lanes (16 merges instead of 12 butterflies of 5); lane 2 q ends with quantity q.
                const bool works = 32 * warp < nr || warp < nsmall || nlong > nsmall;
                if (works) {
                    A v[16]{};
#pragma unroll
                    for (int m = 0; m < kWin; ++m) {
                        v[3 * m] = q[m];
                        v[3 * m + 1] = n2[m];
                        v[3 * m + 2] = ph[m];
                    }
                    if (first && wn == 0) v[kQA] = o2;
#pragma unroll
                    for (int o = 16, n = 8; n >= 1; o >>= 1, n >>= 1) {
                        const bool up = lane & o;
#pragma unroll
                        for (int x = 0; x < n; ++x) {
                            A mine = up ? v[x + n] : v[x];
                            const A other = shfl_xor_acc(up ? v[x] : v[x + n], o);
                            acc_merge(mine, other);
                            v[x] = mine;
                        }
                    }
                    acc_merge(v[0], shfl_xor_acc(v[0], 1));
                    const int qi = lane >> 1;
                    if (!(lane & 1)) {
                        if (qi < kQA) sm.red_a[warp][wn * kQA + qi] = acc_value(v[0]);
                        else if (qi == kQA && first && wn == 0) sm.red_a[warp][2 * kQA] = acc_value(v[0]);
                    }
                } else {
                    if (lane < kQA) sm.red_a[warp][wn * kQA + lane] = 0.0;
                    if (lane == kQA && first && wn == 0) sm.red_a[warp][2 * kQA] = 0.0;
                }
#pragma unroll
                for (int m = 0; m < kWin; ++m) {
                    const int d = __reduce_add_sync(kFull, ib[m]), e = __reduce_add_sync(kFull, iz[m]);
                    if (lane == 0) {
                        sm.red_i[warp][wn * kQI + 2 * m] = d;
                        sm.red_i[warp][wn * kQI + 2 * m + 1] = e;
                    }
                }
            }
            if (first) {
                const int d = __reduce_add_sync(kFull, em), e = __reduce_add_sync(kFull, bad),
                          f = __reduce_add_sync(kFull, full);
                if (lane == 0) {
                    sm.red_i[warp][2 * kQI] = d;
                    sm.red_i[warp][2 * kQI + 1] = e;
                    sm.red_i[warp][2 * kQI + 2] = f;
                    sm.red_i[warp][2 * kQI + 3] = warp == 0 ? sm.halves : 0;
                    sm.red_i[warp][2 * kQI + 4] = warp == 0 ? sm.off : 0;
                }
            }
            __syncthreads();
            const int na = nwin * kQA, nii = nwin * kQI;
            for (int t = tid; t < kNA + kNI; t += kLT) {
                if (t < kNA) {
                    if (t < na || (first && t == 2 * kQA)) {
                        k.part_a[((size_t)pbuf * kNA + t) * nb + bid] = warps_sum(sm.red_a, t);
                    }
                } else {
                    const int u = t - kNA;
                    if (u < nii || (first && u >= 2 * kQI)) {
                        int a = 0;
                        for (int w = 0; w < kLW; ++w) a += sm.red_i[w][u];
                        k.part_i[((size_t)pbuf * kNI + u) * nb + bid] = a;
                    }
                }
            }
            alive = loop_barrier(k.bar, target, ctrl, &sm.ok);
            if (!alive) break;
            // ---------------- decide: every block the same sums in the same order, eight lanes
            // per quantity
            static_assert((kNA + kNI) * 8 <= kLT, "one pass over the quantities");
            {
                const int t = tid >> 3, sub = tid & 7;
                double a = 0.0;
                int c = 0, pre = 0;
                if (t < kNA) {
                    if (t < na || (first && t == 2 * kQA)) {
                        const double* src = k.part_a + ((size_t)pbuf * kNA + t) * nb;
#pragma unroll 8
                        for (int b = sub; b < nb; b += 8) a += __ldcg(src + b);
                    }
                } else if (t < kNA + kNI) {
                    const int u = t - kNA;
                    if (u < nii || (first && u >= 2 * kQI)) {
                        const int* src = k.part_i + ((size_t)pbuf * kNI + u) * nb;
#pragma unroll 8
                        for (int b = sub; b < nb; b += 8) {
                            const int v = __ldcg(src + b);
                            c += v;
                            pre += b < bid ? v : 0;
                        }
                    }
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    a += __shfl_xor_sync(kFull, a, o);
                    c += __shfl_xor_sync(kFull, c, o);
                    pre += __shfl_xor_sync(kFull, pre, o);
                }
                // quantities that this window did not write keep their earlier sums
                if (sub == 0 && t < kNA && (t < na || (first && t == 2 * kQA))) sm.sum_a[t] = a;
                if (sub == 0 && t >= kNA && t < kNA + kNI && (t - kNA < nii || (first && t - kNA >= 2 * kQI))) {
                    sm.sum_i[t - kNA] = c;
                    sm.pre_i[t - kNA] = pre;
                }
            }
            pbuf ^= 1;
            __syncthreads();
            if (warp == 0) {
                // lane x: step size h_base + x
                int flags = 0, full_rows = 0;
                if (first) {
                    // the entries emitted, against the handle's candidate capacity (as the chain's
                    // list has them: up to p / 2 rows with neighbours, two rows with the
                    // diagonal alone emit both entries or none)
                    if (lane == 0 && 2 * sm.sum_i[2 * kQI + 4] <= k.p) sm.sum_i[2 * kQI] += sm.sum_i[2 * kQI + 3];
                    __syncwarp();
                    if (sm.sum_i[2 * kQI] > k.em_cap) flags = kFlagEmOverflow;
                    else if (sm.sum_i[2 * kQI + 2] > 0) full_rows = 1;
                    else if (sm.sum_i[2 * kQI + 1] > 0) flags = kFlagNaN;
                }
                int accept = -1;
                if (!flags && !full_rows) {
                    const int w = lane / kWin, m = lane % kWin, h = h_base + lane;
                    bool pass = false, nan = false;
                    if (w < nwin && h <= k.max_halvings && sm.sum_i[w * kQI + 2 * m] == 0) {
                        const double* x = sm.sum_a + w * kQA + 3 * m;
                        const double excess = 0.5 * x[0] + 0.5 * lam2d * x[1] + x[2];
                        // excess <= ||D||^2 / (2 tau), 1 / (2 tau) = 2^(h-1) exactly (h <= 1000)
                        pass = excess <= x[1] * __longlong_as_double((long long)(1022 + h) << 52);
                        nan = !pass && !(excess == excess);
                    }
                    const unsigned bp = __ballot_sync(kFull, pass), bn = __ballot_sync(kFull, nan);
                    if (bp | bn) {
                        const int x = __ffs(bp | bn) - 1;
                        if ((bp >> x) & 1u) accept = h_base + x;
                        else flags = kFlagNaN;
                    } else if (h_base + nwin * kWin > k.max_halvings) {
                        flags = kFlagLsFail;
                    }
                    if (accept >= 0 && lane == accept - h_base) {
                        sm.n2 = sm.sum_a[w * kQA + 3 * m + 1];
                        sm.nnz = sm.sum_i[w * kQI + 2 * m + 1];
                        sm.nnz_pre = sm.pre_i[w * kQI + 2 * m + 1];
                    }
                    __syncwarp();
                    if (accept >= 0 && sm.nnz > k.csr_cap) flags |= kFlagNnzOverflow;
                }
                if (lane == 0) {
                    sm.flags = flags;
                    sm.full = full_rows;
                    sm.accept = accept;
                }
            }
            __syncthreads();
            h_base += nwin * kWin;
            first = false;
            if (sm.flags || sm.full || sm.accept >= 0) break;
        }
        if (!alive || sm.flags || sm.full) break;
        const int h = sm.accept;
        last_h = h;
        trials += h + 1;
        nnz_now = sm.nnz;

        // ---------------- accept: the owned rows of Omega+
        const T tau = tau_pow2<T>(h), tl1 = tau * lam1;
        const int par2 = par ^ 1;
        if (tid == 0) { sm.ni = 0; sm.npl = 0; sm.sup = 0; sm.units = 0; sm.halves = 0; sm.off = 0; }
        __syncthreads();
        if (bid == 0 && tid == 0) { k.ctr[kCtrPage] = 0; k.ctr[kCtrFull] = 0; }
        // entries per row (s_rc of a long row becomes its entry count)
        for (int li = warp; li < nlong; li += kLW) {
            const int r = row_at(li), i = i0 + r;
            const int L = k.len[i];
            const Ent<T>* re = ents_of(r);
            int c = 0;
            for (int a = 0; a < L; a += 32) {
                bool nz = false;
                if (a + lane < L) {
                    const Ent<T> x = ld_ent(re + a + lane);
                    nz = (int)(x.cf & kColMask) == i || prox_entry(x.om, x.g, tau, tl1, false) != T(0);
                }
                c += __popc(__ballot_sync(kFull, nz));
            }
            if (lane == 0) s_rc[r] = c;
        }
        __syncthreads();
        // exclusive scan over the owned rows, then rows with only the diagonal
        int run_base = sm.nnz_pre;
        for (int r0 = 0; r0 < nr; r0 += kLT) {
            const int r = r0 + tid;
            const bool in = r < nr;
            const bool alone = in && s_rc[r] == -1;
            const int c = in ? (alone ? 1 : s_rc[r]) : 0;
            const int incl = warp_incl_scan(c, lane);
            if (lane == 31) sm.wsum[warp] = incl;
            __syncthreads();
            int before = run_base, all = 0;
#pragma unroll
            for (int w = 0; w < kLW; ++w) {
                before += w < warp ? sm.wsum[w] : 0;
                all += sm.wsum[w];
            }
            const int start = before + incl - c;
            if (in) {
                const int i = i0 + r;
                out.rp[i] = start;
                s_rb[r] = start;
                if (alone) {
                    const T v = prox_entry(s_om[r], s_g[r], tau, tl1, true);
                    out.ci[start] = i;
                    out.cv[start] = v;
                    k.rinfo[i] = make_int4(start, start + 1, start, 1);
                    k.rds[i] = v;
                    s_dv[r] = v;
                    s_mv[r] = 0;
                    if (k.m1 && !(mulT(v, (T)s_m1[r]) <= lam1)) s_pl[atomicAdd(&sm.npl, 1)] = r;
                }
                if (i == k.p - 1) out.rp[k.p] = start + c;
            }
            run_base += all;
            __syncthreads();
        }
        if (tid == 0) { sm.e0 = sm.nnz_pre; sm.e1 = run_base; }
        for (int li = warp; li < nlong; li += kLW) {
            const int r = row_at(li), i = i0 + r;
            const int L = k.len[i];
            const Ent<T>* re = ents_of(r);
            const int rb = s_rb[r];
            int o = rb, pd = -1;
            T dv = T(0);
            float sw = 0.0f;
            for (int a = 0; a < L; a += 32) {
                bool nz = false, dg = false;
                int j = 0;
                T v = T(0);
                if (a + lane < L) {
                    const Ent<T> x = ld_ent(re + a + lane);
                    j = (int)(x.cf & kColMask);
                    dg = j == i;
                    v = prox_entry(x.om, x.g, tau, tl1, dg);
                    nz = dg || v != T(0);
                    sw = __fadd_ru(sw, abs_up(v));
                }
                const unsigned bal = __ballot_sync(kFull, nz), bd = __ballot_sync(kFull, dg);
                const int q = o + __popc(bal & ((1u << lane) - 1u));
                if (nz) { out.ci[q] = j; out.cv[q] = v; }
                if (bd) {
                    const int src = __ffs(bd) - 1;
                    pd = __shfl_sync(kFull, q, src);
                    dv = __shfl_sync(kFull, v, src);
                }
                o += __popc(bal);
            }
            const bool pure = o - rb == 1;
            const bool init = !s_mv[r];
            __syncwarp();
            if (!pure) {
                int at = 0;
                if (lane == 0) {
                    at = atomicAdd(&sm.ni, o - rb);
                    atomicAdd(&sm.sup, row_sup(o - rb));
                    atomicAdd(&sm.off, 1);
                }
                at = __shfl_sync(kFull, at, 0);
                for (int q = lane; q < o - rb; q += 32)
                    if (at + q < kItemCap) { sm.items[at + q] = rb + q; sm.item_r[at + q] = (short)r; }
            }
            if (lane == 0) {
                k.rinfo[i] = make_int4(rb, o, pd, pure ? 1 : 0);
                k.rds[i] = pure ? dv : -dv;
                s_dv[r] = dv;
                s_rc[r] = pure ? -1 : 0;
                s_mv[r] = pure ? 0 : 1;
                if (pure && k.m1 && !(mulT(dv, (T)s_m1[r]) <= lam1)) s_pl[atomicAdd(&sm.npl, 1)] = r;
            }
            if (!pure && k.bnd) {
                const float slack = slack_of<T>(o - rb + 1, warp_sum_up(sw), mg);
                if (lane == 0) k.slack[i] = slack;
                bound_row(k, i, L, init, o - rb, slack, lam1, par2, lane, [&](int e, int& c, float& w, bool& left) {
                    const Ent<T> x = ld_ent(re + e);
                    c = (int)(x.cf & kColMask);
                    const T v = prox_entry(x.om, x.g, tau, tl1, c == i);
                    // the change itself is rounded: a little more than half a unit covers it
                    w = init ? abs_up(v) : __fmul_ru(abs_up(v - x.om), 1.0f + 0x1p-22f);
                    left = !init && (x.cf & kFSupp) && c != i && v == T(0);
                });
            }
        }
        __syncthreads();
        if (k.m1)
            for (int li = warp; li < sm.npl; li += kLW) pure_row_tasks(k, i0 + s_pl[li], s_dv[s_pl[li]], lam1, par2, lane);
        // the stopping rule ||dOmega||_F < eps ||Omega||_F
        if (tid == 0) {
            sm.converged = sm.n2 < (k.eps * k.eps) * sm.sum_a[2 * kQA] ? 1 : 0;
            sm.more = iter + 1 < iter_limit && !(use_stop && sm.converged);
        }
        __syncthreads();
        ++iter;
        buf ^= 1;
        par = par2;
        run = sm.more != 0;
        if (run) alive = loop_barrier(k.bar, target, ctrl, &sm.ok);
        if (!alive) break;
    }

    if (!alive) {
        // a wait gave up: the flag is up, and the host reports it
        if (bid == 0 && tid == 0) end_loops(k);
        return;
    }
    // ---------------- the accepted iterate back into `cur` (own rows: written by this block)
    __syncthreads();
    if (buf && nr > 0) {
        const int e0 = k.next.rp[i0];
        for (int r = tid; r < nr; r += kLT) k.cur.rp[i0 + r] = k.next.rp[i0 + r];
        if (i0 + nr == k.p) {
            if (tid == 0) k.cur.rp[k.p] = k.next.rp[k.p];
        }
        // this block's entries: up to its last row's end
        const int4 last = __ldcg(k.rinfo + i0 + nr - 1);
        for (int q = e0 + tid; q < last.y; q += kLT) {
            k.cur.ci[q] = k.next.ci[q];
            k.cur.cv[q] = k.next.cv[q];
        }
    }
    // ---------------- the objective at the last gradient pass
    if (attempts > 0 && !sm.full && !(sm.flags & kFlagEmOverflow)) {
        A ow{}, lg{}, ab{};
        for (int r = tid; r < nr; r += kLT) {
            const int i = i0 + r;
            const T o = s_om[r];
            acc_add(ow, mulT(o, s_w[r]));
            acc_add(lg, logT(o));
            const int L = k.len[i];
            const Ent<T>* re = L == 0 || s_eo[r] < 0 ? k.ents + (size_t)i * kSlots : k.big + s_eo[r];
            k.eoff[i] = L == 0 ? -1 : s_eo[r];
            // a row of the diagonal alone: its candidate, for the host's queries
            if (L == 0) st_ent(k.ents + (size_t)i * kSlots, (unsigned)i | kFSupp, o, s_g[r], s_w[r]);
            for (int e = 0; e < L; ++e) {
                const Ent<T> x = ld_ent(re + e);
                if ((x.cf & kFSupp) && (int)(x.cf & kColMask) != i) {
                    acc_add(ow, mulT(x.om, x.w));
                    acc_add(ab, (T)fabs(x.om));
                }
            }
        }
        const A a = warp_sum(ow), b = warp_sum(lg), c = warp_sum(ab);
        if (lane == 0) {
            sm.red_a[warp][0] = acc_value(a);
            sm.red_a[warp][1] = acc_value(b);
            sm.red_a[warp][2] = acc_value(c);
        }
        __syncthreads();
        if (tid < 3) k.part_a[((size_t)pbuf * kNA + tid) * nb + bid] = warps_sum(sm.red_a, tid);
        if (!loop_barrier(k.bar, target, ctrl, &sm.ok)) {
            if (bid == 0 && tid == 0) end_loops(k);
            return;
        }
        if (bid == 0 && warp < 3) {
            double x = 0.0;
            for (int t = lane; t < nb; t += 32) x += __ldcg(k.part_a + ((size_t)pbuf * kNA + warp) * nb + t);
            x = warp_sum(x);
            if (lane == 0) sm.red_a[0][kQA + warp] = x;
        }
        __syncthreads();
        if (bid == 0 && tid == 0) {
            const double norm2 = sm.sum_a[2 * kQA];
            ctrl->f_cur = -sm.red_a[0][kQA + 1] + 0.5 * sm.red_a[0][kQA] + 0.5 * lam2d * norm2;
            ctrl->pen_cur = ctrl->lam1 * sm.red_a[0][kQA + 2];
            ctrl->norm2_cur = norm2;
        }
    }
    if (bid == 0 && tid == 0) {
        ctrl->iter = iter;
        ctrl->iter_attempts += attempts;
        ctrl->loop_attempts += attempts;
        ctrl->loop_launches += 1;
        ctrl->ls_trials += trials;
        ctrl->screen_ns += screen_ns;
        ctrl->nnz_cur = nnz_now;
        if (attempts > 0) {
            ctrl->flags = sm.flags;
            ctrl->em_count = sm.sum_i[2 * kQI];
            ctrl->ls_accept = sm.accept;
            ctrl->converged = sm.flags || sm.full ? 0 : sm.converged;
            if (sm.accept >= 0 && !sm.full) {
                ctrl->nnz_next = sm.nnz;
                if (!sm.flags) {
                    ctrl->tau = tau_pow2<double>(sm.accept);
                    ctrl->delta2 = sm.n2;
                    ctrl->rel = sqrt(sm.n2) / sqrt(ctrl->norm2_cur);
                }
            }
        }
        const int leave = sm.full || (dense && run) ? 1 : 0;
        ctrl->loop_full = leave;
        ctrl->loop_debt = leave ? 0u : sm.debt;
        if (leave) ctrl->chain_left = 1 << min(ctrl->loop_fulls++, 6);
        if (k.use_cond) {
            cudaGraphSetConditional(k.chain_cond, leave ? 1u : 0u);
            cudaGraphSetConditional(k.outer_cond, leave ? 1u : 0u);
        }
    }
}

// Before the loop: its counters.
template <typename T>
__global__ void k_loop_arm(LoopK<T> k) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
    for (int i = t; i < k.p; i += n) k.cnt[i] = 0;
    for (size_t i = t; i < (size_t)k.p * kPages; i += n) k.pages[i] = 0;
    if (t < kCtrCount) k.ctr[t] = 0;
    if (t < 2) k.todo[t] = make_ulonglong2(0, 0);
    if (t == 0) {
        *k.bar = 0u;
        *k.mg = 0u;
        k.ctrl->flags = 0;
        k.ctrl->ls_accept = -1;
        k.ctrl->converged = 0;
    }
}

// The candidates of the last pass, row by row, a warp per row: row i's from place at[i] on, n in all.
template <typename T>
__global__ void __launch_bounds__(256) k_loop_candidates(LoopK<T> k, const int* __restrict__ at, int64_t n,
                                                         LoopCandidate* __restrict__ out) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= k.p) return;
    const int L = max(1, k.len[i]), off = k.eoff[i];
    if (off >= 0 && off + L > 2 * k.npool * kSlots) return;
    const Ent<T>* e = off < 0 ? k.ents + (size_t)i * kSlots : k.big + off;
    for (int q = threadIdx.x & 31; q < min(L, off < 0 ? kSlots : L) && at[i] + q < n; q += 32) {
        const Ent<T> x = ld_ent(e + q);
        out[at[i] + q] = LoopCandidate{i, (int)(x.cf & kColMask), (double)x.om, (double)x.g};
    }
}

size_t align256(size_t b) { return (b + 255) / 256 * 256; }

template <typename T>
LoopK<T> loop_args(const IterBufs<T>& b, void* ws, int R, size_t* bytes) {
    LoopK<T> k{};
    k.S = b.S;
    k.ld = b.ld;
    k.p = b.p;
    k.R = R;
    k.cur = b.cur;
    k.next = b.next;
    k.csr_cap = b.csr_cap;
    k.em_cap = b.em.cap;
    k.cnt = b.bk.cnt;
    k.len = b.bk.len;
    k.rinfo = b.rinfo;
    k.rds = b.rdv;
    k.bar = b.bar;
    k.ctrl = b.ctrl;
    k.symmetric = b.symmetric;
    k.eps = b.eps;
    k.max_halvings = b.max_halvings;
    k.m1 = b.m1;
    k.m1g = b.m1 ? b.m1g : nullptr;
    k.nbm = b.nbm;
    k.ngl = b.ngl;
    k.symmetric = b.symmetric;
    uint8_t* q = static_cast<uint8_t*>(ws);
    auto take = [&](size_t n) { uint8_t* r = q; q += align256(n); return r; };
    const size_t p = (size_t)b.p;
    k.slots = reinterpret_cast<Ent<T>*>(take(p * kSlots * sizeof(Ent<T>)));
    k.ents = reinterpret_cast<Ent<T>*>(take(p * kSlots * sizeof(Ent<T>)));
    k.npool = (int)std::max<size_t>(64, p / 8);
    k.pages = reinterpret_cast<int*>(take(p * kPages * sizeof(int)));
    k.pool = reinterpret_cast<Ent<T>*>(take((size_t)k.npool * kSlots * sizeof(Ent<T>)));
    // rows with a page fit twice the pool
    k.big = reinterpret_cast<Ent<T>*>(take(2 * (size_t)k.npool * kSlots * sizeof(Ent<T>)));
    k.eoff = reinterpret_cast<int*>(take(p * sizeof(int)));
    k.nbp = (b.nbm + 7) / 8 * 8;
    k.ntask_cap = (int)std::min<size_t>(p * (size_t)b.nbm / 4 + 65536, (size_t)1 << 28);
    k.tasks = reinterpret_cast<int*>(take(2 * (size_t)k.ntask_cap * sizeof(int)));
    k.bnd = reinterpret_cast<float*>(take(p * k.nbp * sizeof(float)));
    if (!b.m1) k.bnd = nullptr;
    k.slack = reinterpret_cast<float*>(take(p * sizeof(float)));
    k.mg = reinterpret_cast<unsigned*>(take(sizeof(unsigned)));
    k.part_a = reinterpret_cast<double*>(take(2 * (size_t)kNA * b.num_sms * sizeof(double)));
    k.part_i = reinterpret_cast<int*>(take(2 * (size_t)kNI * b.num_sms * sizeof(int)));
    k.ctr = reinterpret_cast<int*>(take(kCtrCount * sizeof(int)));
    k.todo = reinterpret_cast<ulonglong2*>(take(2 * sizeof(ulonglong2)));
    if (bytes) *bytes = (size_t)(q - static_cast<uint8_t*>(ws));
    return k;
}

}  // namespace

// Rows per block and blocks: at least 8 rows (one per half warp pair of work) per
// block, at most one block per SM.  0 blocks: the sizes do not fit the loop.
template <typename T>
int loop_grid(int p, int nbm, int num_sms, int* rows) {
    const int nb = std::max(1, std::min(num_sms, (p + 7) / 8));
    const int R = (p + nb - 1) / nb;
    if (rows) *rows = R;
    if (R > kMaxR || (long long)p * nbm > 0x7fffffffll ||
        loop_smem_bytes<T>(R) > 220 * 1024)
        return 0;
    int v = 0;
    if (set_smem_once((const void*)k_loop<T>, 220 * 1024, sizeof(T) == 4 ? kSmemSlotLoopF : kSmemSlotLoopD) !=
        cudaSuccess)
        return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_loop<T>, kLT, loop_smem_bytes<T>(R)) != cudaSuccess ||
        v < 1)
        return 0;
    return (p + R - 1) / R;
}

template <typename T>
size_t loop_workspace_bytes(int p, int nbm, int num_sms) {
    IterBufs<T> b{};
    b.p = p;
    b.nbm = nbm;
    b.num_sms = num_sms;
    size_t n = 0;
    loop_args<T>(b, nullptr, 1, &n);
    return n;
}

template <typename T>
cudaError_t loop_candidate_places(const IterBufs<T>& b, std::vector<int>& at, int64_t* n, cudaStream_t s) {
    at.resize((size_t)b.p);
    cudaError_t e = cudaMemcpyAsync(at.data(), b.bk.len, at.size() * sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    *n = 0;
    for (int& a : at) {
        const int L = std::max(1, a);
        a = (int)*n;
        *n += L;
    }
    return e;
}

size_t loop_candidate_bytes(int64_t p, int64_t n) {
    return align256((size_t)p * sizeof(int)) + (size_t)n * sizeof(LoopCandidate);
}

template <typename T>
cudaError_t loop_candidates(const IterBufs<T>& b, void* ws, const std::vector<int>& at, int64_t n, void* tmp,
                            LoopCandidate* out, cudaStream_t s) {
    const LoopK<T> k = loop_args<T>(b, ws, 1, nullptr);
    LoopCandidate* d = reinterpret_cast<LoopCandidate*>(static_cast<uint8_t*>(tmp) + align256(at.size() * sizeof(int)));
    cudaError_t e = cudaMemcpyAsync(tmp, at.data(), at.size() * sizeof(int), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    k_loop_candidates<T><<<(unsigned)((b.p + 7) / 8), 256, 0, s>>>(k, static_cast<const int*>(tmp), n, d);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = cudaMemcpyAsync(out, d, (size_t)n * sizeof(LoopCandidate), cudaMemcpyDeviceToHost, s);
    return e != cudaSuccess ? e : cudaStreamSynchronize(s);
}

template <typename T>
cudaError_t launch_loop(const IterBufs<T>& b, void* ws, const LoopCond& lc, cudaStream_t s) {
    int R = 0;
    const int nb = loop_grid<T>(b.p, b.nbm, b.num_sms, &R);
    if (nb < 1) return cudaErrorInvalidConfiguration;
    LoopK<T> k = loop_args<T>(b, ws, R, nullptr);
    k.use_cond = lc.use;
    k.chain_cond = lc.iter;
    k.outer_cond = lc.outer;
    k_loop_arm<T><<<std::max(1, std::min(2 * b.num_sms, (b.p + 15) / 16)), 256, 0, s>>>(k);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)nb);
    cfg.blockDim = dim3(kLT);
    cfg.dynamicSmemBytes = loop_smem_bytes<T>(R);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_loop<T>, k);
}

#define HPC_LOOP_INSTANTIATE(T)                                                                              \
    template int loop_grid<T>(int, int, int, int*);                                                          \
    template size_t loop_workspace_bytes<T>(int, int, int);                                                  \
    template cudaError_t loop_candidate_places<T>(const IterBufs<T>&, std::vector<int>&, int64_t*, cudaStream_t); \
    template cudaError_t loop_candidates<T>(const IterBufs<T>&, void*, const std::vector<int>&, int64_t, void*,   \
                                            LoopCandidate*, cudaStream_t);                                   \
    template cudaError_t launch_loop<T>(const IterBufs<T>&, void*, const LoopCond&, cudaStream_t);

HPC_LOOP_INSTANTIATE(float)
HPC_LOOP_INSTANTIATE(double)

}  // namespace hpc
