// bound.cu -- bound of candidate allocations on fixed schedule structures, and the argmin
// over candidates per DAG.
//
// A plan is the schedule of one structure variant: rows ordered by the group they run in,
// each with its load, parallel fraction and scheduled SMs. For candidate allocation m^c
// the bound is a max-plus sweep along the group chain (Theorem 1): F_j = F_{j-1} + R_j,
// with R_j = max C_i over the group if its SMs fit in M (Lemma 1), else sum C_i.
//
// Three paths. Materialised candidates in blocks of 64 (n_alloc a multiple of 64) take the
// balanced work items (k_bound_items + k_bound_finish, below): chunks of whole groups of
// every plan, one warp per (chunk, 64-candidate block), its rows staged by 2-D TMA tensor
// copies, partial bounds added into per-candidate accumulators. The exhaustive search
// enumerates per DAG (k_bound_exhaustive). Everything else (random levels, perturbations,
// other n_alloc) takes k_bound_rows: one CTA per DAG, its warps sharing windows of plan rows.
#include <cooperative_groups.h>
#include <cuda.h>  // CUtensorMap and its encoding enums (header only)

#include <cstring>
#include <type_traits>

#include "bound.cuh"
#include "dagrt_internal.cuh"

namespace dagrt {

constexpr uint32_t kSpinLimit = 1u << 24;  // bounded mbarrier wait

// ------------------------------------------------------------------ TMA / mbarrier
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// global -> shared bulk copy (16-byte aligned addresses, size a multiple of 16)
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// bounded wait on a stage; false after `limit` polls
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint32_t limit = kSpinLimit) {
    for (uint32_t i = 0; i < limit; i++)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__global__ void k_selftest_wait(uint32_t limit, int32_t *word) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    // nothing arrives: the wait must give up and report, leaving the CTA free to exit
    const bool ok = mbar_wait(&bar, 0, limit);
    if (!ok && threadIdx.x == 0) atomicExch(word, DAGRT_E_TIMEOUT);
}

cudaError_t bound_selftest_wait(uint32_t limit, int32_t *word, cudaStream_t st) {
    k_selftest_wait<<<1, 32, 0, st>>>(limit, word);
    return cudaGetLastError();
}

// argmin helper: smaller bound wins, then the smaller candidate id
__device__ __forceinline__ void better(int64_t &bb, int32_t &bc, int64_t ob, int32_t oc) {
    if (oc < 0) return;
    if (bc < 0 || ob < bb || (ob == bb && oc < bc)) {
        bb = ob;
        bc = oc;
    }
}

// SMs of plan row `row` (owner node `owner`, scheduled on m0 SMs) for generated candidate c
// of DAG d; 0 keeps the schedule's m.
__device__ __forceinline__ uint32_t gen_alloc(const BoundArgs &a, int d, int c, int row, uint32_t owner, uint32_t m0,
                                              const uint8_t *s_lev) {
    const int al = c % a.n_alloc;
    if (a.gen_mode == DAGRT_SEARCH_EXHAUSTIVE) {
        const uint32_t dg = exh_digit((uint32_t)al, owner, (uint32_t)a.n_levels + 1u);
        return dg ? s_lev[dg - 1] : 0u;
    }
    if (al == 0) return 0u;
    const uint32_t x = s_lev[gen_level(a.seed, d, c, row, a.n_levels)];
    if (a.gen_mode != DAGRT_SEARCH_PERTURB) return x;
    return x == 0 ? 0u : perturb_m(m0, x);  // code 0 keeps the row's own m (even above 255)
}

// ------------------------------------------------------------------ rows of one DAG per CTA
// Candidates that the balanced work items below do not take: generated ones (random levels,
// perturbations) and materialised ones whose count is not a multiple of 64. One CTA takes a
// DAG; its warps share the DAG's (variant, window of kRowWindow plan rows, block of 32 CPT
// candidates) tasks, so a DAG of 1,000 rows keeps 16 warps busy, where one thread per
// candidate walked all rows of its variant alone. A window's groups are those that start in
// it: no chunk index is needed, nor scratch in global memory, and partial bounds add up in
// shared memory (Theorem 1's sum splits at group ends).
//
// Eq.1's division is out of the inner loop: generated candidates look {C, m} up in a table of the
// row's few possible choices, and a byte m <= M divides by 64 m with a multiply and a shift. Per
// candidate and row that leaves SplitMix64 (two 64-bit multiplications) or ten instructions. What
// bounds it: perturbations issue in 59% of the cycles with 16 warps an SM, between dependent
// instructions for the most part; bytes of 74 candidates in 42% with 22 warps, which wait at the
// DAGs' barriers (3.7 of 13 cycles between a warp's instructions) and for loads. Two candidates
// a lane above 32 allocations (one: 359 us instead of 279 below). Windows of 32 rows: 64 and
// 128 take 65 and 92 us instead of 58 on the second workload, the first does not care.
// 500 DAGs of 100-1,000 nodes x 256 perturbations: 3.06 -> 0.28 ms; 1,000 DAGs of 20-200 nodes
// x 74 allocations: 116 -> 53 us a call; 5,000 DAGs of 3-6 nodes x 100 allocations: 31 -> 29.
constexpr int kRowWindow = 32;
constexpr int kRowTile = 2048;   // candidates of one pass over the DAG (shared-memory sums)
enum { SRC_BYTES = 0, SRC_RANDOM = 1, SRC_PERTURB = 2 };
constexpr int kPerturbCodes = 5;

// n / (64 m) for n < 2^31 as (n * x >> 32) >> y: x = ceil(2^(32+y) / 64 m), exact while
// n (64 m x - 2^(32+y)) < 2^(32+y). Not a power of two: 2^y > 32 m, the bracket is below
// 64 m <= 16320 and n < 2^17 * 64 m, so the product stays below 2^(32+y). A power of two:
// the bracket is 0.
struct Div64m {
    uint32_t x[256], y[256];
    constexpr Div64m() : x(), y() {
        for (uint32_t m = 0; m < 256; m++) {
            const uint64_t D = 64ull * (m ? m : 1);
            int l = 0;
            while ((D >> (l + 1)) != 0) l++;
            y[m] = (uint32_t)((D & (D - 1)) ? l : l - 1);
            x[m] = (uint32_t)(((1ull << (32 + y[m])) + D - 1) / D);
        }
    }
};
__device__ constexpr Div64m kDiv64m;

// Registers: where a lane's loads wait for bytes, warps in flight count (118 registers: 1,000 DAGs of
// 20-200 nodes x 1,000 allocations 408 us, 80: 326); generated candidates do not care for more.
template <int CPT, int SRC>
__global__ void __maxnreg__(CPT == 1 ? 64 : SRC == SRC_BYTES ? 80 : 104) k_bound_rows(BoundArgs a, int entries) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ uint8_t s_lev[16];
    __shared__ int64_t s_bb[16];
    __shared__ int32_t s_bc[16];
    __shared__ bool s_ok[kMaxVariantsPerCall];
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int rank = (int)cl.block_rank(), nct = (int)cl.num_blocks(), NW = nct * (int)(blockDim.x >> 5);
    const int nv = a.n_variants, n_cand = nv * a.n_alloc;
    const int tile = min(n_cand, kRowTile);
    const uint32_t M = (uint32_t)a.M;
    unsigned long long *s_acc = (unsigned long long *)sm;
    uint2 *s_div = (uint2 *)(s_acc + tile);  // SRC_BYTES: n / (64 m)
    // per warp, 32 rows: {C, m} by choice, or (SRC_BYTES) {x (64 - k), x k - 1, C, m}
    uint2 *tab = s_div + (SRC == SRC_BYTES ? 256 : 0) + (tile & 1) + w * 32 * entries;
    if (SRC != SRC_BYTES && tid < 16) s_lev[tid] = a.levels[tid];
    if (SRC == SRC_BYTES)
        for (int m = tid; m < 256; m += blockDim.x) s_div[m] = make_uint2(kDiv64m.x[m], kDiv64m.y[m]);

    for (int d = blockIdx.x / nct; d < a.n_dags; d += gridDim.x / nct) {  // the same in a cluster's CTAs
        const int64_t rbase = 2 * a.node_off[d];
        int64_t best_b = 0;
        int32_t best_c = -1;
        for (int t0 = 0; t0 < n_cand; t0 += tile) {
            const int t1 = min(n_cand, t0 + tile);
            for (int i = tid; i < tile; i += blockDim.x) s_acc[i] = 0;
            __syncthreads();
            int task = rank * (int)(blockDim.x >> 5) + w;  // tasks are numbered variant by variant; a warp takes every NW-th
            for (int vi = t0 / a.n_alloc; vi * a.n_alloc < t1; vi++) {
                // allocations of this variant in this pass
                const int a0 = max(t0 - vi * a.n_alloc, 0), a1 = min(t1 - vi * a.n_alloc, a.n_alloc);
                const int st = a.status[vi][d], nr = a.nrows[vi][d], pf = a.pflag[vi][d];  // (together: one latency)
                const int rows = st == DAGRT_OK ? nr : 0;
                if (tid == 0) s_ok[vi] = st == DAGRT_OK;
                const bool fit = rows && (pf & 1);
                const int nwin = (rows + kRowWindow - 1) / kRowWindow;
                const int nblk = (a1 - a0 + 32 * CPT - 1) / (32 * CPT);
                const uint4 *plan = a.plan[vi] + rbase;
                // FIT: 32-bit sums, else 64-bit ones (apart, so that neither holds the other's registers)
                auto run = [&](auto fitc) {
                    constexpr bool FIT = decltype(fitc)::value;
                    const int win = task / nblk, al0 = a0 + (task - win * nblk) * 32 * CPT + lane;
                    const int wend = (win + 1) * kRowWindow;  // groups that start before it
                    bool on[CPT];
#pragma unroll
                    for (int q = 0; q < CPT; q++) on[q] = al0 + 32 * q < a1;
                    using S = typename std::conditional<FIT, uint32_t, uint64_t>::type;
                    S b[CPT], gmax[CPT], gsum[CPT];
                    uint32_t gm[CPT];
#pragma unroll
                    for (int q = 0; q < CPT; q++) b[q] = gmax[q] = gsum[q] = 0, gm[q] = 0;
                    // is row `base` the start of a group?
                    bool prev = win == 0 || (plan[win * kRowWindow - 1].z >> 24) != 0, open = false;
                    for (int base = win * kRowWindow; base < rows && (open || base < wend); base += 32) {
                        const int rn = min(32, rows - base);
                        uint4 x = make_uint4(0, 0, 0, 0);
                        if (lane < rn) x = plan[base + lane];
                        const uint32_t k = (x.z >> 16) & 0xffu, m0 = x.z & 0xffffu;
                        const uint32_t endm = __ballot_sync(FULL, (x.z >> 24) != 0);
                        uint32_t startm = (endm << 1) | (prev ? 1u : 0u);
                        if (rn < 32) startm &= (1u << rn) - 1;
                        prev = (endm >> 31) != 0;
                        // rows [ra, rb): from the first start (an open group: from 0) to the end
                        // of the last group that starts before wend
                        const int inwin = wend - base;  // rows of the window from here on
                        const uint32_t mine = inwin >= 32 ? startm : (inwin > 0 ? startm & ((1u << inwin) - 1) : 0u);
                        if (!open && !mine) continue;
                        const int ra = open ? 0 : __ffs(mine) - 1;
                        int rb = rn;
                        const uint32_t later = startm & ~mine;  // groups of the next window
                        if (later && inwin < 32) rb = __ffs(later) - 1;
                        open = rb == 32 && !(endm >> 31);
                        __syncwarp();
                        if constexpr (!FIT) {
                        } else if (SRC == SRC_BYTES) {
                            ((uint4 *)tab)[lane] = make_uint4(x.x * (64u - k), x.x * k - 1u, x.y, m0);
                        } else {  // 2^l lanes for the rows, the rest of the bits for a row's choices
                            const int l = 32 - __clz(rn - 1), row = lane & ((1 << l) - 1), part = lane >> l;
                            const uint32_t tx = __shfl_sync(FULL, x.x, row), tz = __shfl_sync(FULL, x.z, row);
                            uint2 *t = tab + row * entries;
                            if (lane < rn) t[0] = make_uint2(x.y, m0);  // keep
                            for (int e = 1 + part; row < rn && e < entries; e += 32 >> l) {
                                const uint32_t m = SRC == SRC_PERTURB ? perturb_m(tz & 0xffffu, e) : s_lev[e - 1];
                                t[e] = make_uint2((uint32_t)exec_time(tx, (tz >> 16) & 0xffu, m, M), m);
                            }
                        }
                        __syncwarp();
                        if constexpr (FIT) {
                            const uint8_t *src = a.m_alloc + (rbase + base) * a.stride + vi * a.n_alloc + al0;
                            constexpr int U = SRC == SRC_BYTES ? 8 : 2;  // rows in flight together
                            for (int rr = ra; rr < rb; rr += U) {
                                uint32_t mb[U][CPT];
                                if constexpr (SRC == SRC_BYTES) {
#pragma unroll
                                    for (int i = 0; i < U; i++)
#pragma unroll
                                        for (int q = 0; q < CPT; q++)
                                            mb[i][q] = on[q] && rr + i < rb ? src[(int64_t)(rr + i) * a.stride + 32 * q] : 0u;
                                }
#pragma unroll
                                for (int i = 0; i < U; i++) {
                                    const int r = rr + i;
                                    if (r >= rb) break;
                                    uint2 cm[CPT];
                                    if constexpr (SRC == SRC_BYTES) {
                                        const uint4 y = ((const uint4 *)tab)[r];
#pragma unroll
                                        for (int q = 0; q < CPT; q++) {
                                            const uint32_t m = mb[i][q];
                                            const uint2 dv = s_div[m];
                                            cm[q].x = (__umulhi(y.x * m + y.y, dv.x) >> dv.y) + 1u;
                                            cm[q].y = m;
                                            if (m - 1u >= M) {  // the schedule's own SMs (0), or more than M
                                                const uint4 z = plan[base + r];
                                                cm[q] = m ? make_uint2((uint32_t)exec_time(z.x, (z.z >> 16) & 0xffu, m, M), m)
                                                          : make_uint2(y.z, y.w);
                                            }
                                        }
                                    } else {
#pragma unroll
                                        for (int q = 0; q < CPT; q++) {
                                            const int al = al0 + 32 * q;
                                            const int lv = gen_level(a.seed, d, vi * a.n_alloc + al, base + r, a.n_levels);
                                            const int e = al == 0 ? 0 : (SRC == SRC_PERTURB ? (int)s_lev[lv] : lv + 1);
                                            cm[q] = tab[r * entries + e];
                                        }
                                    }
                                    const bool first = (startm >> r) & 1u, last = (endm >> r) & 1u;
                                    if (first && last) {
#pragma unroll
                                        for (int q = 0; q < CPT; q++) b[q] += cm[q].x;
                                        continue;
                                    }
#pragma unroll
                                    for (int q = 0; q < CPT; q++) {
                                        gmax[q] = first ? cm[q].x : max(gmax[q], cm[q].x);
                                        gsum[q] = first ? cm[q].x : gsum[q] + cm[q].x;
                                        gm[q] = first ? cm[q].y : gm[q] + cm[q].y;
                                        if (last) b[q] += gm[q] <= M ? gmax[q] : gsum[q];
                                    }
                                }
                            }
                        } else {  // 64-bit sums: Eq.1 for every candidate
                            for (int r = ra; r < rb; r++) {
                                const uint4 y = plan[base + r];
                                const uint32_t ky = (y.z >> 16) & 0xffu, my = y.z & 0xffffu;
                                const bool first = (startm >> r) & 1u, last = (endm >> r) & 1u;
#pragma unroll
                                for (int q = 0; q < CPT; q++) {
                                    const int al = al0 + 32 * q;
                                    uint32_t m = 0;
                                    if (SRC != SRC_BYTES) m = gen_alloc(a, d, vi * a.n_alloc + al, base + r, y.w, my, s_lev);
                                    else if (on[q]) m = a.m_alloc[(rbase + base + r) * a.stride + vi * a.n_alloc + al];
                                    const uint64_t c = m ? exec_time(y.x, ky, m, M) : (uint64_t)y.y;
                                    gmax[q] = first || c > gmax[q] ? c : gmax[q];
                                    gsum[q] = first ? c : gsum[q] + c;
                                    gm[q] = (first ? 0u : gm[q]) + (m ? m : my);
                                    if (last) b[q] += gm[q] <= M ? gmax[q] : gsum[q];
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int q = 0; q < CPT; q++)
                        if (on[q] && rows)
                            atomicAdd(&s_acc[vi * a.n_alloc + al0 + 32 * q - t0], (unsigned long long)b[q]);
                };
                for (; task < nwin * nblk; task += NW) {
                    if (fit) run(std::true_type());
                    else run(std::false_type());
                }
                task -= nwin * nblk;
            }
            if (nct > 1) {  // the cluster's sums to its first CTA
                cl.sync();
                if (rank > 0) {
                    unsigned long long *acc0 = cl.map_shared_rank(s_acc, 0);
                    for (int i = tid; t0 + i < t1; i += blockDim.x) atomicAdd(&acc0[i], s_acc[i]);
                }
                cl.sync();
            } else {
                __syncthreads();
            }
            for (int i = tid; rank == 0 && t0 + i < t1; i += blockDim.x) {
                const int c = t0 + i;
                const bool ok = s_ok[nv == 1 ? 0 : c / a.n_alloc];
                const int64_t v = ok ? (int64_t)s_acc[i] : -1;
                if (a.out) a.out[(int64_t)d * n_cand + c] = v;
                if (ok) better(best_b, best_c, v, c);
            }
            __syncthreads();
        }
        if (rank == 0 && (a.best_bound || a.best_cand || a.best_m)) {
            for (int o = 16; o > 0; o >>= 1) {
                const int64_t ob = __shfl_xor_sync(FULL, best_b, o);
                const int32_t oc = __shfl_xor_sync(FULL, best_c, o);
                better(best_b, best_c, ob, oc);
            }
            if (lane == 0) {
                s_bb[w] = best_b;
                s_bc[w] = best_c;
            }
            __syncthreads();
            best_c = -1;
            for (int i = 0; i < (int)(blockDim.x >> 5); i++) better(best_b, best_c, s_bb[i], s_bc[i]);
            if (tid == 0) {
                if (a.best_bound) a.best_bound[d] = best_c < 0 ? -1 : best_b;
                if (a.best_cand) a.best_cand[d] = best_c;
            }
            if (SRC != SRC_BYTES && a.best_m && best_c >= 0) {  // the winning allocation, row by row
                const int wv = best_c / a.n_alloc;
                for (int r = tid; r < a.nrows[wv][d]; r += blockDim.x) {
                    const uint4 x = a.plan[wv][rbase + r];
                    a.best_m[rbase + r] = (uint8_t)gen_alloc(a, d, best_c, r, x.w, x.z & 0xffffu, s_lev);
                }
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ exhaustive enumeration
// Allocation a gives node u the level of digit (a / B^u) mod B, B = n_levels + 1. A cluster
// of CTAs takes a DAG and shares its allocations; candidates beyond B^V repeat earlier ones
// (the digits of the DAG's own nodes repeat) and cannot win, so they are only evaluated when
// every bound is asked for. Each thread fixes the digits of nodes 1.. and runs through node
// 0's B levels: only the groups that hold a row of node 0 (mostly one) change, the sum of
// the others is kept. {C, m} of every row and digit come from a table in shared memory.
// Ties go to the smaller allocation, as everywhere.
// Bound by instruction issue (76% of the issue slots); 2,000 DAGs of 3-6 nodes x 9^6
// allocations: 41.9 -> 0.51 ms (the duplicates are 72% of the candidates; the rest was a
// division per digit and per C). One CTA per DAG takes 0.96 ms there, two 0.67, eight 0.60.
constexpr int kExhThreads = 256;
constexpr int kExhMaxRows = 64;  // rows of a plan that the table and the row records hold

// a row in the kernel's shared memory: first table entry | shift of its node's digit in the
// packed digits << 16 (0xff: node 0) | last row of its group << 24
constexpr uint32_t kExhNode0 = 0xffu << 16, kExhLast = 1u << 24;

__global__ void __launch_bounds__(kExhThreads) k_bound_exhaustive(BoundArgs a, int bits) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    __shared__ uint32_t s_row[kExhMaxRows];  // groups without a row of node 0, then the others
    __shared__ uint2 s_tab[kExhMaxRows * 16];  // {C, m} by digit
    __shared__ int64_t s_bb[kExhThreads / 32 + 1];
    __shared__ int32_t s_bc[kExhThreads / 32 + 1];
    __shared__ uint8_t s_lev[16];
    __shared__ int s_split;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t rank = cl.block_rank(), nct = cl.num_blocks();
    const int d = blockIdx.x / nct;
    const uint32_t B = (uint32_t)a.n_levels + 1u, M = (uint32_t)a.M, msk = (1u << bits) - 1;
    const uint32_t rcpB = (uint32_t)(((1ull << 32) + B - 1) / B);  // t / B = t * rcpB >> 32 for t < 2^20
    if (tid < 16) s_lev[tid] = a.levels[tid];
    const int64_t n0 = a.node_off[d], rbase = 2 * n0;
    const int V = (int)(a.node_off[d + 1] - n0), n_cand = a.n_variants * a.n_alloc;
    uint32_t T = (uint32_t)a.n_alloc;  // allocations to evaluate
    int digits = 0;                    // nodes whose digit can be other than 0
    for (uint64_t p = 1; digits < V; digits++, p *= B)
        if (p >= T) break;
    if (!a.out) {
        uint64_t p = 1;
        for (int u = 0; u < digits; u++) p *= B;
        if (p < T) T = (uint32_t)p;
    }
    int64_t best_b = 0;
    int32_t best_c = -1;
    for (int v = 0; v < a.n_variants; v++) {
        const bool ok = a.status[v][d] == DAGRT_OK;
        const int rows = ok ? a.nrows[v][d] : 0;
        const uint4 *plan = a.plan[v] + rbase;
        const int c0 = v * a.n_alloc;
        if (!ok || (a.pflag[v][d] & 1) == 0 || rows > kExhMaxRows) {
            // failed, 64-bit sums or a long plan: candidate by candidate
            for (uint32_t al = rank * kExhThreads + tid; al < T; al += nct * kExhThreads) {
                uint64_t b = 0, mx = 0, sum = 0;
                uint32_t ms = 0;
                for (int r = 0; r < rows; r++) {
                    const uint4 x = plan[r];
                    const uint32_t m = gen_alloc(a, d, (int)al, r, x.w, x.z & 0xffffu, s_lev);
                    const uint64_t c = m ? exec_time(x.x, (x.z >> 16) & 0xffu, m, M) : (uint64_t)x.y;
                    mx = c > mx ? c : mx;
                    sum += c;
                    ms += m ? m : x.z & 0xffffu;
                    if (x.z >> 24) {
                        b += ms <= M ? mx : sum;
                        mx = sum = 0;
                        ms = 0;
                    }
                }
                if (a.out) a.out[(int64_t)d * n_cand + c0 + al] = ok ? (int64_t)b : -1;
                if (ok) better(best_b, best_c, (int64_t)b, c0 + (int)al);
            }
            continue;
        }
        __syncthreads();  // the table of the variant before is read
        if (w < 2) {      // 64 rows, one per thread: which groups hold a row of node 0
            __shared__ uint32_t s_end[2], s_zero[2];
            const int r = tid;
            const uint4 x = r < rows ? plan[r] : make_uint4(0, 0, 0, 0);
            const uint32_t eb = __ballot_sync(FULL, (x.z >> 24) != 0);
            const uint32_t zb = __ballot_sync(FULL, r < rows && x.w == 0);
            if (lane == 0) {
                s_end[w] = eb;
                s_zero[w] = zb;
            }
            asm volatile("bar.sync 1, 64;" ::: "memory");
            const uint64_t end = s_end[0] | ((uint64_t)s_end[1] << 32), zero = s_zero[0] | ((uint64_t)s_zero[1] << 32);
            // rows of r's group: after the last end before r, up to the first end at or after r
            const uint64_t below = r ? end & ((1ull << r) - 1) : 0ull;
            const int first = below ? 64 - __clzll((long long)below) : 0;
            const uint64_t from = end >> r << r;
            const int lastr = from ? __ffsll((long long)from) - 1 : 63;
            const uint64_t grp = (lastr == 63 ? ~0ull : (1ull << (lastr + 1)) - 1) & ~((1ull << first) - 1);
            const bool hot = r < rows && (zero & grp) != 0;
            const uint32_t hb = __ballot_sync(FULL, hot);
            asm volatile("bar.sync 1, 64;" ::: "memory");  // both warps have read s_zero
            if (lane == 0) s_zero[w] = hb;
            asm volatile("bar.sync 1, 64;" ::: "memory");
            const uint64_t hots = s_zero[0] | ((uint64_t)s_zero[1] << 32);
            const int cold = rows - __popcll(hots), hbef = __popcll(hots & ((1ull << r) - 1));
            if (r < rows) {
                const int at = hot ? cold + hbef : r - hbef;
                // node 0's digit is the innermost loop's: digits are packed from node 1 on
                const uint32_t sh = x.w == 0 ? 0xffu : (int)x.w < digits ? (x.w - 1) * bits : 31u;
                s_row[at] = (uint32_t)(r * 16) | (sh << 16) | (x.z >> 24 ? kExhLast : 0u);
            }
            if (r == 0) s_split = cold;
        }
        for (int i = tid; i < rows * (int)B; i += kExhThreads) {
            const int r = i / (int)B, dg = i - r * (int)B;
            const uint4 x = plan[r];
            const uint32_t m = dg ? s_lev[dg - 1] : 0u;
            s_tab[r * 16 + dg] = m ? make_uint2((uint32_t)exec_time(x.x, (x.z >> 16) & 0xffu, m, M), m)
                                   : make_uint2(x.y, x.z & 0xffffu);
        }
        __syncthreads();
        const int cold = s_split;
        const uint32_t H = (T + B - 1) / B;
        uint32_t lb = ~0u, la = 0;  // this variant's best; a later allocation wins only if smaller
        for (uint32_t h = rank * kExhThreads + tid; h < H; h += nct * kExhThreads) {
            uint32_t pk = 0;
            for (uint32_t u = 1, t = h; u < (uint32_t)digits; u++) {
                const uint32_t q = __umulhi(t, rcpB);
                pk |= (t - q * B) << ((u - 1) * bits);
                t = q;
            }
            auto entry = [&](uint32_t x) { return s_tab[(x & 0xffffu) + ((pk >> ((x >> 16) & 31u)) & msk)]; };
            uint32_t fixed = 0, mx = 0, sum = 0, ms = 0;
            for (int r = 0; r < cold; r++) {
                const uint32_t x = s_row[r];
                const uint2 e = entry(x);
                mx = max(mx, e.x);
                sum += e.x;
                ms += e.y;
                if (x & kExhLast) {
                    fixed += ms <= M ? mx : sum;
                    mx = sum = ms = 0;
                }
            }
            uint32_t tot[16];  // by node 0's digit
#pragma unroll
            for (int dg = 0; dg < 16; dg++) tot[dg] = fixed;
            for (int r = cold, z = 0; r < rows; r++) {
                const uint32_t x = s_row[r];
                if ((x & kExhNode0) == kExhNode0) {  // the group's row of node 0
                    z = (int)(x & 0xffffu);
                } else {
                    const uint2 e = entry(x);
                    mx = max(mx, e.x);
                    sum += e.x;
                    ms += e.y;
                }
                if (x & kExhLast) {
#pragma unroll
                    for (int dg = 0; dg < 16; dg++) {
                        if (dg >= (int)B) break;
                        const uint2 e = s_tab[z + dg];
                        tot[dg] += ms + e.y <= M ? max(mx, e.x) : sum + e.x;
                    }
                    mx = sum = ms = 0;
                }
            }
#pragma unroll
            for (int dg = 0; dg < 16; dg++) {
                const uint32_t al = h * B + dg;
                if (dg >= (int)B || al >= T) break;
                if (a.out) a.out[(int64_t)d * n_cand + c0 + al] = (int64_t)tot[dg];
                if (tot[dg] < lb) {
                    lb = tot[dg];
                    la = al;
                }
            }
        }
        if (lb != ~0u) better(best_b, best_c, (int64_t)lb, c0 + (int)la);
    }
    for (int o = 16; o > 0; o >>= 1) {
        const int64_t ob = __shfl_xor_sync(FULL, best_b, o);
        const int32_t oc = __shfl_xor_sync(FULL, best_c, o);
        better(best_b, best_c, ob, oc);
    }
    if (lane == 0) {
        s_bb[w] = best_b;
        s_bc[w] = best_c;
    }
    __syncthreads();
    if (tid == 0) {
        for (int i = 1; i < kExhThreads / 32; i++) better(best_b, best_c, s_bb[i], s_bc[i]);
        s_bb[kExhThreads / 32] = best_b;
        s_bc[kExhThreads / 32] = best_c;
    }
    cl.sync();
    if (rank == 0) {
        best_c = -1;
        for (uint32_t i = 0; i < nct; i++)
            better(best_b, best_c, *cl.map_shared_rank(&s_bb[kExhThreads / 32], i),
                   *cl.map_shared_rank(&s_bc[kExhThreads / 32], i));
        if (tid == 0) {
            if (a.best_bound) a.best_bound[d] = best_c < 0 ? -1 : best_b;
            if (a.best_cand) a.best_cand[d] = best_c;
        }
        if (a.best_m && best_c >= 0) {  // the winning allocation, row by row
            const int wv = best_c / a.n_alloc;
            for (int r = tid; r < a.nrows[wv][d]; r += kExhThreads) {
                const uint4 x = a.plan[wv][rbase + r];
                a.best_m[rbase + r] = (uint8_t)gen_alloc(a, d, best_c, r, x.w, x.z & 0xffffu, s_lev);
            }
        }
    }
    cl.sync();  // the CTAs' shared memory is read until here
}

// ------------------------------------------------------------------ balanced work items
constexpr int kSubRows = 32;      // plan rows staged per load phase of a work item
// rows of one TMA box of candidate bytes (64 bytes wide): a whole phase, one copy (a short
// last phase copies rows it does not use; boxes of 8 or 16 rows measured slower)
constexpr int kBoxRows = kSubRows;
constexpr int kMaxItemWarps = 8;  // warps per CTA of the work-item kernel: ChunkArgs::warps <= this
// per warp: two staging buffers (the candidate bytes of a phase, then its plan rows) and the
// {C, m} table of the phase's rows; every piece 128-byte aligned
constexpr int kStageCand = kSubRows * 64;
constexpr int kStageBytes = kStageCand + kSubRows * 16;
constexpr int kWarpBytes = 2 * kStageBytes + kSubRows * 9 * 8;
static_assert(kStageCand % 128 == 0 && kStageBytes % 128 == 0 && kWarpBytes % 128 == 0, "TMA buffer alignment");

// Chunk starts of every DAG of one plan (one warp per DAG). Chunk 0 starts at row 0; each
// chunk takes whole groups, as many as fit in chunk_rows rows (at least one group), so a
// chunk ends at the last group end within chunk_rows rows of its start, or at the end of
// its first group if that group alone is longer. Any two neighbouring chunks hold more than
// chunk_rows rows together. The group-end bits of 32 rows at a time come from one ballot;
// every lane walks the same masks, lane 0 writes.
__global__ void k_plan_chunks(int32_t n_dags, const int64_t *node_off, const uint4 *plan, const int32_t *nrows,
                              const int32_t *status, int32_t *chunk, int32_t *nchunk, int chunk_rows) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int d = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; d < n_dags; d += warps) {
        const int rows = status[d] == DAGRT_OK ? nrows[d] : 0;
        const uint4 *pr = plan + 2 * node_off[d];
        int count = 0;
        for (int cur = 0; cur < rows;) {
            if (lane == 0) chunk[2 * node_off[d] + count] = cur;
            count++;
            const int limit = min(rows, cur + chunk_rows);
            int next = -1;  // one past the chunk's last row
            for (int base = cur; base < limit; base += 32) {
                const int r = base + lane;
                const uint32_t mask = __ballot_sync(FULL, r < limit && (pr[r].z >> 24) != 0);
                if (mask) next = base + 32 - __clz(mask);
            }
            for (int base = limit; next < 0 && base < rows; base += 32) {  // a group longer than chunk_rows
                const int r = base + lane;
                const uint32_t mask = __ballot_sync(FULL, r < rows && (pr[r].z >> 24) != 0);
                if (mask) next = base + __ffs(mask);
            }
            cur = next < 0 ? rows : next;
        }
        if (lane == 0) nchunk[d] = count;
    }
}

// exclusive prefix sum of n counts (one CTA of 1024 threads); out[n] = total
__global__ void __launch_bounds__(1024) k_scan_excl(int32_t n, const int32_t *in, int32_t *out) {
    __shared__ int32_t ws[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int32_t carry = 0;
    for (int base = 0; base < n; base += 1024) {
        const int i = base + tid;
        const int32_t x = i < n ? in[i] : 0;
        int32_t incl = x;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) ws[w] = incl;
        __syncthreads();
        if (w == 0) {
            int32_t v = ws[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(FULL, v, o);
                if (lane >= o) v += y;
            }
            ws[lane] = v;
        }
        __syncthreads();
        if (i < n) out[i] = carry + (w ? ws[w - 1] : 0) + incl - x;
        const int32_t tot = ws[31];
        __syncthreads();
        carry += tot;
    }
    if (tid == 0) out[n] = carry;
}

// item records {d, first row, end row, flags} in global plan-row numbering; flags bit 0:
// the DAG's sums fit 32-bit arithmetic
__global__ void k_fill_items(int32_t n_dags, const int64_t *node_off, const int32_t *nrows, const int32_t *pflag,
                             const int32_t *chunk, const int32_t *nchunk, const int32_t *cpre, int4 *item) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int d = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; d < n_dags; d += warps) {
        const int64_t rbase = 2 * node_off[d];
        const int nch = nchunk[d];
        const int flags = nch ? (pflag[d] & 1) : 0;
        for (int k = lane; k < nch; k += 32) {
            const int r0 = chunk[rbase + k], r1 = k + 1 < nch ? chunk[rbase + k + 1] : nrows[d];
            item[cpre[d] + k] = make_int4(d, (int)(rbase + r0), (int)(rbase + r1), flags);
        }
    }
}

cudaError_t bound_build_chunks(int32_t n_dags, const int64_t *node_off, const uint4 *plan, const int32_t *nrows,
                               const int32_t *status, const int32_t *pflag, const ChunkIndex &ci, int chunk_rows,
                               int n_sm, cudaStream_t st) {
    if (n_dags == 0) return cudaMemsetAsync(ci.cpre, 0, sizeof(int32_t), st);
    int grid = (n_dags + 7) / 8;
    if (grid > 16 * n_sm) grid = 16 * n_sm;
    k_plan_chunks<<<grid, 256, 0, st>>>(n_dags, node_off, plan, nrows, status, ci.chunk, ci.nchunk, chunk_rows);
    k_scan_excl<<<1, 1024, 0, st>>>(n_dags, ci.nchunk, ci.cpre);
    k_fill_items<<<grid, 256, 0, st>>>(n_dags, node_off, nrows, pflag, ci.chunk, ci.nchunk, ci.cpre, ci.item);
    return cudaGetLastError();
}

static int64_t chunk_items_call(int32_t n_dags, int64_t total_nodes, int32_t n_variants, int32_t n_alloc,
                                int chunk_rows) {
    return (int64_t)n_variants * chunk_items_bound(total_nodes, n_dags, chunk_rows) * (n_alloc / 64);
}

bool bound_chunk_eligible(const BoundArgs &a, int64_t total_nodes, int chunk_rows) {
    return !a.gen && a.n_alloc % 64 == 0 && a.n_dags > 0 &&
           chunk_items_call(a.n_dags, total_nodes, a.n_variants, a.n_alloc, chunk_rows) < (1ll << 30) &&
           2 * total_nodes < (1ll << 31);
}

size_t bound_chunk_scratch(int32_t n_dags, int64_t total_nodes, int32_t n_variants, int32_t n_alloc, int chunk_rows) {
    (void)total_nodes;
    (void)chunk_rows;
    return 256 + (size_t)n_dags * n_variants * n_alloc * 8;
}

// After the work items (programmatic launch: they let this kernel start early, and it waits for
// them before it touches their partial sums), one warp per DAG: the items have added their partial bounds into
// the DAG's per-candidate accumulators; lane l reads candidates 2l and 2l + 1 of four
// 64-candidate blocks at a time, writes the bounds (-1 for a variant whose schedule
// failed), clears the accumulators for the next call and takes the argmin by shuffles. The
// statuses are read before the wait on the work items. Block 0 also resets the work-item
// counter.
__global__ void __launch_bounds__(32) k_bound_finish(BoundArgs a, ChunkArgs ch) {
    const int nv = a.n_variants, ncb = a.n_alloc / 64, n_cand = nv * a.n_alloc, nblk = nv * ncb;
    const int lane = threadIdx.x;
    int32_t st = 0;
    if (lane < nv && (int)blockIdx.x < a.n_dags) st = a.status[lane][blockIdx.x];
    griddep_wait();
    if (blockIdx.x == 0 && lane == 0) *ch.counter = 0u;
    for (int d = blockIdx.x; d < a.n_dags; d += gridDim.x) {
        if (d != (int)blockIdx.x && lane < nv) st = a.status[lane][d];
        unsigned long long *acc = ch.acc + (int64_t)d * n_cand;
        int64_t best_b = 0;
        int32_t best_c = -1;
        for (int k0 = 0; k0 < nblk; k0 += 4) {
            ulonglong2 x[4];
#pragma unroll
            for (int k = 0; k < 4; k++)
                x[k] = k0 + k < nblk ? __ldcg((const ulonglong2 *)(acc + (k0 + k) * 64 + 2 * lane))
                                     : make_ulonglong2(0, 0);
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (k0 + k >= nblk) break;
                const int c = (k0 + k) * 64 + 2 * lane;
                const bool ok = __shfl_sync(FULL, st, (k0 + k) / ncb) == DAGRT_OK;
                const int64_t s0 = ok ? (int64_t)x[k].x : -1, s1 = ok ? (int64_t)x[k].y : -1;
                if (ok) {
                    better(best_b, best_c, s0, c);
                    better(best_b, best_c, s1, c + 1);
                    *(ulonglong2 *)(acc + c) = make_ulonglong2(0, 0);
                }
                if (a.out) {  // the caller's buffer is only 8-byte aligned
                    a.out[(int64_t)d * n_cand + c] = s0;
                    a.out[(int64_t)d * n_cand + c + 1] = s1;
                }
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const int64_t ob = __shfl_xor_sync(FULL, best_b, o);
            const int32_t oc = __shfl_xor_sync(FULL, best_c, o);
            better(best_b, best_c, ob, oc);
        }
        if (lane == 0) {
            if (a.best_bound) a.best_bound[d] = best_c < 0 ? -1 : best_b;
            if (a.best_cand) a.best_cand[d] = best_c;
        }
    }
}

// nonzero iff some byte of w is neither 0 nor a power of two: per byte, (b | 0x80) - 1
// cannot borrow from the next byte, and its AND with b is 0 exactly for 0 and powers of two
__device__ __forceinline__ uint32_t bytes_not_pow2(uint32_t w) { return ((w | 0x80808080u) - 0x01010101u) & w; }

// index of the highest set bit, -1 for 0 (PTX bfind)
__device__ __forceinline__ int high_bit(uint32_t x) {
    int r;
    asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

// One plan row of Lemma 1's group sweep for two candidates (C, m in ta, tb): a row that
// starts and ends its group adds C; a group's first row sets max / sum / SMs, later rows
// accumulate, its last row adds R_j = max C if the SMs fit in M, else sum C. `start` and
// `end` are the same in every lane, so the branches are uniform (bra.uni).
__device__ __forceinline__ void group_step(uint32_t start, uint32_t end, uint2 ta, uint2 tb, uint32_t M,
                                           uint32_t &gmax0, uint32_t &gmax1, uint32_t &gsum0, uint32_t &gsum1,
                                           uint32_t &gm0, uint32_t &gm1, uint32_t &b0, uint32_t &b1) {
    asm("{\n\t"
        ".reg .pred ps, pe, q0, q1;\n\t"
        ".reg .u32 t0, t1;\n\t"
        "setp.ne.u32 ps, %8, 0;\n\t"
        "setp.ne.u32 pe, %9, 0;\n\t"
        "@!ps bra.uni MID;\n\t"
        "@!pe bra.uni FIRST;\n\t"
        "add.u32 %6, %6, %10;\n\t"
        "add.u32 %7, %7, %12;\n\t"
        "bra.uni DONE;\n"
        "FIRST:\n\t"
        "mov.u32 %0, %10;\n\t"
        "mov.u32 %1, %12;\n\t"
        "mov.u32 %2, %10;\n\t"
        "mov.u32 %3, %12;\n\t"
        "mov.u32 %4, %11;\n\t"
        "mov.u32 %5, %13;\n\t"
        "bra.uni DONE;\n"
        "MID:\n\t"
        "max.u32 %0, %0, %10;\n\t"
        "max.u32 %1, %1, %12;\n\t"
        "add.u32 %2, %2, %10;\n\t"
        "add.u32 %3, %3, %12;\n\t"
        "add.u32 %4, %4, %11;\n\t"
        "add.u32 %5, %5, %13;\n\t"
        "@!pe bra.uni DONE;\n\t"
        "setp.le.u32 q0, %4, %14;\n\t"
        "setp.le.u32 q1, %5, %14;\n\t"
        "selp.u32 t0, %0, %2, q0;\n\t"
        "selp.u32 t1, %1, %3, q1;\n\t"
        "add.u32 %6, %6, t0;\n\t"
        "add.u32 %7, %7, t1;\n"
        "DONE:\n\t"
        "}"
        : "+r"(gmax0), "+r"(gmax1), "+r"(gsum0), "+r"(gsum1), "+r"(gm0), "+r"(gm1), "+r"(b0), "+r"(b1)
        : "r"(start), "r"(end), "r"(ta.x), "r"(ta.y), "r"(tb.x), "r"(tb.y), "r"(M));
}

// 2-D tensor copy (TMA) of one box of candidate bytes: x = first candidate column (a
// multiple of 64), y = first allocation row; rows past the end of the tensor read as zero
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ void bulk_g2s_u32(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Persistent warps over the work items. Per item: its rows (64 candidate bytes and the plan
// row each, at most kSubRows per phase) are staged into one of the warp's two buffers by
// lane 0 -- a 2-D TMA tensor copy of the candidate bytes and a bulk copy of the plan rows,
// completing on the buffer's mbarrier -- and the next phase (of this item or the next one)
// is issued into the other buffer before the current one is evaluated.
//
// Items whose DAG's sums fit 32 bits: per phase, lane r handles plan row r -- it builds the
// row's {C, m} table (m = 0: the schedule's own C and m; m = 1, 2, 4, ..., 128: the 32-bit
// shift form, exec_time above M when CHECK_M) and checks whether all 64 candidate bytes of
// the row are 0 or powers of two; two ballots give the phase's group-end and exact-path row
// masks, and the group starts follow from the ends. Each lane then runs 2 candidates along
// the rows with table lookups; rows with other bytes take exec_time for those bytes. A
// group of one row adds its C directly; the first row of a longer group sets its running
// max / sum / SMs, its last row adds R_j (Lemma 1). Other items run their rows in 64-bit
// arithmetic with exec_time for every byte. Each item adds its 64 partial sums into the
// DAG's per-candidate 64-bit accumulators (the bound is their sum); k_bound_finish reads
// them once every item is done. At most 64 registers a thread, so that eight CTAs of four
// warps fit an SM by registers. A copy that does not land within the bounded wait sets
// DAGRT_E_TIMEOUT; the warp then waits (bounded) for its copies in flight and stops.
template <bool CHECK_M>
__global__ void __launch_bounds__(kMaxItemWarps * 32, 4)
    k_bound_items(const __grid_constant__ CUtensorMap tmap, BoundArgs a, ChunkArgs ch) {
    extern __shared__ unsigned char sm[];
    __shared__ int64_t s_cum[kMaxVariantsPerCall + 1];
    __shared__ __align__(8) uint64_t s_bar[kMaxItemWarps][2];
    __shared__ uint32_t s_drawn;  // the first item off the counter: one per warp comes before it
    griddep_launch_dependents();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // the warps' buffers from a 128-byte boundary (TMA destinations)
    unsigned char *wbase = sm + (((smem_addr(sm) + 127u) & ~127u) - smem_addr(sm)) + w * kWarpBytes;
    uint64_t *bar = s_bar[w];
    uint2 *tbuf = (uint2 *)(wbase + 2 * kStageBytes);
    const int nv = a.n_variants, ncb = a.n_alloc / 64, n_cand = nv * a.n_alloc;
    const uint32_t M = (uint32_t)a.M;
    if (threadIdx.x == 0) {
        s_cum[0] = 0;
        for (int v = 0; v < nv; v++) s_cum[v + 1] = s_cum[v] + (int64_t)ch.cpre[v][a.n_dags] * ncb;
        s_drawn = gridDim.x * (blockDim.x >> 5);
    }
    if (lane == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    const uint32_t total = (uint32_t)s_cum[nv];

    // Every warp's first item is its own (the CTAs' first warps, then their second ones); items are
    // unequal, so the others are drawn. A call of no more items than warps then has no counter to
    // wait for: 10 DAGs of 300-1,000 nodes x 256 candidates 12.3 us (18.3 with every item drawn).
    // Runs of items dealt out in advance instead: 1,000 DAGs of 50-500 nodes of which 2% need 64-bit
    // sums 137 us (now 80).
    auto grab = [&]() -> uint32_t {
        uint32_t v = s_drawn;
        if (lane == 0 && v < total) v += atomicAdd(ch.counter, 1u);
        return __shfl_sync(FULL, v, 0);
    };
    // variant slot, 64-candidate block and record of item j
    auto locate = [&](uint32_t j, int &vi, int &cb, int4 &rec) {
        vi = 0;
        while ((int64_t)j >= s_cum[vi + 1]) vi++;
        const uint32_t jj = j - (uint32_t)s_cum[vi];
        const uint32_t q = ncb == 1 ? jj : jj / (uint32_t)ncb;
        cb = (int)(jj - q * (uint32_t)ncb);
        rec = ch.item[vi][q];
    };
    uint32_t parity = 0u;    // bit b: parity of the next wait on buffer b
    uint32_t inflight = 0u;  // bit b: a copy issued into buffer b and not yet waited for
    // rows [g0, g1) of item (vi, cb) into staging buffer b (the warp is done reading it): one
    // 2-D TMA box per kBoxRows rows of the 64 candidate bytes, one bulk copy of the plan rows
    auto stage = [&](int b, int vi, int cb, int g0, int g1) {
        inflight |= 1u << b;
        if (lane == 0) {
            const int rn = g1 - g0, nb = (rn + kBoxRows - 1) / kBoxRows;
            const uint32_t dst = smem_addr(wbase + b * kStageBytes);
            fence_proxy_async();  // the warp's reads of the buffer come before the copy's writes
            mbar_expect_tx(&bar[b], (uint32_t)(nb * kBoxRows * 64 + rn * 16));
            const int x = vi * a.n_alloc + cb * 64;
            for (int i = 0; i < nb; i++) tma_load_2d(dst + i * kBoxRows * 64, &tmap, x, g0 + i * kBoxRows, &bar[b]);
            bulk_g2s_u32(dst + kSubRows * 64, a.plan[vi] + g0, (uint32_t)(rn * 16), &bar[b]);
        }
    };
    auto wait_buf = [&](int b) -> bool {
        const bool ok = __all_sync(FULL, mbar_wait(&bar[b], (parity >> b) & 1u));
        if (ok) {
            parity ^= 1u << b;
            inflight &= ~(1u << b);
        }
        return ok;
    };

    uint32_t j = __shfl_sync(FULL, w * gridDim.x + blockIdx.x, 0);  // (the warp's, not a lane's)
    int vi = 0, cb = 0, buf = 0;
    int4 rec = make_int4(0, 0, 0, 0);
    if (j < total) {
        locate(j, vi, cb, rec);
        stage(0, vi, cb, rec.y, min(rec.z, rec.y + kSubRows));
    }
    bool failed = false;
    while (j < total && !failed) {
        const uint32_t jn = grab();
        int vn = 0, cbn = 0;
        int4 recn = make_int4(0, 0, 0, 0);
        if (jn < total) locate(jn, vn, cbn, recn);
        // the item's phases; FIT: 32-bit table path, else 64-bit sums with exec_time
        auto run_item = [&](auto fitc) {
            constexpr bool FIT = decltype(fitc)::value;
            using acc_t = typename std::conditional<FIT, uint32_t, uint64_t>::type;
            acc_t gmax0 = 0, gmax1 = 0, gsum0 = 0, gsum1 = 0, b0 = 0, b1 = 0;
            uint32_t gm0 = 0, gm1 = 0;
            uint32_t carry = 1u;  // chunks start at a group start
            for (int g0 = rec.y; g0 < rec.z; g0 += kSubRows) {
                const int rn = min(kSubRows, rec.z - g0);
                if (!wait_buf(buf)) {
                    failed = true;
                    return;
                }
                // the next phase into the other buffer, read completely by the last phase: the
                // item's next rows, or the first rows of the next item
                if (g0 + kSubRows < rec.z)
                    stage(buf ^ 1, vi, cb, g0 + kSubRows, min(rec.z, g0 + 2 * kSubRows));
                else if (jn < total)
                    stage(buf ^ 1, vn, cbn, recn.y, min(recn.z, recn.y + kSubRows));
                const unsigned char *cbuf = wbase + buf * kStageBytes;
                const uint4 *pbuf = (const uint4 *)(cbuf + kSubRows * 64);
                if constexpr (FIT) {
                    bool endg = false, odd = false;
                    if (lane < rn) {  // {C, m} table, group end and byte check of row `lane`
                        const uint4 x = pbuf[lane];
                        const uint32_t kk = (x.z >> 16) & 0xffu;
                        const uint32_t A1 = x.x * (64u - kk) + 64u, B1 = x.x * kk - 1u;
                        uint2 *t = tbuf + lane * 9;
                        t[0] = make_uint2(x.y, x.z & 0xffffu);
#pragma unroll
                        for (int l = 0; l < 8; l++) {
                            uint32_t v = ((A1 << l) + B1) >> (l + 6);
                            if (CHECK_M && (1u << l) > M) v = (uint32_t)exec_time(x.x, kk, 1u << l, M);
                            t[l + 1] = make_uint2(v, 1u << l);
                        }
                        endg = (x.z >> 24) != 0;
                        const uint4 *cw = (const uint4 *)(cbuf + lane * 64);
                        uint32_t acc = 0;
#pragma unroll
                        for (int q = 0; q < 4; q++) {  // rotated: 8 lanes hit 8 distinct 16-byte bank groups
                            const uint4 v = cw[(q + (lane >> 1)) & 3];
                            acc |= bytes_not_pow2(v.x) | bytes_not_pow2(v.y) | bytes_not_pow2(v.z) |
                                   bytes_not_pow2(v.w);
                        }
                        odd = acc != 0;
                    }
                    const uint32_t endm = __ballot_sync(FULL, endg);
                    const uint32_t oddm = __ballot_sync(FULL, odd);
                    const uint32_t startm = (endm << 1) | carry;
                    carry = (endm >> (rn - 1)) & 1u;
                    __syncwarp();
                    auto rows = [&](auto exact) {
#pragma unroll 4
                        for (int r = 0; r < rn; r++) {
                            const uint32_t w2 = *(const uint16_t *)(cbuf + r * 64 + 2 * lane);
                            const uint32_t ma = w2 & 0xffu, mb = w2 >> 8;
                            const uint2 *tr = tbuf + r * 9 + 1;
                            uint2 ta = tr[high_bit(ma)], tb = tr[high_bit(mb)];
                            const uint32_t bit = 1u << r;
                            if (decltype(exact)::value && (oddm & bit)) {
                                const uint4 x = pbuf[r];
                                const uint32_t kk = (x.z >> 16) & 0xffu;
                                if (ma & (ma - 1)) ta = make_uint2((uint32_t)exec_time(x.x, kk, ma, M), ma);
                                if (mb & (mb - 1)) tb = make_uint2((uint32_t)exec_time(x.x, kk, mb, M), mb);
                            }
                            group_step(startm & bit, endm & bit, ta, tb, M, gmax0, gmax1, gsum0, gsum1, gm0, gm1,
                                       b0, b1);
                        }
                    };
                    if (oddm)
                        rows(std::true_type());
                    else
                        rows(std::false_type());
                } else {  // 64-bit sums: exec_time for every byte
                    for (int r = 0; r < rn; r++) {
                        const uint4 x = pbuf[r];
                        const uint32_t kk = (x.z >> 16) & 0xffu, m0 = x.z & 0xffffu;
                        const uint32_t w2 = *(const uint16_t *)(cbuf + r * 64 + 2 * lane);
                        const uint32_t ma = w2 & 0xffu, mb = w2 >> 8;
                        const uint64_t ca = ma ? exec_time(x.x, kk, ma, M) : (uint64_t)x.y;
                        const uint64_t cv = mb ? exec_time(x.x, kk, mb, M) : (uint64_t)x.y;
                        gmax0 = ca > gmax0 ? ca : gmax0;
                        gmax1 = cv > gmax1 ? cv : gmax1;
                        gsum0 += ca;
                        gsum1 += cv;
                        gm0 += ma ? ma : m0;
                        gm1 += mb ? mb : m0;
                        if (x.z >> 24) {
                            b0 += gm0 <= M ? gmax0 : gsum0;
                            b1 += gm1 <= M ? gmax1 : gsum1;
                            gmax0 = gmax1 = gsum0 = gsum1 = 0;
                            gm0 = gm1 = 0;
                        }
                    }
                }
                __syncwarp();  // the buffer and the table are read
                buf ^= 1;
            }
            // add the item's partial bounds into its DAG's accumulators (reductions: no wait)
            unsigned long long *acc = ch.acc + (int64_t)rec.x * n_cand + vi * a.n_alloc + cb * 64 + 2 * lane;
            atomicAdd(acc, (unsigned long long)b0);
            atomicAdd(acc + 1, (unsigned long long)b1);
        };
        if (rec.w & 1)
            run_item(std::true_type());
        else
            run_item(std::false_type());
        j = jn;
        vi = vn;
        cb = cbn;
        rec = recn;
    }
    if (failed) {
        // a copy stalled: report it, and give the copies in flight a bounded chance to land
        // before the CTA's shared memory is released
        if (lane == 0) {
            if (a.err) atomicExch(a.err, DAGRT_E_TIMEOUT);
            for (int b = 0; b < 2; b++)
                if ((inflight >> b) & 1u) mbar_wait(&bar[b], (parity >> b) & 1u);
        }
        __syncwarp();
    }
}

// The candidate bytes as a 2-D tensor of bytes for TMA: `rows` allocation rows of `stride`
// bytes (a multiple of 16, the base 16-byte aligned: both checked by the API), boxes of 64
// bytes x kBoxRows rows, no swizzle, zero fill past the last row. cuTensorMapEncodeTiled
// (host-side encoding only) is taken from the driver through the runtime's entry-point query,
// so the library links no driver stub.
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeTiledFn) nullptr;
        return (EncodeTiledFn)p;
    }();
    return fn;
}

static cudaError_t encode_alloc_map(const BoundArgs &a, int64_t rows, CUtensorMap *map) {
    std::memset(map, 0, sizeof *map);
    if (rows <= 0) return cudaSuccess;  // no candidate rows: no work item copies any
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dim[2] = {(cuuint64_t)a.stride, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)a.stride};
    const cuuint32_t box[2] = {64u, (cuuint32_t)kBoxRows};
    const cuuint32_t estr[2] = {1u, 1u};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, (void *)a.m_alloc, dim, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t bound_launch(const BoundArgs &a, const ChunkArgs *ch, int n_sm, cudaStream_t st, int *launches) {
    *launches = 0;
    if (a.n_dags == 0) return cudaSuccess;
    const int n_cand = a.n_variants * a.n_alloc;
    const bool items = ch != nullptr;
    if (items) {
        // the item counter is zero here: set when the scratch was allocated, and reset by
        // k_bound_finish at the end of every call
        cudaError_t e;
        CUtensorMap tmap;
        if ((e = encode_alloc_map(a, ch->alloc_rows, &tmap)) != cudaSuccess) return e;
        const int warps = ch->warps < 1 ? 1 : (ch->warps > kMaxItemWarps ? kMaxItemWarps : ch->warps);
        const int smem = warps * kWarpBytes + 128;  // + alignment of the warps' buffers to 128 bytes
        auto kern = a.M < 128 ? k_bound_items<true> : k_bound_items<false>;
        int per_sm = 0;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxItemWarps * kWarpBytes + 128);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, warps * 32, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        kern<<<per_sm * n_sm, warps * 32, smem, st>>>(tmap, a, *ch);
        const int g = a.n_dags < 32 * n_sm ? a.n_dags : 32 * n_sm;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(g);
        cfg.blockDim = dim3(32);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if ((e = cudaLaunchKernelEx(&cfg, k_bound_finish, a, *ch)) != cudaSuccess) return e;
        *launches += 2;
        return cudaSuccess;  // (the items evaluate the DAGs that need 64-bit sums too)
    }
    using K = void (*)(BoundArgs, int);
    if (a.gen && a.gen_mode == DAGRT_SEARCH_EXHAUSTIVE) {
        // CTAs per DAG: enough of them for every SM, while each thread keeps a run of node 0's levels
        const int B = a.n_levels + 1;
        int bits = 1;
        while ((1 << bits) < B) bits++;
        int cl = 1;
        while (cl < 8 && (int64_t)a.n_dags * cl < 32ll * n_sm && a.n_alloc / B >= 2 * cl * kExhThreads) cl *= 2;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)a.n_dags * cl);
        cfg.blockDim = dim3(kExhThreads);
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cl;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        ++*launches;
        return cudaLaunchKernelEx(&cfg, k_bound_exhaustive, a, bits);
    }
    // warps per CTA, and CTAs per DAG when even 16 leave SMs without work: enough warps for
    // every SM (500 DAGs: 16 warps 279 us, 8 315, 4 396; 1,000 small ones: 4 or 8 57-62 us, 16
    // 76; clusters only cost where the DAGs fill the chip)
    int warps = 4, cl = 1;
    while (warps < 16 && (int64_t)a.n_dags * warps < 32ll * n_sm) warps *= 2;
    while (cl < 8 && (int64_t)a.n_dags * cl * warps < 16ll * n_sm) cl *= 2;
    const bool two = a.n_alloc > 32;
    const int src = !a.gen ? SRC_BYTES : a.gen_mode == DAGRT_SEARCH_PERTURB ? SRC_PERTURB : SRC_RANDOM;
    const K kern = src == SRC_BYTES    ? (two ? (K)k_bound_rows<2, SRC_BYTES> : (K)k_bound_rows<1, SRC_BYTES>)
                   : src == SRC_RANDOM ? (two ? (K)k_bound_rows<2, SRC_RANDOM> : (K)k_bound_rows<1, SRC_RANDOM>)
                                       : (two ? (K)k_bound_rows<2, SRC_PERTURB> : (K)k_bound_rows<1, SRC_PERTURB>);
    const int entries = src == SRC_BYTES ? 2 : src == SRC_PERTURB ? kPerturbCodes : a.n_levels + 1;
    const int tile = n_cand < kRowTile ? n_cand : kRowTile;
    const int smem = 8 * (tile + (tile & 1) + (src == SRC_BYTES ? 256 : 0) + warps * 32 * entries);
    const int mx = max_dynamic_smem(kern);
    if (smem > mx) return cudaErrorInvalidValue;
    int per_sm = 0;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, warps * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cl * (a.n_dags < 8 * per_sm * n_sm ? a.n_dags : 8 * per_sm * n_sm)));
    cfg.blockDim = dim3(warps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ++*launches;
    return cudaLaunchKernelEx(&cfg, kern, a, entries);
}

}  // namespace dagrt
