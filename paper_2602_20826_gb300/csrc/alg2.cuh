// alg2.cuh -- Alg.2 (scheduling with parallel launches and node segmentation, Lemma 1,
// Theorem 1) on one DAG by one warp, and what the scheduling kernels share: per-DAG context,
// failure and result outputs, the baselines' arithmetic.
#pragma once

#include <type_traits>

#include "dagrt_internal.cuh"
#include "sched.cuh"

namespace dagrt {

// ------------------------------------------------------------------ per-DAG context
struct Dag {
    int64_t n0, rbase, ebase, ecap;
    int V, W, variant;
    uint32_t M;
    bool want_edges;
};

// Alg.2's totals, valid in the team's first warp
struct Acc {
    uint64_t bound;
    int64_t nextra;
    int nrows, nseg, nrel;  // plan rows, segments; in: nodes released at the start
    bool err;
};

__device__ inline void write_failure(const SchedArgs &a, int d, int code) {
    a.status[d] = code;
    a.bound[d] = -1;
    if (a.nrows) a.nrows[d] = 0;
    if (a.o.status) a.o.status[d] = code;
    if (a.o.bound) a.o.bound[d] = -1;
    if (a.o.n_groups) a.o.n_groups[d] = 0;
    if (a.o.n_seg) a.o.n_seg[d] = 0;
    if (a.o.n_rows) a.o.n_rows[d] = 0;
    if (a.o.n_extra) a.o.n_extra[d] = 0;
    if (a.o.greedy) a.o.greedy[d] = -1;
    if (a.o.greedy_unaware) a.o.greedy_unaware[d] = -1;
    if (a.o.graham_para) a.o.graham_para[d] = -1;
    if (a.o.crit_path) a.o.crit_path[d] = -1;
}

// What a scheduled DAG writes besides Alg.2's own outputs. One thread.
struct Totals {
    uint64_t mx;  // largest load
    uint64_t greedy, unaware, vol;  // baseline sums (Evaluation section)
    int G, nlev;
};
__device__ inline void write_totals(const SchedArgs &a, const Dag &g, int d, const Acc &acc, const Totals &t) {
    const uint32_t M = g.M;
    // candidate bounds fit 32-bit arithmetic: loads < 2^17 and every group sum of
    // C <= ceil(255/M) * max C^ over at most 2V rows below 2^31
    const uint64_t waves = (255 + M - 1) / M;
    if (a.pflag) a.pflag[d] = (t.mx < (1ull << 17) && t.mx * waves * 2ull * (uint64_t)g.V < (1ull << 31)) ? 1 : 0;
    int code = DAGRT_OK;
    if (acc.err) code = DAGRT_E_INTERNAL;
    else if (g.want_edges && acc.nextra > g.ecap) code = DAGRT_E_CAP;
    const int64_t bnd = code == DAGRT_E_INTERNAL ? -1 : (int64_t)acc.bound;
    a.status[d] = code;
    a.bound[d] = bnd;
    if (a.nrows) a.nrows[d] = acc.nrows;
    if (a.o.status) a.o.status[d] = code;
    if (a.o.bound) a.o.bound[d] = bnd;
    if (a.o.n_groups) a.o.n_groups[d] = t.G;
    if (a.o.n_seg) a.o.n_seg[d] = acc.nseg;
    if (a.o.n_rows) a.o.n_rows[d] = acc.nrows;
    if (a.o.n_extra) a.o.n_extra[d] = acc.nextra;
    // baselines: Greedy (sequential, m = min(C^, M)), Greedy + unaware (sequential, m = C^),
    // Graham_para (unit-load nodes: L + ceil((vol - L) / M), L = nodes on the longest path)
    if (a.o.greedy) a.o.greedy[d] = (int64_t)t.greedy;
    if (a.o.greedy_unaware) a.o.greedy_unaware[d] = (int64_t)t.unaware;
    if (a.o.graham_para) a.o.graham_para[d] = (int64_t)(t.nlev + (t.vol - t.nlev + M - 1) / M);
}

// The critical-path lower bound `cp` of the schedule, and the check of Theorem 1's bound
// against it. One thread.
__device__ inline void write_crit_path(const SchedArgs &a, const Dag &g, int d, const Acc &acc, uint64_t cp) {
    a.o.crit_path[d] = a.plan ? (int64_t)cp : -1;
    // Theorem 1's bound below a lower bound of every execution: an internal error
    if (a.plan && g.variant != DAGRT_VAR_LITERAL && acc.bound < cp && a.status[d] == DAGRT_OK) {
        write_failure(a, d, DAGRT_E_INTERNAL);
        a.o.crit_path[d] = (int64_t)cp;
    }
}

__device__ inline void write_empty(const SchedArgs &a, int d) {  // a DAG without nodes
    a.status[d] = DAGRT_OK;
    a.bound[d] = 0;
    if (a.nrows) a.nrows[d] = 0;
    if (a.o.status) a.o.status[d] = DAGRT_OK;
    if (a.o.bound) a.o.bound[d] = 0;
    if (a.o.n_groups) a.o.n_groups[d] = 0;
    if (a.o.n_seg) a.o.n_seg[d] = 0;
    if (a.o.n_rows) a.o.n_rows[d] = 0;
    if (a.o.n_extra) a.o.n_extra[d] = 0;
    if (a.o.greedy) a.o.greedy[d] = 0;
    if (a.o.greedy_unaware) a.o.greedy_unaware[d] = 0;
    if (a.o.graham_para) a.o.graham_para[d] = 0;
    if (a.o.crit_path) a.o.crit_path[d] = 0;
}

// Greedy + unaware kernel time (baseline of the Evaluation section): the kernel runs on
// m = x SMs whatever M is, so Eq.1's wave factor ceil(x / M) applies. Exact in 128-bit
// arithmetic, saturated at 2^63 - 1.
__device__ __forceinline__ uint64_t exec_time_unaware(uint64_t x, uint32_t k, uint32_t M) {
    const unsigned __int128 waves = (x + M - 1) / M;
    const unsigned __int128 num = waves * x * (64ull * x - (uint64_t)k * (x - 1));
    const unsigned __int128 den = 64ull * x;
    const unsigned __int128 c = (num + den - 1) / den;
    return c > (unsigned __int128)INT64_MAX ? (uint64_t)INT64_MAX : (c < 1 ? 1ull : (uint64_t)c);
}
__device__ __forceinline__ uint64_t sat_add(uint64_t a, uint64_t b) {
    const uint64_t s = a + b;
    return s > (uint64_t)INT64_MAX || s < a ? (uint64_t)INT64_MAX : s;
}

// ------------------------------------------------------------------ Alg.2
// Alg.2's working set in rank space: node r is the r-th in descending W^anc order (ties:
// lower id), so the released set is a bit mask over r whose lowest bits come first, and an
// edge leads from a rank to a smaller one.
//
// ID: the type of a rank and of a count of predecessors (8 bits for up to 256 nodes). The
// arrays are 32-bit offsets, from the kernel's dynamic shared memory (SH) or from a
// global workspace: the compiler then knows the memory space of every access in the chain,
// and the whole set costs ten registers.
template <bool SH, class ID>
struct A2 {
    unsigned char *base;  // !SH: the global workspace
    uint32_t o_rc, o_col, o_cnt, o_gstart, o_gmem, o_byrank, o_lst, o_mm;
    uint32_t o_rel, o_sum;  // always in shared memory

    template <class T>
    __device__ __forceinline__ T *at(uint32_t off) const {
        extern __shared__ __align__(16) unsigned char smem[];
        if constexpr (SH) return (T *)(smem + off);
        else return (T *)(base + off);
    }
    // {load left (0: finished), C at min(load left, M) SMs (0: recompute), first edge,
    //  out-degree | k << 16}
    __device__ __forceinline__ uint4 &rc(uint32_t r) const { return at<uint4>(o_rc)[r]; }
    __device__ __forceinline__ uint32_t &left(uint32_t r) const { return at<uint32_t>(o_rc)[4 * r]; }
    __device__ __forceinline__ ID &col(uint32_t e) const { return at<ID>(o_col)[e]; }  // successors by edge, as ranks
    __device__ __forceinline__ ID &cnt(uint32_t r) const { return at<ID>(o_cnt)[r]; }  // predecessors not yet finished
    __device__ __forceinline__ uint16_t &gstart(int j) const { return at<uint16_t>(o_gstart)[j]; }
    __device__ __forceinline__ ID &gmem(int i) const { return at<ID>(o_gmem)[i]; }  // members of each group, as ranks, in id order
    __device__ __forceinline__ ID &byrank(uint32_t r) const { return at<ID>(o_byrank)[r]; }
    __device__ __forceinline__ ID &lst(int i) const { return at<ID>(o_lst)[i]; }  // launched nodes of the group
    __device__ __forceinline__ uint16_t &mm(int i) const { return at<uint16_t>(o_mm)[i]; }    // SMs of a large group's members
    // released and unfinished nodes, 32 ranks a word; SUM: bit w of sum set: 64-bit word w of
    // rel may be non-zero (cleared lazily by the scan)
    __device__ __forceinline__ uint32_t *rel() const {
        extern __shared__ __align__(16) unsigned char smem[];
        return (uint32_t *)(smem + o_rel);
    }
    __device__ __forceinline__ uint32_t *sum() const {
        extern __shared__ __align__(16) unsigned char smem[];
        return (uint32_t *)(smem + o_sum);
    }
};

// Arithmetic of one DAG: NARROW if 64 M max C^ fits 32 bits, so that every product and sum
// over a group below does (loads below 453,000 ticks at M = 148): 64-bit products and the
// branch on the size of a division are a third of the group step's instructions otherwise.
template <bool NARROW>
struct Arith {
    using T = typename std::conditional<NARROW, uint32_t, uint64_t>::type;
    static __device__ __forceinline__ T div(T n, T d) {
        if constexpr (NARROW) return n / d;
        else return udiv(n, d);
    }
    static __device__ __forceinline__ T sum(uint32_t x) {  // over the warp
        if constexpr (NARROW) return __reduce_add_sync(FULL, x);
        else return ((uint64_t)__reduce_add_sync(FULL, x >> 16) << 16) + __reduce_add_sync(FULL, x & 0xffffu);
    }
    // Eq.5 before the repair: round(x M / Wg) half up, at least 1, at most x
    static __device__ __forceinline__ uint32_t eq5(uint32_t x, uint32_t M, T Wg) {
        const T r = div((T)2 * x * M + Wg, (T)2 * Wg);
        return r < 1 ? 1u : (r < x ? (uint32_t)r : x);
    }
    // Eq.1 on m <= M SMs
    static __device__ __forceinline__ uint32_t time(uint32_t x, uint32_t k, uint32_t m) {
        const T num = (T)x * (64u * m - k * (m - 1));
        return (uint32_t)div((num - 1) >> 6, m) + 1u;
    }
    // does load x finish within R on S <= M SMs?
    static __device__ __forceinline__ bool fits(uint32_t x, uint32_t k, uint32_t S, T R) {
        return (T)x * (64u * S - k * (S - 1)) <= (T)(64u * S) * R;
    }
    // the largest load p in [1, x - 1] that finishes within R on min(p, S) SMs, for an x that
    // does not: on S SMs if that leaves at least S ticks, else on p SMs (k < 64 then)
    static __device__ __forceinline__ uint32_t split(uint32_t x, uint32_t k, uint32_t S, T R) {
        T p = div((T)(64u * S) * R, 64u * S - k * (S - 1));
        if (p < S) p = min(div((T)64 * R - k, 64u - k), (T)(S - 1));
        return (uint32_t)min(p, (T)(x - 1));
    }
};

template <bool SH, class ID>
__device__ __forceinline__ void clear_released(const A2<SH, ID> &w, uint32_t r) {
    atomicAnd(w.rel() + (r >> 5), ~(1u << (r & 31)));
}

// The 32 lanes decrement the open-predecessor counts of a finished node's successors (its
// edges [eb, eb + deg), targets distinct; `s` holds the first 32 edges' targets) and mark
// the ones that reach zero as released; with COUNT, returns how many did.
template <bool SUM, bool COUNT, bool SH, class ID>
__device__ __forceinline__ int release_succ(const A2<SH, ID> &w, uint32_t eb, uint32_t deg, uint32_t s, int lane) {
    int n = 0;
    for (uint32_t b = 0; b < deg; b += 32) {
        const bool act = b + lane < deg;
        if (b > 0 && act) s = w.col(eb + b + lane);
        uint32_t c = 1;
        if (act) {
            c = w.cnt(s) - 1u;
            w.cnt(s) = (ID)c;
        }
        if (c == 0) {
            atomicOr(w.rel() + (s >> 5), 1u << (s & 31));
            if constexpr (SUM) atomicOr(w.sum() + (s >> 11), 1u << ((s >> 6) & 31));
        }
        if constexpr (COUNT) n += __popc(__ballot_sync(FULL, c == 0));
    }
    __syncwarp();  // counts and released bits before the next release or scan
    return n;
}

// Extra dependencies of group j (Alg.2's segmentation step): (v_n, succ(v_R)) for every
// launched part in launch order (the ranks in w.lst, then segment `seg` if one was cut) and
// (v_R, v_n) for every parallel node left in the released set, the split node's residual
// included. Before any node of the group is released from. One lane.
template <bool SH, class ID>
__device__ __noinline__ void write_extra_edges(const A2<SH, ID> w, int32_t *src, int32_t *dst, int64_t cap,
                                               int V, uint32_t vR, int nwhole, int seg, int64_t idx) {
    const uint4 q = w.rc(vR);
    const uint32_t deg = q.w & 0xffffu;
    const int id = w.byrank(vR);
    for (int i = 0; i < nwhole + (seg >= 0); i++)
        for (uint32_t e = q.z; e < q.z + deg; e++, idx++)
            if (idx < cap) {
                src[idx] = i < nwhole ? (int)w.byrank(w.lst(i)) : V + seg;
                dst[idx] = w.byrank(w.col(e));
            }
    for (int i = 0; i < (V + 31) / 32; i++)
        for (uint32_t bits = w.rel()[i]; bits; bits &= bits - 1, idx++)
            if (idx < cap) {
                src[idx] = id;
                dst[idx] = w.byrank(i * 32 + __ffs(bits) - 1);
            }
}

// Members of a group of more than 32: Eq.5 with the repair, Eq.1 and Lemma 1, 32 members at
// a time. The SMs go to w.mm, C to the members' records; members leave the released set.
// Returns the unfinished members; with one only, *vR is that member and nothing else is set.
template <bool SH, class ID>
__device__ __noinline__ int members_large(const A2<SH, ID> w, int variant, uint32_t M, int gb, int n, int lane, uint64_t *R,
                                          uint32_t *vR, uint32_t *sum_m) {
    using Ar = Arith<false>;
    int np = 0;
    uint64_t Wg = 0;
    uint32_t one = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const uint32_t r = i0 + lane < n ? w.gmem(gb + i0 + lane) : 0;
        const uint32_t x = i0 + lane < n ? w.rc(r).x : 0;
        const uint32_t live = __ballot_sync(FULL, x > 0);
        if (live) one = __shfl_sync(FULL, r, __ffs(live) - 1);
        np += __popc(live);
        Wg += Ar::sum(x);
    }
    *vR = one;
    if (np < 2) return np;
    uint32_t sum = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t r = i < n ? w.gmem(gb + i) : 0;
        const uint32_t x = i < n ? w.rc(r).x : 0;
        const uint32_t m = x ? Ar::eq5(x, M, Wg) : 0;
        if (i < n) w.mm(i) = (uint16_t)m;
        if (x) clear_released(w, r);
        sum += __reduce_add_sync(FULL, m);
    }
    __syncwarp();
    if (variant != DAGRT_VAR_NOREPAIR && sum > M) {
        // taking one SM at a time from the largest m (ties: higher id) t times leaves every
        // m at most L + 1, L the largest level with sum max(0, m - L) >= t, and then takes
        // the rest from the members still at L + 1, highest id first
        const uint32_t t = sum - M;
        uint32_t lo = 0, hi = M;  // above(lo) >= t > above(hi)
        auto above = [&](uint32_t L) {
            uint32_t s = 0;
            for (int i0 = 0; i0 < n; i0 += 32) {
                const uint32_t m = i0 + lane < n ? w.mm(i0 + lane) : 0;
                s += __reduce_add_sync(FULL, m > L ? m - L : 0);
            }
            return s;
        };
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (above(mid) >= t) lo = mid;
            else hi = mid;
        }
        uint32_t left = t - above(lo + 1);
        __syncwarp();
        for (int i0 = (n - 1) & ~31; i0 >= 0; i0 -= 32) {
            const uint32_t m = i0 + lane < n ? w.mm(i0 + lane) : 0;
            const uint32_t top = __ballot_sync(FULL, m > lo);
            const uint32_t before = lane < 31 ? __popc(top >> (lane + 1)) : 0;
            if (m > lo) w.mm(i0 + lane) = (uint16_t)(before < left ? lo : lo + 1);
            left -= min(left, (uint32_t)__popc(top));
        }
        __syncwarp();
        sum = M;
    }
    uint64_t csum = 0;
    uint32_t Rm = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t r = i < n ? w.gmem(gb + i) : 0;
        const uint4 q = i < n ? w.rc(r) : make_uint4(0, 0, 0, 0);
        uint32_t c = 0;
        if (q.x) {
            c = Ar::time(q.x, q.w >> 16, w.mm(i));
            w.rc(r).y = c;
        }
        csum += Ar::sum(c);
        const uint32_t cm = __reduce_max_sync(FULL, c);
        const uint32_t at = __ballot_sync(FULL, c == cm);
        if (cm > Rm) {
            Rm = cm;
            *vR = __shfl_sync(FULL, r, __ffs(at) - 1);
        }
    }
    __syncwarp();
    *sum_m = sum;
    *R = sum > M ? csum : (uint64_t)Rm;  // over-full (no repair): members one after another
    return np;
}

constexpr uint32_t kOwnSucc = 8;  // successors that a lane releases by itself (groups of more than 32)

// Alg.2 over all groups of a DAG with Lemma 1 and Theorem 1, by one warp. The group step is
// a serial chain, so it is written for latency: every lane runs the scalar part on the same
// values (no divergence, no hand-over between lanes), a node's record is one 16-byte load,
// the time of a whole launch comes precomputed (on x <= S SMs it is C at min(x, M) SMs), a
// segment's time is R itself (below), and the successors of a finished node are counted
// down by the 32 lanes with plain loads and stores while the first candidate's record is on
// its way. Ranks instead of ids take the lookups out of the chain: the released set is one
// 32-bit word per lane (up to 1,024 nodes) or a mask with a summary word per lane (SUM).
//
// Where all lanes store alike, each has read what it needs from there first: a warp barrier (the
// one that ends release_succ, or one of its own) stands between the records' loads and the stores
// that change them, and between a plan row and the store that marks it the last of its group.
//
// A segment p is the largest load that finishes within R on min(p, S) SMs, and adding one
// tick of load adds at most one tick of time: the part takes exactly R.
//
// What bounds it: the latency of one warp's dependent instructions (a third of the stalls are
// shared-memory loads, the rest fixed-latency arithmetic). One lane walking id-indexed arrays took
// 3,800 cycles a group, this 1,500 in shared memory and 2,600 in a global workspace; by itself
// that took a call of 10,000 DAGs of 20-200 nodes from 1.80 to 1.42 ms (now 0.67, by what
// sched_warp.cuh changed).
//
// FULL_OUT: another variant than the paper's, no plan, or some of the outputs that few callers
// ask for (rows, segments, group times, extra dependencies); without it the chain does not
// carry what only they need.
template <bool SUM, bool NARROW, bool FULL_OUT, bool SH, class ID>
__device__ __forceinline__ void alg2_warp(const A2<SH, ID> &w, const SchedArgs &a, const Dag &g, int G, Acc &acc, int lane) {
    using Ar = Arith<NARROW>;
    using T = typename Ar::T;
    const uint32_t M = g.M;
    const int variant = FULL_OUT ? g.variant : (int)DAGRT_VAR_PAPER;
    const bool node_out = a.o.m || a.o.exec_group;
    const bool defer = FULL_OUT && g.want_edges;  // nothing is released before the extra edges are written
    uint4 *plan = !FULL_OUT || a.plan ? a.plan + g.rbase : nullptr;
    uint64_t bound = 0;
    int64_t nextra = 0;
    int nrows = 0, nseg = 0, nrel = acc.nrel;
    // The scalar part is stored by all lanes alike (one transaction, and no divergent branch);
    // the optional outputs of one row, segment or node by a lane per field: lanes 0 .. 4 hold
    // {id, group, SMs, load's two halves} and where they go, so five stores are one.
    struct Field {
        int32_t *p;  // NULL: not wanted, or no field of this lane
        int step;
    };
    auto field = [&](int32_t *id, int32_t *group, int32_t *m, int64_t *load) {
        Field f;
        f.p = lane == 0 ? id : lane == 1 ? group : lane == 2 ? m : nullptr;
        f.step = 1;
        if (load && (lane == 3 || lane == 4)) {
            f.p = (int32_t *)load + (lane - 3);
            f.step = 2;
        }
        return f;
    };
    auto store = [&](const Field &f, int i, int id, int j, uint32_t m, uint32_t load) {
        if (f.p) f.p[(int64_t)i * f.step] = lane == 0 ? id : lane == 1 ? j : lane == 2 ? (int)m : lane == 3 ? (int)load : 0;
    };
    auto at = [](auto *p, int64_t i) { return p ? p + i : nullptr; };
    Field f_row = {nullptr, 1}, f_seg = {nullptr, 1};
    if constexpr (FULL_OUT) {
        f_row = field(at(a.o.row_id, g.rbase), at(a.o.row_group, g.rbase), at(a.o.row_m0, g.rbase), at(a.o.row_load, g.rbase));
        f_seg = field(at(a.o.seg_parent, g.n0), at(a.o.seg_group, g.n0), at(a.o.seg_m, g.n0), at(a.o.seg_load, g.n0));
    }
    Field f_node = {nullptr, 1};
    if constexpr (FULL_OUT) f_node = field(nullptr, at(a.o.exec_group, g.n0), at(a.o.m, g.n0), nullptr);
    // Plan row i runs `id` (a segment: >= V) of node `owner` with `load`; z = m | k << 16
    auto write_row = [&](int i, int id, int owner, int j, uint32_t load, uint32_t z, uint32_t c, bool last) {
        if (!FULL_OUT || plan) plan[i] = make_uint4(load, c, z | (last ? 1u << 24 : 0u), (uint32_t)owner);
        if constexpr (FULL_OUT) store(f_row, i, id, j, z & 0xffffu, load);
    };
    // ... a different row in every lane
    auto write_own_row = [&](int i, int id, int j, uint32_t load, uint32_t z, uint32_t c, bool last) {
        if (!FULL_OUT || plan) plan[i] = make_uint4(load, c, z | (last ? 1u << 24 : 0u), (uint32_t)id);
        if constexpr (FULL_OUT) {
            if (a.o.row_id) a.o.row_id[g.rbase + i] = id;
            if (a.o.row_group) a.o.row_group[g.rbase + i] = j;
            if (a.o.row_m0) a.o.row_m0[g.rbase + i] = (int32_t)(z & 0xffffu);
            if (a.o.row_load) a.o.row_load[g.rbase + i] = load;
        }
    };
    // node r finishes with group j on m SMs
    auto finish = [&](uint32_t r, int id, int j, uint32_t m) {
        w.left(r) = 0;
        if constexpr (FULL_OUT) {
            store(f_node, id, id, j, m, 0u);
        } else if (node_out) {
            if (a.o.exec_group) a.o.exec_group[g.n0 + id] = j;
            if (a.o.m) a.o.m[g.n0 + id] = (int32_t)m;
        }
    };
    // ... a different node in every lane
    auto finish_own = [&](uint32_t r, int id, int j, uint32_t m) {
        w.left(r) = 0;
        if (node_out) {
            if (a.o.exec_group) a.o.exec_group[g.n0 + id] = j;
            if (a.o.m) a.o.m[g.n0 + id] = (int32_t)m;
        }
    };
    uint32_t pend = 0;  // !SUM: bits of the lane's word that finished nodes leave set until the next look
    int gn = w.gstart(0);
    int ge = w.gstart(1);
    uint32_t rn = w.gmem(gn);
    for (int j = 0; j < G; j++) {
        const int gb = gn, n = ge - gb;
        uint32_t mw = 0;  // !SUM: the lane's word of the released set
        if constexpr (!SUM)
            if (lane < 2 * g.W) {
                mw = w.rel()[lane] & ~pend;
                w.rel()[lane] = mw;
                pend = 0;
            }
        __syncwarp();
        uint32_t r = rn;  // one member: its rank; up to 32: one per lane
        gn = ge;          // the next group's bounds and first member
        if (j + 1 < G) {
            ge = w.gstart(j + 2);
            rn = w.gmem(gn);
        }
        // ---- members: Eq.5, Eq.1, Lemma 1
        int np;
        T R = 0;
        uint32_t sum_m = 0, vR = 0;
        uint4 q = make_uint4(0, 0, 0, 0);
        uint32_t m = 0, c = 0, live = 0;
        if (n == 1) {
            q = w.rc(r);
            np = q.x > 0;
        } else if (n <= 32) {
            if (lane < n) {
                r = w.gmem(gb + lane);
                q = w.rc(r);
            }
            live = __ballot_sync(FULL, q.x > 0);
            np = __popc(live);
            if (np > 1) {
                const T Wg = Ar::sum(q.x);
                if (q.x) {
                    m = Ar::eq5(q.x, M, Wg);
                    clear_released(w, r);
                }
                __syncwarp();
                if constexpr (!SUM)
                    if (lane < 2 * g.W) mw = w.rel()[lane];
                sum_m = __reduce_add_sync(FULL, m);
                // keep sum m <= M: take from the largest m (ties: higher id); the no-repair
                // variant leaves the rounded SMs as they are
                while (sum_m > M && variant != DAGRT_VAR_NOREPAIR) {
                    const uint32_t top = __reduce_max_sync(FULL, (m << 5) | (uint32_t)lane);
                    m -= (top & 31u) == (uint32_t)lane;
                    sum_m--;
                }
                if (q.x) c = q.y && m == min(q.x, M) ? q.y : Ar::time(q.x, q.w >> 16, m);
                const uint32_t Rm = __reduce_max_sync(FULL, c);
                if constexpr (FULL_OUT) vR = __shfl_sync(FULL, r, __ffs(__ballot_sync(FULL, c == Rm)) - 1);
                R = Rm;
                if (sum_m > M) R = Ar::sum(c);  // over-full (no repair): members one after another
                __syncwarp();
            } else if (np == 1) {
                r = __shfl_sync(FULL, r, __ffs(live) - 1);
                q = w.rc(r);
            }
        } else {
            uint64_t RL;
            np = members_large(w, variant, M, gb, n, lane, &RL, &vR, &sum_m);
            if (np == 1) {
                r = vR;
                q = w.rc(r);
            } else {
                R = (T)RL;
                if constexpr (!SUM)
                    if (lane < 2 * g.W) mw = w.rel()[lane];
            }
        }
        if (np == 0) {  // every member already ran as a parallel node: the group is dropped
            if constexpr (FULL_OUT)
                if (a.o.group_R && lane == 0) a.o.group_R[g.n0 + j] = 0;
            continue;
        }
        const uint32_t deg = q.w & 0xffffu;
        uint32_t s0 = 0;
        if (np == 1) {  // Eq.5 gives m = min(C^, M)
            if ((uint32_t)lane < deg) s0 = w.col(q.z + lane);
            m = min(q.x, M);
            c = q.y;
            if (c == 0) c = Ar::time(q.x, q.w >> 16, m);  // the rest of a split node
            sum_m = m;
            R = c;
            vR = r;
        }
        // ---- parallel launches and node segmentation: released, unfinished nodes outside
        //      pi_j in rank order
        if constexpr (!SUM)  // the only member leaves the released set
            if (np == 1 && (uint32_t)lane == r >> 5) {
                pend = 1u << (r & 31);
                mw &= ~pend;
            }
        const int nrel0 = nrel;
        int nwhole = 0, seg = -1;
        const bool early = !SUM && np == 1 && !defer;
        uint32_t S = sum_m < M && variant != DAGRT_VAR_NOPARA ? M - sum_m : 0u;
        if (S > 0) {
            uint32_t lastz = 0;
            int row = nrows + np, id = 0;
            // next candidate of the scan, -1 at the end; mw (!SUM): the lane's candidates
            int cw = -1, sl = -1;
            uint64_t bits = 0, sbits = 0, sums = 0;
            if constexpr (SUM) {
                if (np == 1 && lane == 0) clear_released(w, r);
                __syncwarp();
                if (lane < ((g.W + 63) >> 6)) sums = ((const uint64_t *)w.sum())[lane];
            }
            auto next = [&]() -> int {
                if constexpr (!SUM) {
                    const uint32_t u = __reduce_min_sync(FULL, mw ? 32u * lane + __ffs(mw) - 1u : 0x7fffffffu);
                    if (u >> 5 == (uint32_t)lane) mw &= mw - 1;
                    return u == 0x7fffffffu ? -1 : (int)u;
                } else {
                    while (!bits) {
                        if (!sbits) {
                            const uint32_t bal = __ballot_sync(FULL, sums != 0) & (sl < 0 ? ~0u : ~0u << sl << 1);
                            if (!bal) return -1;
                            sl = __ffs(bal) - 1;
                            sbits = __shfl_sync(FULL, sums, sl);
                        }
                        const int b = __ffsll((long long)sbits) - 1;
                        sbits &= sbits - 1;
                        cw = sl * 64 + b;
                        bits = ((const uint64_t *)w.rel())[cw];
                        if (!bits) {  // emptied since it was marked
                            if (lane == 0) atomicAnd(w.sum() + 2 * sl + (b >> 5), ~(1u << (b & 31)));
                            __syncwarp();  // before a release marks it again
                        }
                    }
                    const int b = __ffsll((long long)bits) - 1;
                    bits &= bits - 1;
                    return cw * 64 + b;
                }
            };
            int u = next();
            uint4 qu = make_uint4(0, 0, 0, 0);
            if (u >= 0) qu = w.rc(u);
            if (early) {  // every lane has its copy of the released set
                __syncwarp();
                nrel += release_succ<SUM, FULL_OUT>(w, q.z, deg, s0, lane);
            } else if constexpr (!FULL_OUT) {
                __syncwarp();  // (from here on every release ends with one)
            }
            T WS = R * (T)S;  // Eq.6 (literal variant)
            while (u >= 0) {
                if constexpr (FULL_OUT) __syncwarp();  // (not every round has a release)
                const uint32_t x = qu.x, k = qu.w >> 16;
                uint32_t mu = min(x, S), p = 0, cu;
                bool fits;
                id = w.byrank(u);
                if (variant == DAGRT_VAR_LITERAL) {
                    if (WS == 0) break;
                    fits = x <= WS;
                    p = (uint32_t)WS;
                    if (fits) WS -= x;
                    else mu = min(p, S);
                    cu = Ar::time(fits ? x : p, k, mu);
                } else {
                    cu = qu.y;
                    if (x <= S) {
                        if (cu == 0) cu = Ar::time(x, k, x);
                        fits = cu <= R;
                    } else {
                        fits = Ar::fits(x, k, S, R);
                        if (fits) cu = Ar::time(x, k, S);
                    }
                    if (fits) {
                        S -= mu;
                    } else if (variant == DAGRT_VAR_NOSEG) {
                        u = next();
                        if (u >= 0) qu = w.rc(u);
                        continue;
                    } else {
                        p = Ar::split(x, k, S, R);
                        mu = min(p, S);
                        cu = (uint32_t)R;
                    }
                }
                lastz = mu | (k << 16);
                if (!fits) {  // node segmentation: the parallel part runs now
                    seg = nseg++;
                    *(uint2 *)&w.rc(u) = make_uint2(x - p, 0u);
                    write_row(row, g.V + seg, id, j, p, lastz, cu, true);
                    if constexpr (FULL_OUT) store(f_seg, seg, id, j, mu, p);
                    break;
                }
                const uint32_t ub = qu.z, ud = qu.w & 0xffffu;
                uint32_t su = 0;
                if ((uint32_t)lane < ud) su = w.col(ub + lane);
                if constexpr (FULL_OUT) w.lst(nwhole) = (ID)u;
                write_row(row, id, id, j, x, lastz, cu, false);
                finish((uint32_t)u, id, j, mu);
                if constexpr (SUM) {
                    if (lane == 0) clear_released(w, (uint32_t)u);
                } else if ((uint32_t)u >> 5 == (uint32_t)lane) {
                    pend |= 1u << (u & 31);
                }
                row++;
                nwhole++;
                const int u1 = S == 0 ? -1 : next();
                if (u1 >= 0) qu = w.rc(u1);
                // the scan has passed every rank below u, so u's successors, released now,
                // are not seen before the next group
                if (!defer) nrel += release_succ<SUM, FULL_OUT>(w, ub, ud, su, lane);
                u = u1;
            }
            if constexpr (FULL_OUT) __syncwarp();
            // the last launch ends the group
            if (nwhole && seg < 0 && (!FULL_OUT || plan)) plan[row - 1].z = lastz | (1u << 24);
        } else {
            __syncwarp();  // every lane has its copy of the member's record
            if (early) nrel += release_succ<SUM, FULL_OUT>(w, q.z, deg, s0, lane);
        }
        const int nl = nwhole + (seg >= 0);
        if constexpr (FULL_OUT) {
            __syncwarp();
            if (variant != DAGRT_VAR_NOPARA) {  // extra dependencies: counted, and written on request
                if (defer) {
                    if constexpr (SUM) {
                        if (np == 1 && lane == 0) clear_released(w, r);
                    } else if (lane < 2 * g.W) {
                        atomicAnd(w.rel() + lane, ~pend);
                    }
                    __syncwarp();
                    if (lane == 0)
                        write_extra_edges(w, a.o.extra_src + g.ebase, a.o.extra_dst + g.ebase, g.ecap, g.V, vR, nwhole,
                                          seg, nextra);
                    __syncwarp();
                }
                nextra += (int64_t)nl * (w.rc(vR).w & 0xffffu) + (int64_t)(nrel0 - np - nwhole);
            }
        }
        // ---- the members' rows; members finish with pi_j and release their successors
        auto release_lanes = [&](uint32_t b) {  // lane by lane: targets of different members may coincide
            for (; b; b &= b - 1) {
                const int l = __ffs(b) - 1;
                const uint32_t eb = __shfl_sync(FULL, q.z, l), dl = __shfl_sync(FULL, q.w, l) & 0xffffu;
                if (!dl) continue;
                const uint32_t s = (uint32_t)lane < dl ? w.col(eb + lane) : 0u;
                nrel += release_succ<SUM, FULL_OUT>(w, eb, dl, s, lane);
            }
        };
        if (np == 1) {
            const int idm = w.byrank(r);
            write_row(nrows, idm, idm, j, q.x, m | (q.w & 0xffff0000u), c, nl == 0);
            finish(r, idm, j, m);
            if (!early) {
                if (SUM && lane == 0) clear_released(w, r);
                nrel += release_succ<SUM, FULL_OUT>(w, q.z, deg, s0, lane);
            }
        } else if (n <= 32) {
            if (q.x) {
                const int i = __popc(live & ((1u << lane) - 1)), idm = w.byrank(r);
                write_own_row(nrows + i, idm, j, q.x, m | (q.w & 0xffff0000u), c, nl == 0 && i == np - 1);
                finish_own(r, idm, j, m);
            }
            release_lanes(live);
        } else {
            int i = 0;  // rows written
            for (int i0 = 0; i0 < n; i0 += 32) {
                q = make_uint4(0, 0, 0, 0);
                if (i0 + lane < n) {
                    r = w.gmem(gb + i0 + lane);
                    q = w.rc(r);
                }
                live = __ballot_sync(FULL, q.x > 0);
                if (q.x) {
                    const int x = i + __popc(live & ((1u << lane) - 1)), idm = w.byrank(r);
                    const uint32_t mr = w.mm(i0 + lane);
                    write_own_row(nrows + x, idm, j, q.x, mr | (q.w & 0xffff0000u), q.y, nl == 0 && x == np - 1);
                    finish_own(r, idm, j, mr);
                }
                i += __popc(live);
                uint32_t dl = q.x ? q.w & 0xffffu : 0u;
                if constexpr (sizeof(ID) == 2) {
                    // members with few successors (leaves of wide graphs) each by their own lane, the
                    // counts by atomics on their words: targets of different members may coincide
                    uint32_t freed = 0;
                    for (uint32_t e = 0; dl <= kOwnSucc && e < dl; e++) {
                        const uint32_t t = w.col(q.z + e), sh = 16 * (t & 1);
                        const uint32_t old = atomicSub(w.template at<uint32_t>(w.o_cnt) + (t >> 1), 1u << sh);
                        if ((old >> sh & 0xffffu) != 1u) continue;
                        freed++;
                        atomicOr(w.rel() + (t >> 5), 1u << (t & 31));
                        if constexpr (SUM) atomicOr(w.sum() + (t >> 11), 1u << ((t >> 6) & 31));
                    }
                    if constexpr (FULL_OUT) nrel += __reduce_add_sync(FULL, freed);
                    if (dl <= kOwnSucc) dl = 0;
                    __syncwarp();
                }
                release_lanes(__ballot_sync(FULL, dl > 0));
            }
        }
        if constexpr (FULL_OUT) {
            if (defer)  // whole launches, whose release waited for the extra edges
                for (int i = 0; i < nwhole; i++) {
                    const uint4 x = w.rc(w.lst(i));
                    const uint32_t dl = x.w & 0xffffu;
                    const uint32_t s = (uint32_t)lane < dl ? w.col(x.z + lane) : 0u;
                    nrel += release_succ<SUM, FULL_OUT>(w, x.z, dl, s, lane);
                }
            nrel -= np + nwhole;
            if (a.o.group_R && lane == 0) a.o.group_R[g.n0 + j] = (int64_t)R;
        }
        nrows += np + nl;
        bound += R;
        __syncwarp();
    }
    acc.bound = bound;
    acc.nextra = nextra;
    acc.nrows = nrows;
    acc.nseg = nseg;
    acc.err = nrows > 2 * g.V || nseg > g.V;
}

}  // namespace dagrt
