// sched.cu -- per-DAG scheduling and bound kernels (Alg.1, Alg.2, Lemma 1, Theorem 1).
//
// One team (a warp for DAGs that fit a shared-memory workspace, a CTA otherwise) takes a
// whole DAG from a work-stealing counter and runs every step of the method on it without
// leaving its workspace: CSR validation, Kahn levels, the ancestor closure and W^anc
// (Eq.2), Theta and the blocks of Eq.3, the balanced groups of Alg.1, the scheduling loop
// of Alg.2 and the bound of Theorem 1. The schedule is written out as "plan rows" that the
// candidate-bound kernel evaluates other allocations on.
//
// Alg.2 is sequential over the groups of a DAG: one warp of the team runs it.
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "dagrt_internal.cuh"
#include "sched.cuh"

namespace dagrt {

// node state bits
enum : uint8_t { ST_ACTIVE = 1, ST_INT = 2, ST_SEL = 4, ST_JOIN = 32 };
constexpr uint16_t NONE16 = 0xffff;
constexpr int kRelWords = (DAGRT_MAX_V + 63) / 64;  // words of the largest released-set mask
constexpr int kRelBytes = 8 * (kRelWords + kRelWords / 64);  // ... and of its summary
constexpr int kSumWords = 16;  // released-set masks longer than this keep a summary of non-empty words

// ------------------------------------------------------------------ workspace layout
// Persistent arrays live for the whole DAG; the region after them is overlaid by the
// arrays of one phase at a time (A closure, B ordering, C peeling, D member lists, E Alg.2).
struct Ws {
    // persistent
    uint32_t *load;
    uint8_t *kk, *st;
    int32_t *cnt;  // atomic counters: in-degree, Kahn count, in-block parents, open preds
    uint32_t *srp;  // the DAG's successor CSR, staged: offsets ...
    uint16_t *scol; // ... and successor ids
    uint16_t *indeg, *lvl_off, *topo, *rank, *byrank, *blk, *group_of, *gstart, *gmem;
    uint64_t *relmask;
    uint64_t *relsum;  // bit w: relmask[w] may be non-zero (cleared lazily by the scan)
    int32_t *sc;
    // phase A (+ wanc, kept through phase B)
    uint64_t *wanc, *anc, *planes;
    int32_t *poff;  // CTA teams: predecessor lists by node (inclusive offsets) ...
    uint16_t *pid;  // ... and their entries
    // phase B
    uint64_t *skey;
    uint16_t *bk, *pos;
    int32_t *jcnt, *rs, *re;
    // phase C
    int32_t *fcnt, *nround;
    uint64_t *bigk;
    uint16_t *rnd;
    int32_t *thr, *ovl;  // per over-full block: rank of its M-th head; list of over-full blocks
    uint16_t *fr0, *fr1; // the heads of the current round and of the next one (Alg.1)
    uint64_t *hmask;     // CTA teams, Top_M of an over-full block: its heads by rank, one bit each
    int32_t *hcnt;       // ... and the heads in rank words 0..w
    // phase D
    uint16_t *gtmp;
    int32_t *gfill;
    // phase E
    uint4 *rc;  // node records and counters by rank (struct A2)
    uint16_t *lst, *mm;
    // phase F (after Alg.2): the critical-path lower bound
    uint64_t *cpT, *cpM;
};

__host__ __device__ inline int pow2_ceil(int v) {
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Carve a workspace for DAGs of up to vc nodes and ec edges out of `base`; returns the
// bytes used.
__host__ __device__ inline int64_t ws_carve(unsigned char *base, int vc, int ec, Ws *ws, bool cta = false) {
    const int W = ceil_div(vc, 64) > 0 ? ceil_div(vc, 64) : 1;
    const int P = pow2_ceil(vc > 0 ? vc : 1);
    int64_t off = 0;
    auto take = [&](int64_t bytes) {
        unsigned char *p = base + off;
        off = align_up(off + bytes, 16);
        return p;
    };
    Ws w;
    w.load = (uint32_t *)take(4ll * vc);
    w.kk = (uint8_t *)take(vc);
    w.st = (uint8_t *)take(vc);
    w.cnt = (int32_t *)take(4ll * vc);
    w.srp = (uint32_t *)take(4ll * (vc + 1));
    w.scol = (uint16_t *)take(2ll * (ec > 0 ? ec : 1));
    w.indeg = (uint16_t *)take(2ll * vc);
    w.lvl_off = (uint16_t *)take(2ll * (vc + 1));
    w.topo = (uint16_t *)take(2ll * vc);
    w.rank = (uint16_t *)take(2ll * vc);
    w.byrank = (uint16_t *)take(2ll * vc);
    w.blk = (uint16_t *)take(2ll * vc);
    w.group_of = (uint16_t *)take(2ll * vc);
    w.gstart = (uint16_t *)take(2ll * (vc + 2));
    w.gmem = (uint16_t *)take(2ll * vc);
    w.relmask = (uint64_t *)take(8ll * W);
    w.relsum = (uint64_t *)take(8ll * ((W + 63) / 64));
    w.sc = (int32_t *)take(4 * 16);
    const int64_t x0 = off;
    int64_t end = off;
    auto mark = [&]() { end = off > end ? off : end; };
    w.wanc = (uint64_t *)take(8ll * vc);
    const int64_t xa = off;  // phases A and B keep wanc
    w.anc = (uint64_t *)take(8ll * vc * W);
    w.planes = (uint64_t *)take(8ll * 32 * W);
    w.poff = cta ? (int32_t *)take(4ll * (vc + 1)) : nullptr;
    w.pid = cta ? (uint16_t *)take(2ll * (ec > 0 ? ec : 1)) : nullptr;
    mark();
    off = xa;
    w.skey = (uint64_t *)take(8ll * P);
    w.bk = (uint16_t *)take(2ll * vc);
    w.pos = (uint16_t *)take(2ll * vc);
    w.jcnt = (int32_t *)take(4ll * vc);
    w.rs = (int32_t *)take(4ll * vc);
    w.re = (int32_t *)take(4ll * vc);
    mark();
    off = x0;
    w.fcnt = (int32_t *)take(4ll * (vc + 1));
    w.nround = (int32_t *)take(4ll * (vc + 1));
    w.bigk = (uint64_t *)take(8ll * (vc + 1));
    w.rnd = (uint16_t *)take(2ll * vc);
    w.thr = (int32_t *)take(4ll * (vc + 1));
    w.ovl = (int32_t *)take(4ll * (vc + 1));
    w.fr0 = (uint16_t *)take(2ll * vc);
    w.fr1 = (uint16_t *)take(2ll * vc);
    w.hmask = (uint64_t *)take(8ll * W);
    w.hcnt = (int32_t *)take(4ll * W);
    mark();
    off = x0;
    w.gtmp = (uint16_t *)take(2ll * vc);
    w.gfill = (int32_t *)take(4ll * (vc + 1));
    mark();
    off = x0;
    w.rc = (uint4 *)take(16ll * vc);
    w.lst = (uint16_t *)take(2ll * vc);
    w.mm = (uint16_t *)take(2ll * vc);
    mark();
    off = x0;
    w.cpT = (uint64_t *)take(8ll * vc);
    w.cpM = (uint64_t *)take(8ll * vc);
    mark();
    if (ws) *ws = w;
    return align_up(end, 128);
}

int64_t sched_ws_bytes(int vc, int ec) { return ws_carve(nullptr, vc, ec, nullptr, true); }

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
// The arrays are 32-bit offsets, from the kernel's dynamic shared memory (SH) or from a
// global workspace: the compiler then knows the memory space of every access in the chain,
// and the whole set costs ten registers.
template <bool SH>
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
    __device__ __forceinline__ uint16_t &col(uint32_t e) const { return at<uint16_t>(o_col)[e]; }  // successors by edge, as ranks
    __device__ __forceinline__ uint16_t &cnt(uint32_t r) const { return at<uint16_t>(o_cnt)[r]; }  // predecessors not yet finished
    __device__ __forceinline__ uint16_t &gstart(int j) const { return at<uint16_t>(o_gstart)[j]; }
    __device__ __forceinline__ uint16_t &gmem(int i) const { return at<uint16_t>(o_gmem)[i]; }  // members of each group, as ranks, in id order
    __device__ __forceinline__ uint16_t &byrank(uint32_t r) const { return at<uint16_t>(o_byrank)[r]; }
    __device__ __forceinline__ uint16_t &lst(int i) const { return at<uint16_t>(o_lst)[i]; }  // launched nodes of the group
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

template <bool SH>
__device__ __forceinline__ void clear_released(const A2<SH> &w, uint32_t r) {
    atomicAnd(w.rel() + (r >> 5), ~(1u << (r & 31)));
}

// The 32 lanes decrement the open-predecessor counts of a finished node's successors (its
// edges [eb, eb + deg), targets distinct; `s` holds the first 32 edges' targets) and mark
// the ones that reach zero as released; with COUNT, returns how many did.
template <bool SUM, bool COUNT, bool SH>
__device__ __forceinline__ int release_succ(const A2<SH> &w, uint32_t eb, uint32_t deg, uint32_t s, int lane) {
    int n = 0;
    for (uint32_t e = lane; __any_sync(FULL, e < deg); e += 32) {
        bool z = false;
        if (e < deg) {
            if (e >= 32) s = w.col(eb + e);
            const uint32_t c = w.cnt(s) - 1u;
            w.cnt(s) = (uint16_t)c;
            z = c == 0;
            if (z) {
                atomicOr(w.rel() + (s >> 5), 1u << (s & 31));
                if constexpr (SUM) atomicOr(w.sum() + (s >> 11), 1u << ((s >> 6) & 31));
            }
        }
        if constexpr (COUNT) n += __popc(__ballot_sync(FULL, z));
    }
    __syncwarp();  // counts and released bits before the next release or scan
    return n;
}

// Extra dependencies of group j (Alg.2's segmentation step): (v_n, succ(v_R)) for every
// launched part in launch order (the ranks in w.lst, then segment `seg` if one was cut) and
// (v_R, v_n) for every parallel node left in the released set, the split node's residual
// included. Before any node of the group is released from. One lane.
template <bool SH>
__device__ __noinline__ void write_extra_edges(const A2<SH> w, int32_t *src, int32_t *dst, int64_t cap,
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
template <bool SH>
__device__ __noinline__ int members_large(const A2<SH> w, int variant, uint32_t M, int gb, int n, int lane, uint64_t *R,
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

// Alg.2 over all groups of a DAG with Lemma 1 and Theorem 1, by one warp. The group step is
// a serial chain, so it is written for latency: every lane runs the scalar part on the same
// values (no divergence, no hand-over between lanes), a node's record is one 16-byte load,
// the time of a whole launch comes precomputed (on x <= S SMs it is C at min(x, M) SMs), a
// segment's time is R itself (below), and the successors of a finished node are counted
// down by the 32 lanes with plain loads and stores while the first candidate's record is on
// its way. Ranks instead of ids take the lookups out of the chain: the released set is one
// 32-bit word per lane (up to 1,024 nodes) or a mask with a summary word per lane (SUM).
//
// A segment p is the largest load that finishes within R on min(p, S) SMs, and adding one
// tick of load adds at most one tick of time: the part takes exactly R.
//
// What bounds it: the latency of one warp's dependent instructions (a third of the stalls are
// shared-memory loads, the rest fixed-latency arithmetic). Against one lane walking id-indexed
// arrays, a group went from 3,800 to 2,100-2,500 cycles and a call of 10,000 DAGs of 20-200
// nodes from 1.80 to 1.42 ms; 300 DAGs of 100-1,000 nodes from 3.7 to 2.4 ms.
//
// FULL_OUT: some of the outputs that few callers ask for (rows, segments, group times, extra
// dependencies) are wanted; without it the chain does not carry what only they need.
template <bool SUM, bool SH, bool NARROW, bool FULL_OUT>
__device__ __forceinline__ void alg2_warp(const A2<SH> &w, const SchedArgs &a, const Dag &g, int G, Acc &acc, int lane) {
    using Ar = Arith<NARROW>;
    using T = typename Ar::T;
    const uint32_t M = g.M;
    const int variant = g.variant;
    const bool node_out = a.o.m || a.o.exec_group;
    const bool defer = FULL_OUT && g.want_edges;  // nothing is released before the extra edges are written
    uint4 *plan = a.plan ? a.plan + g.rbase : nullptr;
    uint64_t bound = 0;
    int64_t nextra = 0;
    int nrows = 0, nseg = 0, nrel = acc.nrel;
    // plan row i runs `id` (a segment: >= V) of node `owner` with `load`; z = m | k << 16
    auto write_row = [&](int i, int id, int owner, int j, uint32_t load, uint32_t z, uint32_t c, bool last) {
        if (plan) plan[i] = make_uint4(load, c, z | (last ? 1u << 24 : 0u), (uint32_t)owner);
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
        if (node_out) {
            if (a.o.exec_group) a.o.exec_group[g.n0 + id] = j;
            if (a.o.m) a.o.m[g.n0 + id] = (int32_t)m;
        }
    };
    int gn = w.gstart(0);
    int ge = w.gstart(1);
    uint32_t rn = w.gmem(gn);
    for (int j = 0; j < G; j++) {
        const int gb = gn, n = ge - gb;
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
            }
        }
        if (np == 0) {  // every member already ran as a parallel node: the group is dropped
            if constexpr (FULL_OUT)
                if (a.o.group_R && lane == 0) a.o.group_R[g.n0 + j] = 0;
            continue;
        }
        const uint32_t deg = q.w & 0xffffu;
        uint32_t s0 = 0, mw = 0;
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
            } else {
                if (lane < 2 * g.W) mw = w.rel()[lane];
                if (np == 1 && (uint32_t)lane == r >> 5) mw &= ~(1u << (r & 31));
            }
            auto next = [&]() -> int {
                if constexpr (!SUM) {
                    const uint32_t bal = __ballot_sync(FULL, mw != 0);
                    if (!bal) return -1;
                    const int l = __ffs(bal) - 1;
                    const int u = __shfl_sync(FULL, 32 * lane + __ffs(mw) - 1, l);
                    if (lane == l) mw &= mw - 1;
                    return u;
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
                        if (!bits && lane == 0)  // emptied since it was marked
                            atomicAnd(w.sum() + 2 * sl + (b >> 5), ~(1u << (b & 31)));
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
                if (lane == 0) clear_released(w, r);
                nrel += release_succ<SUM, FULL_OUT>(w, q.z, deg, s0, lane);
            }
            T WS = R * (T)S;  // Eq.6 (literal variant)
            while (u >= 0) {
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
                    if (lane == 0) {
                        *(uint2 *)&w.rc(u) = make_uint2(x - p, 0u);
                        write_row(row, g.V + seg, id, j, p, lastz, cu, true);
                        if constexpr (FULL_OUT)
                            if (a.o.seg_parent) {
                                a.o.seg_parent[g.n0 + seg] = id;
                                a.o.seg_load[g.n0 + seg] = (int64_t)p;
                                a.o.seg_m[g.n0 + seg] = (int32_t)mu;
                                a.o.seg_group[g.n0 + seg] = j;
                            }
                    }
                    break;
                }
                const uint32_t ub = qu.z, ud = qu.w & 0xffffu;
                uint32_t su = 0;
                if ((uint32_t)lane < ud) su = w.col(ub + lane);
                if (lane == 0) {
                    w.lst(nwhole) = (uint16_t)u;
                    write_row(row, id, id, j, x, lastz, cu, false);
                    finish((uint32_t)u, id, j, mu);
                    clear_released(w, (uint32_t)u);
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
            // the last launch ends the group
            if (lane == 0 && nwhole && seg < 0 && plan) plan[row - 1].z = lastz | (1u << 24);
        } else if (early) {
            if (lane == 0) clear_released(w, r);
            nrel += release_succ<SUM, FULL_OUT>(w, q.z, deg, s0, lane);
        }
        const int nl = nwhole + (seg >= 0);
        if constexpr (FULL_OUT) {
            __syncwarp();
            if (variant != DAGRT_VAR_NOPARA) {  // extra dependencies: counted, and written on request
                if (defer) {
                    if (np == 1 && lane == 0) clear_released(w, r);
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
        auto release_lanes = [&]() {  // lane by lane: targets of different members may coincide
            for (uint32_t b = live; b; b &= b - 1) {
                const int l = __ffs(b) - 1;
                const uint32_t eb = __shfl_sync(FULL, q.z, l), dl = __shfl_sync(FULL, q.w, l) & 0xffffu;
                const uint32_t s = (uint32_t)lane < dl ? w.col(eb + lane) : 0u;
                nrel += release_succ<SUM, FULL_OUT>(w, eb, dl, s, lane);
            }
        };
        if (np == 1) {
            if (lane == 0) {
                const int idm = w.byrank(r);
                write_row(nrows, idm, idm, j, q.x, m | (q.w & 0xffff0000u), c, nl == 0);
                finish(r, idm, j, m);
            }
            if (!early) {
                if (lane == 0) clear_released(w, r);
                nrel += release_succ<SUM, FULL_OUT>(w, q.z, deg, s0, lane);
            }
        } else if (n <= 32) {
            if (q.x) {
                const int i = __popc(live & ((1u << lane) - 1)), idm = w.byrank(r);
                write_row(nrows + i, idm, idm, j, q.x, m | (q.w & 0xffff0000u), c, nl == 0 && i == np - 1);
                finish(r, idm, j, m);
            }
            release_lanes();
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
                    write_row(nrows + x, idm, idm, j, q.x, mr | (q.w & 0xffff0000u), q.y, nl == 0 && x == np - 1);
                    finish(r, idm, j, mr);
                }
                i += __popc(live);
                release_lanes();
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

// ------------------------------------------------------------------ one DAG
// SH: the workspace is in the kernel's dynamic shared memory
template <int NT, bool SH, bool FULL_OUT>
__device__ void schedule_one(const Team<NT> &tm, const Ws &ws, const SchedArgs &a, int d, int vc, int ec) {
    const int64_t n0 = a.node_off[d];
    const int V = (int)(a.node_off[d + 1] - n0);
    const int64_t e0 = a.edge_off[d];
    const int64_t E = a.edge_off[d + 1] - e0;
    const int32_t *__restrict__ grp = a.row_ptr + n0 + d;
    const int32_t *__restrict__ gcol = a.col + e0;
    const int64_t *__restrict__ wc = a.wcet + n0;
    const uint8_t *__restrict__ kp = a.k64 + n0;
    const uint32_t M = (uint32_t)a.M;
    volatile int32_t *sc = ws.sc;
    const bool lead = tm.t == 0;

    // does not fit this workspace, or its offsets reach outside the arrays
    if (V < 0 || E < 0 || V > vc || E > ec ||
        (a.tot_nodes >= 0 && (n0 < 0 || n0 + V > a.tot_nodes || e0 < 0 || e0 + E > a.tot_edges))) {
        if (lead) write_failure(a, d, a.oversize_status);
        return;
    }

    // ---- validation: row_ptr shape, then loads and fractions, then successor ids; the
    //      CSR is staged into the workspace on the way (all later phases read the copy)
    bool bad = false;
    if (lead) bad = grp[0] != 0 || (int64_t)grp[V] != E;
    for (int v = tm.t; v <= V; v += NT) {
        const int x = grp[v];
        if (v < V && grp[v + 1] < x) bad = true;
        ws.srp[v] = (uint32_t)x;
    }
    if (tm.any(bad)) {
        if (lead) write_failure(a, d, DAGRT_E_INVAL);
        return;
    }
    bool badv = false, badc = false;
    for (int e = tm.t; e < (int)E; e += NT) {
        const int c = gcol[e];
        if (c < 0 || c >= V) badc = true;
        ws.scol[e] = (uint16_t)c;
    }
    for (int v = tm.t; v < V; v += NT) {
        const int64_t w = wc[v];
        const uint8_t k = kp[v];
        if (w < 1 || w > 0xffffffffll || k > 64) badv = true;
        ws.load[v] = (uint32_t)w;
        ws.kk[v] = k;
        ws.cnt[v] = 0;
    }
    tm.sync();
    const uint32_t *__restrict__ rp = ws.srp;
    const uint16_t *__restrict__ col = ws.scol;
    if (!badc) {  // self loops, unsorted or repeated successors (ids are in range here)
        for (int v = tm.t; v < V; v += NT) {
            int prev = -1;
            for (int e = rp[v]; e < (int)rp[v + 1]; e++) {
                const int c = col[e];
                if (c == v || c <= prev) badc = true;
                prev = c;
            }
        }
    }
    if (tm.any(badv)) {
        if (lead) write_failure(a, d, DAGRT_E_INVAL);
        return;
    }
    if (tm.any(badc)) {
        if (lead) write_failure(a, d, DAGRT_E_RANGE);
        return;
    }
    if (V == 0) {
        if (lead) {
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
        return;
    }
    tm.sync();

    // ---- in-degrees (a join has at least two predecessors), one edge per thread
    for (int e = tm.t; e < (int)E; e += NT) atomicAdd(&ws.cnt[col[e]], 1);
    const int W = (V + 63) >> 6;
    if constexpr (NT == 32)  // CTA teams write every word of the closure (pulled below)
        for (int i = tm.t; i < V * W; i += NT) ws.anc[i] = 0;
    if (lead) sc[0] = 0;
    tm.sync();

    // ---- Kahn levels, and (warp teams) the ancestor closure pushed along each level's
    //      out-edges: everything that reaches u, and u itself, reaches each successor of u
    for (int v = tm.t; v < V; v += NT) {
        const int dg = ws.cnt[v];
        ws.indeg[v] = (uint16_t)dg;
        ws.st[v] = dg >= 2 ? ST_JOIN : 0;
        if (dg == 0) {
            const int p = atomicAdd((int *)&sc[0], 1);
            ws.topo[p] = (uint16_t)v;
            if (a.o.level) a.o.level[n0 + v] = 0;
        }
    }
    tm.sync();
    int ls = 0, le = sc[0], L = 0;
    if (lead) ws.lvl_off[0] = 0;
    while (ls < le) {
        // every warp spreads the out-edges of a slice of up to 32 of the level's nodes over
        // its lanes, each lane finding the owner of its edge by a binary search over the
        // slice's edge offsets (an exclusive scan of their out-degrees)
        const int ln = tm.lane();
        for (int base = ls + 32 * tm.warp(); base < le; base += NT) {
            const int i = base + ln;
            const int u = i < le ? ws.topo[i] : 0;
            const int eb = i < le ? (int)rp[u] : 0;
            const int deg = i < le ? (int)rp[u + 1] - eb : 0;
            int x = deg;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, x, o);
                if (ln >= o) x += y;
            }
            const int start = x - deg, total = __shfl_sync(FULL, x, 31);
            for (int f0 = 0; f0 < total; f0 += 32) {
                const int f = f0 + ln;
                int j = 0;  // the last node whose edges start at or before f
                for (int step = 16; step; step >>= 1) {
                    const int sj = __shfl_sync(FULL, start, j + step);
                    if (sj <= f) j += step;
                }
                const int uo = __shfl_sync(FULL, u, j), eo = __shfl_sync(FULL, eb, j);
                const int so = __shfl_sync(FULL, start, j);
                bool rel = false;
                int s = 0;
                if (f < total) {
                    s = col[eo + f - so];
                    if constexpr (NT == 32) {  // warp teams push the closure along the edge
                        const uint64_t *au = ws.anc + (int64_t)uo * W;
                        unsigned long long *as = (unsigned long long *)(ws.anc + (int64_t)s * W);
                        for (int w = 0; w < W; w++) {
                            const uint64_t y = au[w];
                            if (y) atomicOr(&as[w], (unsigned long long)y);
                        }
                        atomicOr(&as[uo >> 6], 1ull << (uo & 63));
                    }
                    rel = atomicSub(&ws.cnt[s], 1) == 1;
                }
                const uint32_t rm = __ballot_sync(FULL, rel);
                int p0 = 0;
                if (ln == 0 && rm) p0 = atomicAdd((int *)&sc[0], __popc(rm));
                p0 = __shfl_sync(FULL, p0, 0);
                if (rel) {
                    ws.topo[p0 + __popc(rm & ((1u << ln) - 1))] = (uint16_t)s;
                    if (a.o.level) a.o.level[n0 + s] = L + 1;
                }
            }
        }
        tm.sync();
        const int ne = sc[0];
        tm.sync();
        L++;
        if (lead) ws.lvl_off[L] = (uint16_t)le;
        ls = le;
        le = ne;
    }
    const int nlev = L;
    if (le != V) {
        if (lead) write_failure(a, d, DAGRT_E_CYCLE);
        return;
    }

    // ---- Eq.2: W^anc(v) = C^_v + sum of C^ over ancestors, by bit planes of C^
    uint64_t mx = 0;
    for (int v = tm.t; v < V; v += NT) mx = mx > ws.load[v] ? mx : ws.load[v];
    mx = tm.maxu(mx);
    const int nb = 64 - __clzll((long long)mx);
    for (int i = tm.t; i < nb * W; i += NT) {
        const int b = i / W, w = i - b * W;
        const int vb = w * 64, ve = min(V, vb + 64);
        uint64_t word = 0;
        for (int v = vb; v < ve; v++) word |= (uint64_t)((ws.load[v] >> b) & 1u) << (v - vb);
        ws.planes[i] = word;
    }
    tm.sync();
    if constexpr (NT == 32) {
        for (int v = tm.t; v < V; v += NT) {
            const uint64_t *av = ws.anc + (int64_t)v * W;
            uint64_t acc = ws.load[v];
            for (int b = 0; b < nb; b++) {
                uint32_t c = 0;
                for (int w = 0; w < W; w++) c += __popcll(av[w] & ws.planes[b * W + w]);
                acc += (uint64_t)c << b;
            }
            ws.wanc[v] = acc;
            if (a.o.wanc) a.o.wanc[n0 + v] = (int64_t)acc;
        }
    } else {
        // CTA teams: the closure pulled level by level with plain loads and stores, each
        // thread one (node, 64-bit word) pair -- everything that reaches a predecessor p,
        // and p itself, reaches v -- and the word's share of W^anc added right away
        for (int v = tm.t; v < V; v += NT) {
            ws.poff[v] = ws.indeg[v];
            ws.wanc[v] = ws.load[v];
        }
        tm.sync();
        team_scan_inplace(tm, ws.poff, V, [](uint64_t x, uint64_t y) { return x + y; }, false);
        for (int u = tm.t; u < V; u += NT)  // ws.cnt is zero again after Kahn's pass
            for (int e = rp[u]; e < (int)rp[u + 1]; e++) {
                const int s = col[e];
                ws.pid[ws.poff[s] - ws.indeg[s] + atomicAdd(&ws.cnt[s], 1)] = (uint16_t)u;
            }
        tm.sync();
        for (int l = 0; l < nlev; l++) {
            const int lb = ws.lvl_off[l], lend = (l + 1 < nlev) ? ws.lvl_off[l + 1] : V;
            const int n_items = (lend - lb) * W;
            for (int it = tm.t; it < n_items; it += NT) {
                const int q = it / W, w = it - q * W;
                const int v = ws.topo[lb + q];
                const int pe = ws.poff[v], pb = pe - ws.indeg[v];
                uint64_t word = 0;
                for (int k = pb; k < pe; k++) {
                    const int p = ws.pid[k];
                    word |= ws.anc[(int64_t)p * W + w];
                    if ((p >> 6) == w) word |= 1ull << (p & 63);
                }
                ws.anc[(int64_t)v * W + w] = word;
                if (word) {
                    uint64_t c = 0;
                    for (int b = 0; b < nb; b++) c += (uint64_t)__popcll(word & ws.planes[b * W + w]) << b;
                    atomicAdd((unsigned long long *)&ws.wanc[v], (unsigned long long)c);
                }
            }
            tm.sync();
        }
        if (a.o.wanc)
            for (int v = tm.t; v < V; v += NT) a.o.wanc[n0 + v] = (int64_t)ws.wanc[v];
    }
    tm.sync();

    // ---- order nodes by (W^anc, id): Theta uses it ascending, Top_M and para(pi_j)
    //      descending with ties broken by lower id
    const int P = pow2_ceil(V);
    for (int i = tm.t; i < P; i += NT)
        ws.skey[i] = i < V ? ((ws.wanc[i] << 16) | (uint64_t)i) : KEY_INF;
    tm.sync();
    team_bitonic_sort(tm, ws.skey, P);
    // per sorted position: join flag (-> Theta index), start and end of its W^anc run
    for (int i = tm.t; i < V; i += NT) {
        const int v = (int)(ws.skey[i] & 0xffff);
        const uint64_t wv = ws.skey[i] >> 16;
        ws.jcnt[i] = (ws.st[v] & ST_JOIN) ? 1 : 0;
        ws.rs[i] = (i == 0 || (ws.skey[i - 1] >> 16) != wv) ? i : 0;
        ws.re[i] = (i == V - 1 || (ws.skey[i + 1] >> 16) != wv) ? i : 0x7fffffff;
    }
    tm.sync();
    team_scan_inplace(tm, ws.jcnt, V, [](uint64_t x, uint64_t y) { return x + y; }, false);
    team_scan_inplace(tm, ws.rs, V, [](uint64_t x, uint64_t y) { return x > y ? x : y; }, false);
    team_scan_inplace(tm, ws.re, V, [](uint64_t x, uint64_t y) { return x < y ? x : y; }, true);
    const int N = ws.jcnt[V - 1];  // number of join nodes
    for (int i = tm.t; i < V; i += NT) {
        const int v = (int)(ws.skey[i] & 0xffff);
        const int r = (V - 1 - ws.re[i]) + (i - ws.rs[i]);
        ws.rank[v] = (uint16_t)r;
        ws.byrank[r] = (uint16_t)v;
        ws.pos[v] = (uint16_t)i;
        ws.bk[v] = NONE16;
    }
    tm.sync();

    // ---- Eq.3 blocks: a node belongs to the first join (in Theta order) it is an ancestor
    //      of, i.e. the smallest sorted position among the joins reachable from it; computed
    //      by a min over successors in reverse level order. No reachable join: residual.
    for (int l = nlev - 1; l >= 0; l--) {
        const int lb = ws.lvl_off[l], lend = (l + 1 < nlev) ? ws.lvl_off[l + 1] : V;
        for (int i = lb + tm.t; i < lend; i += NT) {
            const int v = ws.topo[i];
            int b = NONE16;
            for (int e = rp[v]; e < rp[v + 1]; e++) {
                const int s = col[e];
                if (ws.st[s] & ST_JOIN) b = min(b, (int)ws.pos[s]);
                b = min(b, (int)ws.bk[s]);
            }
            ws.bk[v] = (uint16_t)b;
        }
        tm.sync();
    }
    for (int v = tm.t; v < V; v += NT) {
        const int b = ws.bk[v];
        ws.blk[v] = (uint16_t)(b == NONE16 ? N : ws.jcnt[b] - 1);
    }
    tm.sync();

    // ---- Alg.1: peel every block's out-forest (<= 1 in-block predecessor per node)
    //      round by round; a round of a block takes Top_M of its heads by W^anc (Rule 1),
    //      or a single head with C^ >= M (Rule 2). Blocks are independent, so all of them
    //      advance together; round r of block k becomes the group after block k's
    //      earlier rounds and after every group of blocks 0..k-1.
    for (int v = tm.t; v < V; v += NT) ws.cnt[v] = 0;
    for (int b = tm.t; b <= N; b += NT) {
        ws.fcnt[b] = 0;
        ws.nround[b] = 0;
        ws.bigk[b] = 0;
    }
    if (lead) {  // head counts of the current and the next round (sc[12 + (round & 1)])
        sc[12] = 0;
        sc[13] = 0;
    }
    tm.sync();
    // a block of more than M nodes may have more than M heads in a round (Top_M below)
    bool bigblk = false;
    if (V > (int)M) {
        for (int v = tm.t; v < V; v += NT) atomicAdd(&ws.fcnt[ws.blk[v]], 1);
        tm.sync();
        for (int b = tm.t; b <= N; b += NT) {
            bigblk |= ws.fcnt[b] > (int)M;
            ws.fcnt[b] = 0;
        }
        bigblk = tm.any(bigblk);
        tm.sync();
    }
    if constexpr (NT == 32) {
        // in-block parents, one edge per lane: the edges are in CSR order, so a lane finds its
        // source row a few rows after the row of the round's first edge
        for (int e0 = 0, u0 = 0; e0 < (int)E; e0 += 32) {
            const int e = e0 + tm.t;
            int u = u0;
            if (e < (int)E) {
                while ((int)rp[u + 1] <= e) u++;
                if (ws.blk[col[e]] == ws.blk[u]) atomicAdd(&ws.cnt[col[e]], 1);
            }
            u0 = __shfl_sync(FULL, u, 31);  // lane 31 holds the latest row (or u0 past the end)
        }
    } else {
        for (int u = tm.t; u < V; u += NT)
            for (int e = rp[u]; e < rp[u + 1]; e++)
                if (ws.blk[col[e]] == ws.blk[u]) atomicAdd(&ws.cnt[col[e]], 1);
    }
    tm.sync();
    bad = false;
    for (int v = tm.t; v < V; v += NT) {
        if (ws.cnt[v] > 1) bad = true;
        ws.st[v] = (uint8_t)((ws.st[v] & ST_JOIN) | (ws.cnt[v] == 0 ? ST_ACTIVE : 0));
        if (ws.cnt[v] == 0) ws.fr0[atomicAdd((int *)&sc[12], 1)] = (uint16_t)v;  // the first heads
    }
    if (tm.any(bad)) {
        if (lead) write_failure(a, d, DAGRT_E_INTERNAL);
        return;
    }
    tm.sync();
    // Each round works on the list of its heads only (the nodes marked ST_ACTIVE): the heads
    // that are not selected stay, and a selected node's in-block successor (it has no other
    // in-block predecessor) becomes a head of the next round.
    if (lead) sc[10] = 0;
    tm.sync();
    for (int round = 0;; round++) {
        const int cur = 12 + (round & 1), nxt = 12 + ((round + 1) & 1);
        const int nf = sc[cur];
        if (nf == 0) break;
        if (round > V) {  // every round selects a node, so this cannot happen
            if (lead) write_failure(a, d, DAGRT_E_INTERNAL);
            return;
        }
        const uint16_t *F = (round & 1) ? ws.fr1 : ws.fr0;
        uint16_t *Fn = (round & 1) ? ws.fr0 : ws.fr1;
        // heads per block; a block with more heads than SMs (only in a block of more than M
        // nodes) is listed once, by the head that takes its count past M
        for (int i = tm.t; i < nf; i += NT) {
            const int b = ws.blk[F[i]];
            if (atomicAdd(&ws.fcnt[b], 1) == (int)M && bigblk) ws.ovl[atomicAdd((int *)&sc[10], 1)] = b;
        }
        tm.sync();
        const int nov = sc[10];
        // blocks with more heads than SMs keep their M heaviest (Top_M): the heads up to the
        // rank of the block's M-th head (rank order = W^anc descending). A CTA team finds it
        // for a few such blocks from a bit mask of the block's heads over the ranks (a
        // popcount scan over V/64 words); otherwise one warp per block walks the nodes in rank
        // order with ballots until its M-th head.
        bool masked = false;
        if constexpr (NT > 32) {
            masked = nov > 0 && nov <= 2;
            for (int q = 0; masked && q < nov; q++) {
                const int b = ws.ovl[q];
                for (int w2 = tm.t; w2 < W; w2 += NT) ws.hmask[w2] = 0;
                tm.sync();
                for (int i = tm.t; i < nf; i += NT) {
                    const int v = F[i];
                    if (ws.blk[v] == b)
                        atomicOr((unsigned long long *)&ws.hmask[ws.rank[v] >> 6], 1ull << (ws.rank[v] & 63));
                }
                tm.sync();
                for (int w2 = tm.t; w2 < W; w2 += NT) ws.hcnt[w2] = __popcll(ws.hmask[w2]);
                tm.sync();
                team_scan_inplace(tm, ws.hcnt, W, [](uint64_t x, uint64_t y) { return x + y; }, false);
                for (int w2 = tm.t; w2 < W; w2 += NT) {
                    uint64_t mk = ws.hmask[w2];
                    const int upto = ws.hcnt[w2], before = upto - __popcll(mk);
                    if (before < (int)M && (int)M <= upto) {  // the M-th head is in this word
                        for (int i = 1; i < (int)M - before; i++) mk &= mk - 1;
                        ws.thr[b] = w2 * 64 + __ffsll((long long)mk) - 1;
                    }
                }
                tm.sync();
            }
        }
        for (int q = tm.warp(); !masked && q < nov; q += NT / 32) {
            const int b = ws.ovl[q];
            int cnt = 0, th = V;
            for (int base = 0; base < V; base += 32) {
                const int r = base + tm.lane();
                bool f = false;
                if (r < V) {
                    const int u = ws.byrank[r];
                    f = (ws.st[u] & ST_ACTIVE) && ws.blk[u] == b;
                }
                const uint32_t msk = __ballot_sync(FULL, f);
                const int c = __popc(msk);
                if (cnt + c >= (int)M) {  // the M-th head is in these 32 ranks
                    uint32_t mm = msk;
                    for (int i = 1; i < (int)M - cnt; i++) mm &= mm - 1;
                    th = base + __ffs(mm) - 1;
                    break;
                }
                cnt += c;
            }
            if (tm.lane() == 0) ws.thr[b] = th;
        }
        if (nov) tm.sync();
        if (lead) sc[cur] = 0;  // read by every thread above: it counts the round after next
        for (int i = tm.t; i < nf; i += NT) {
            const int v = F[i];
            const int b = ws.blk[v];
            const bool inT = ws.fcnt[b] <= (int)M || (int)ws.rank[v] <= ws.thr[b];
            if (inT) {
                ws.st[v] |= ST_INT;
                if (ws.load[v] >= M)
                    atomicMax((unsigned long long *)&ws.bigk[b],
                              ((unsigned long long)ws.load[v] << 16) | (0xffffu - ws.rank[v]));
            }
        }
        tm.sync();
        for (int i = tm.t; i < nf; i += NT) {
            const int v = F[i];
            const uint8_t s0 = ws.st[v];
            bool sel = false;
            if (s0 & ST_INT) {
                const uint64_t bg = ws.bigk[ws.blk[v]];
                sel = bg == 0 || (int)(bg & 0xffff) == (int)(0xffffu - ws.rank[v]);
            }
            if (sel) {
                ws.st[v] = (uint8_t)((s0 & ~(ST_INT | ST_ACTIVE)) | ST_SEL);
                ws.rnd[v] = (uint16_t)round;
                atomicMax(&ws.nround[ws.blk[v]], round + 1);
            } else {  // still a head next round
                ws.st[v] = (uint8_t)(s0 & ~ST_INT);
                Fn[atomicAdd((int *)&sc[nxt], 1)] = (uint16_t)v;
            }
        }
        tm.sync();
        for (int i = tm.t; i < nf; i += NT) {
            const int v = F[i];
            const uint8_t s0 = ws.st[v];
            ws.fcnt[ws.blk[v]] = 0;
            ws.bigk[ws.blk[v]] = 0;
            if (s0 & ST_SEL) {
                ws.st[v] = (uint8_t)(s0 & ~ST_SEL);
                for (int e = rp[v]; e < rp[v + 1]; e++) {
                    const int s2 = col[e];
                    if (ws.blk[s2] == ws.blk[v]) {
                        ws.st[s2] |= ST_ACTIVE;
                        Fn[atomicAdd((int *)&sc[nxt], 1)] = (uint16_t)s2;
                    }
                }
            }
        }
        if (lead) sc[10] = 0;
        tm.sync();
    }
    // group index = groups of earlier blocks + round within the block
    team_scan_inplace(tm, ws.nround, N + 1, [](uint64_t x, uint64_t y) { return x + y; }, false);
    const int G = ws.nround[N];
    for (int v = tm.t; v < V; v += NT) {
        const int b = ws.blk[v];
        ws.group_of[v] = (uint16_t)((b ? ws.nround[b - 1] : 0) + ws.rnd[v]);
    }
    tm.sync();

    // ---- member lists of each group, ordered by id, as ranks
    for (int q = tm.t; q <= G; q += NT) ws.gfill[q] = 0;
    tm.sync();
    for (int v = tm.t; v < V; v += NT) atomicAdd(&ws.gfill[ws.group_of[v]], 1);
    tm.sync();
    team_scan_inplace(tm, ws.gfill, G, [](uint64_t x, uint64_t y) { return x + y; }, false);
    for (int q = tm.t; q <= G; q += NT) ws.gstart[q] = (uint16_t)(q ? ws.gfill[q - 1] : 0);
    tm.sync();
    for (int q = tm.t; q <= G; q += NT) ws.gfill[q] = 0;
    tm.sync();
    for (int v = tm.t; v < V; v += NT) {
        const int q = ws.group_of[v];
        const int p = atomicAdd(&ws.gfill[q], 1);
        ws.gtmp[ws.gstart[q] + p] = (uint16_t)v;
    }
    tm.sync();
    for (int i = tm.t; i < V; i += NT) {
        const int v = ws.gtmp[i];
        const int q = ws.group_of[v];
        int pos = 0;
        for (int x = ws.gstart[q]; x < ws.gstart[q + 1]; x++) pos += ws.gtmp[x] < v;
        ws.gmem[ws.gstart[q] + pos] = ws.rank[v];
    }
    tm.sync();

    // ---- Alg.2 over the groups in order, with Lemma 1 and Theorem 1
    int nsrc = 0;
    const bool want_base = a.o.greedy || a.o.greedy_unaware || a.o.graham_para;
    uint64_t b_greedy = 0, b_unaware = 0, b_vol = 0;  // baseline sums (Evaluation section)
    uint16_t *cnt = (uint16_t *)ws.cnt;  // predecessors not yet finished, by rank
    for (int v = tm.t; v < V; v += NT) {
        const uint32_t x = ws.load[v], k = ws.kk[v], r = ws.rank[v];
        const uint32_t cf = (uint32_t)exec_time(x, k, x < M ? x : M, M);
        if (want_base) {
            b_greedy += cf;
            b_unaware = sat_add(b_unaware, exec_time_unaware(x, k, M));
            b_vol += x;
        }
        ws.rc[r] = make_uint4(x, cf, rp[v], (rp[v + 1] - rp[v]) | (k << 16));
        cnt[r] = ws.indeg[v];
        nsrc += ws.indeg[v] == 0;
    }
    for (int e = tm.t; e < (int)E; e += NT) ws.scol[e] = ws.rank[ws.scol[e]];
    nsrc = (int)tm.sum(nsrc);
    if (want_base) {
        b_greedy = tm.sum(b_greedy);
        b_unaware = tm.reduce(b_unaware, [](uint64_t p, uint64_t q) { return sat_add(p, q); });
        b_vol = tm.sum(b_vol);
    }
    for (int w = tm.t; w < W; w += NT) ws.relmask[w] = 0;
    for (int w = tm.t; w < (W + 63) / 64; w += NT) ws.relsum[w] = 0;
    tm.sync();
    // the released set; relsum marks its possibly non-empty words
    for (int v = tm.t; v < V; v += NT)
        if (ws.indeg[v] == 0) {
            const uint32_t r = ws.rank[v];
            atomicOr((uint32_t *)ws.relmask + (r >> 5), 1u << (r & 31));
            if (W > kSumWords) atomicOr((uint32_t *)ws.relsum + (r >> 11), 1u << ((r >> 6) & 31));
        }
    tm.sync();

    Dag g;
    g.n0 = n0;
    g.rbase = 2 * n0;
    g.V = V;
    g.W = W;
    g.M = M;
    g.variant = a.variant;
    g.want_edges = a.o.extra_off != nullptr;
    g.ebase = g.want_edges ? a.o.extra_off[d] : 0;
    g.ecap = g.want_edges ? a.o.extra_off[d + 1] - g.ebase : 0;
    Acc acc;
    acc.nrel = nsrc;
    if (tm.t < 32) {  // the team's first warp
        extern __shared__ __align__(16) unsigned char smem[];
        A2<SH> w2;
        unsigned char *b0 = SH ? smem : (unsigned char *)ws.load;
        auto off = [&](const void *p) { return (uint32_t)((const unsigned char *)p - b0); };
        w2.base = b0;
        w2.o_rc = off(ws.rc);
        w2.o_col = off(ws.scol);
        w2.o_cnt = off(cnt);
        w2.o_gstart = off(ws.gstart);
        w2.o_gmem = off(ws.gmem);
        w2.o_byrank = off(ws.byrank);
        w2.o_lst = off(ws.lst);
        w2.o_mm = off(ws.mm);
        w2.o_rel = (uint32_t)((unsigned char *)ws.relmask - smem);
        w2.o_sum = (uint32_t)((unsigned char *)ws.relsum - smem);
        const bool narrow = 64ull * M * mx < (1ull << 32);
        bool done = false;
        if constexpr (NT > 32)
            if (W > kSumWords) {
                if (narrow) alg2_warp<true, SH, true, FULL_OUT>(w2, a, g, G, acc, tm.t);
                else alg2_warp<true, SH, false, FULL_OUT>(w2, a, g, G, acc, tm.t);
                done = true;
            }
        if (!done) {
            if (narrow) alg2_warp<false, SH, true, FULL_OUT>(w2, a, g, G, acc, tm.t);
            else alg2_warp<false, SH, false, FULL_OUT>(w2, a, g, G, acc, tm.t);
        }
    }
    tm.sync();

    // ---- per-DAG and per-node outputs
    if (lead) {
        // candidate bounds fit 32-bit arithmetic: loads < 2^17 and every group sum of
        // C <= ceil(255/M) * max C^ over at most 2V rows below 2^31
        const uint64_t waves = (255 + M - 1) / M;
        if (a.pflag) a.pflag[d] = (mx < (1ull << 17) && mx * waves * 2ull * (uint64_t)V < (1ull << 31)) ? 1 : 0;
        int code = DAGRT_OK;
        if (acc.err) code = DAGRT_E_INTERNAL;
        else if (g.want_edges && acc.nextra > g.ecap) code = DAGRT_E_CAP;
        const int64_t bnd = code == DAGRT_E_INTERNAL ? -1 : (int64_t)acc.bound;
        a.status[d] = code;
        a.bound[d] = bnd;
        if (a.nrows) a.nrows[d] = acc.nrows;
        if (a.o.status) a.o.status[d] = code;
        if (a.o.bound) a.o.bound[d] = bnd;
        if (a.o.n_groups) a.o.n_groups[d] = G;
        if (a.o.n_seg) a.o.n_seg[d] = acc.nseg;
        if (a.o.n_rows) a.o.n_rows[d] = acc.nrows;
        if (a.o.n_extra) a.o.n_extra[d] = acc.nextra;
        // baselines: Greedy (sequential, m = min(C^, M)), Greedy + unaware (sequential,
        // m = C^), Graham_para (unit-load nodes: L + ceil((vol - L) / M), L = nodes on the
        // longest path)
        if (a.o.greedy) a.o.greedy[d] = (int64_t)b_greedy;
        if (a.o.greedy_unaware) a.o.greedy_unaware[d] = (int64_t)b_unaware;
        if (a.o.graham_para) a.o.graham_para[d] = (int64_t)(nlev + (b_vol - nlev + M - 1) / M);
    }
    for (int v = tm.t; v < V; v += NT) {
        if (a.o.block_of) a.o.block_of[n0 + v] = ws.blk[v];
        if (a.o.group_of) a.o.group_of[n0 + v] = ws.group_of[v];
    }
    tm.sync();

    // ---- critical-path lower bound of the schedule: the longest chain of its parts in G
    //      (a node's parts run one after another, and every edge waits for its tail's last
    //      part), weighted by the parts' times, and the work bound ceil(sum m C / M). Every
    //      execution of the schedule takes at least this long, so Theorem 1's bound must be
    //      at least it: a device-side consistency check (for the variants whose groups fit M
    //      or run in sequence). From the plan rows just written, level by level.
    uint64_t cp = 0;
    if (a.o.crit_path && a.plan) {  // uniform over the team
        if (lead) sc[11] = acc.nrows;  // (Alg.2 is done with the region that phase F overlays)
        for (int v = tm.t; v < V; v += NT) {
            ws.cpT[v] = 0;
            ws.cpM[v] = 0;
        }
        __threadfence_block();  // the plan rows written by other threads of the team
        tm.sync();
        const int nr = sc[11];
        uint64_t work = 0;
        for (int r = tm.t; r < nr; r += NT) {
            const uint4 x = a.plan[g.rbase + r];
            atomicAdd((unsigned long long *)&ws.cpT[x.w], (unsigned long long)x.y);
            work += (uint64_t)(x.z & 0xffffu) * x.y;
        }
        work = tm.sum(work);
        tm.sync();
        for (int l = 0; l < nlev; l++) {
            const int lb = ws.lvl_off[l], lend = (l + 1 < nlev) ? ws.lvl_off[l + 1] : V;
            for (int i = lb + tm.t; i < lend; i += NT) {
                const int v = ws.topo[i];
                const uint64_t dv = ws.cpT[v] + ws.cpM[v];
                ws.cpT[v] = dv;
                for (int e = rp[v]; e < (int)rp[v + 1]; e++)
                    atomicMax((unsigned long long *)&ws.cpM[ws.byrank[col[e]]], (unsigned long long)dv);
            }
            tm.sync();
        }
        uint64_t path = 0;
        for (int v = tm.t; v < V; v += NT) path = ws.cpT[v] > path ? ws.cpT[v] : path;
        path = tm.maxu(path);
        const uint64_t wb = (work + M - 1) / M;
        cp = path > wb ? path : wb;
    }

    if (lead && a.o.crit_path) {
        a.o.crit_path[d] = a.plan ? (int64_t)cp : -1;
        // Theorem 1's bound below a lower bound of every execution: an internal error
        if (a.plan && g.variant != DAGRT_VAR_LITERAL && acc.bound < cp && a.status[d] == DAGRT_OK) {
            write_failure(a, d, DAGRT_E_INTERNAL);
            a.o.crit_path[d] = (int64_t)cp;
        }
    }
    tm.sync();
}

// ------------------------------------------------------------------ kernels
// Warp teams for small DAGs: kWarpsPerCta teams per CTA, each with a shared-memory workspace
// sized for (a.vcap, a.ecap), the largest V and E of the launch's size class.
// Five CTAs an SM (96 registers): at four (128) the 10,000-DAG batch is latency-bound on 16 warps.
template <bool FULL_OUT>
__global__ void __launch_bounds__(32 * kWarpsPerCta, 5) k_sched_warp(SchedArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5;
    Ws ws;
    const int64_t bytes = ws_carve(nullptr, a.vcap, a.ecap, nullptr);
    ws_carve(smem + warp * bytes, a.vcap, a.ecap, &ws);
    Team<32> tm{(int)(threadIdx.x & 31), nullptr};
    for (;;) {
        int idx = 0;
        if (tm.t == 0) idx = atomicAdd(a.counter, 1);
        idx = __shfl_sync(FULL, idx, 0);
        if (idx >= a.n_list) break;
        schedule_one<32, true, FULL_OUT>(tm, ws, a, a.list[idx], a.vcap, a.ecap);
        __syncwarp();
    }
}

// CTA teams for large DAGs: the workspace sized for (a.vcap, a.ecap) lives in dynamic shared
// memory (SMEM) or in the global block a.gws + blockIdx.x * a.gws_stride.
template <int NT, bool SMEM, bool FULL_OUT>
__global__ void __launch_bounds__(NT) k_sched_cta(SchedArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t red[NT / 32];
    __shared__ int idx_s;
    Ws ws;
    ws_carve(SMEM ? smem : a.gws + (int64_t)blockIdx.x * a.gws_stride, a.vcap, a.ecap, &ws, true);
    if constexpr (!SMEM) {  // the released set changes with every group: always in shared memory
        ws.relmask = (uint64_t *)smem;
        ws.relsum = ws.relmask + kRelWords;
    }
    Team<NT> tm{(int)threadIdx.x, red};
    for (;;) {
        if (threadIdx.x == 0) idx_s = atomicAdd(a.counter, 1);
        __syncthreads();
        const int idx = idx_s;
        __syncthreads();
        if (idx >= a.n_list) break;
        schedule_one<NT, SMEM, FULL_OUT>(tm, ws, a, a.list ? a.list[idx] : idx, a.vcap, a.ecap);
        __syncthreads();
    }
}

// ------------------------------------------------------------------ launchers
// Does the call ask for an output that only the FULL_OUT kernels write?
static bool full_out(const dagrt_schedule_out &o) {
    return o.n_extra || o.extra_off || o.group_R || o.seg_parent || o.row_id || o.row_group || o.row_m0 || o.row_load;
}

// Occupancy of the warp kernel per (device, dynamic shared memory), queried once per size
// (a schedule call launches up to 16 classes; these host queries were a visible part of
// its enqueue time).
namespace {
struct WarpLaunchCache {
    std::mutex mu;
    std::map<std::pair<int, int64_t>, int> occ;  // (device, bytes) -> CTAs per SM
    std::map<int, int> max_smem;                 // device -> max_dynamic_smem(k_sched_warp)
};
WarpLaunchCache &warp_cache(bool full) {  // one per kernel
    static WarpLaunchCache c[2];
    return c[full];
}
}  // namespace

cudaError_t sched_launch_warp(const SchedArgs &a, int n_sm, cudaStream_t st) {
    const int64_t bytes = ws_carve(nullptr, a.vcap, a.ecap, nullptr) * kWarpsPerCta;
    const bool full = full_out(a.o);
    const auto kern = full ? k_sched_warp<true> : k_sched_warp<false>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    {
        WarpLaunchCache &c = warp_cache(full);
        std::lock_guard<std::mutex> lock(c.mu);
        auto it = c.occ.find({dev, bytes});
        if (it == c.occ.end() && bytes > sched_smem_limit()) return cudaErrorInvalidValue;
        auto mx = c.max_smem.find(dev);
        if (mx == c.max_smem.end()) mx = c.max_smem.emplace(dev, max_dynamic_smem(kern)).first;
        if (bytes > mx->second) return cudaErrorInvalidValue;
        // the classes differ in size: the attribute allows the largest, whatever launched last
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, mx->second);
        if (e != cudaSuccess) return e;
        if (it != c.occ.end()) {
            per_sm = it->second;
        } else {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kWarpsPerCta, bytes);
            if (e != cudaSuccess) return e;
            c.occ[{dev, bytes}] = per_sm;
        }
    }
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    int grid = n_sm * per_sm;
    const int need = ceil_div(a.n_list, kWarpsPerCta);
    if (grid > need) grid = need;
    if (grid < 1) return cudaSuccess;
    kern<<<grid, 32 * kWarpsPerCta, bytes, st>>>(a);
    return cudaGetLastError();
}

int sched_cta_grid(int n_sm) {
    int best = 1;  // CTAs of the variant with more of them: a grid may be larger than what is resident
    for (auto kern : {k_sched_cta<kCtaThreadsGlobal, false, false>, k_sched_cta<kCtaThreadsGlobal, false, true>}) {
        int per_sm = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCtaThreadsGlobal, kRelBytes);
        if (e == cudaSuccess && per_sm > best) best = per_sm;
    }
    return n_sm * best;
}

cudaError_t sched_launch_cta(const SchedArgs &a, int grid, cudaStream_t st) {
    if (grid < 1 || a.n_list < 1) return cudaSuccess;
    const auto kern = full_out(a.o) ? k_sched_cta<kCtaThreadsGlobal, false, true> : k_sched_cta<kCtaThreadsGlobal, false, false>;
    kern<<<grid, kCtaThreadsGlobal, kRelBytes, st>>>(a);
    return cudaGetLastError();
}

int64_t sched_smem_limit() {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    return optin - (int64_t)sizeof(uint64_t) * (kCtaThreads / 32) - 64;  // the kernel's static shared memory
}

cudaError_t sched_launch_cta_smem(const SchedArgs &a, int n_sm, cudaStream_t st) {
    if (a.n_list < 1) return cudaSuccess;
    const int64_t bytes = sched_ws_bytes(a.vcap, a.ecap);
    const auto kern = full_out(a.o) ? k_sched_cta<kCtaThreads, true, true> : k_sched_cta<kCtaThreads, true, false>;
    const int mx = max_dynamic_smem(kern);
    if (bytes > mx) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCtaThreads, bytes);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    int grid = n_sm * per_sm;
    if (grid > a.n_list) grid = a.n_list;
    kern<<<grid, kCtaThreads, bytes, st>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ schedulability
__global__ void k_schedulable(int32_t n_dags, const int32_t *status, const int64_t *bound, const int64_t *deadline,
                              int32_t *ok, unsigned long long *n_ok) {
    __shared__ unsigned int s_cnt;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    unsigned int mine = 0;
    for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < n_dags; d += gridDim.x * blockDim.x) {
        const bool y = status[d] == DAGRT_OK && bound[d] <= deadline[d];
        if (ok) ok[d] = y ? 1 : 0;
        mine += y;
    }
    mine = __reduce_add_sync(FULL, mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s_cnt, mine);
    __syncthreads();
    if (threadIdx.x == 0 && s_cnt && n_ok) atomicAdd(n_ok, (unsigned long long)s_cnt);
}

cudaError_t sched_schedulable(int32_t n_dags, const int32_t *status, const int64_t *bound, const int64_t *deadline,
                              int32_t *ok, unsigned long long *n_ok, int n_sm, cudaStream_t st) {
    if (n_dags < 1) return cudaSuccess;
    int grid = (n_dags + 255) / 256;
    if (grid > 4 * n_sm) grid = 4 * n_sm;
    k_schedulable<<<grid, 256, 0, st>>>(n_dags, status, bound, deadline, ok, n_ok);
    return cudaGetLastError();
}

}  // namespace dagrt
