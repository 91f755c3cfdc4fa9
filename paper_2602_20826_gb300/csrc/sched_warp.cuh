// sched_warp.cuh -- the whole schedule of one DAG of at most 256 nodes by one warp.
//
// What bounds these DAGs is the length of one warp's serial chain, times how many of them an
// SM holds and how many instructions they issue. All three decide the layout. Ids, ranks,
// blocks, groups and in-degrees are bytes and the phases overlay one region: a 208-node DAG of
// 2,400 edges takes 14 instead of 21 KB (16 instead of 8 teams an SM). The closure goes from
// node to node in topological order, a lane per successor and 128 bits, without atomics or
// level barriers (176,000 -> 49,000 cycles at 200 nodes); the (W^anc, id) order is a bitonic
// network in registers (45,000 -> 4,000); every lane reads the blocks of its own nodes off the
// joins' rows (42,000 -> 10,000); a round of Alg.1 asks each node whether its only in-block
// predecessor has been selected (77,000 -> 26,000), large blocks apart (peel_solo). Alg.2 is then
// 65% of a DAG's 396,000 cycles.
// 10,000 DAGs of 20-200 nodes, load and schedule: 1.42 -> 0.67 ms (four warps a CTA, five CTAs
// an SM; 6 CTAs at 80 registers 0.93, 2 warps 0.83, size classes of 32 nodes 0.85 against 0.83
// when these were timed).
#pragma once

#include "alg2.cuh"

namespace dagrt {

constexpr int kWarpMaxV = 256;

// Offsets of one team's arrays in shared memory, from the team's base. vc is a multiple of 16.
struct WarpWs {
    uint32_t load, srp, scol, kk, indeg, lpred;                       // the DAG, kept
    uint32_t wanc;                                                    // until the nodes are ordered; then
    uint32_t rank, byrank, blk, gmem, group_of, gstart;               // ... these
    uint32_t anc, topo, cnt, planes;                                  // closure and Kahn's pass, then
    uint32_t bigk, nround, fcnt, rnd;                                 // ... Alg.1, then
    uint32_t rc, cpT, cpM, acnt, lst, mm, rel;                        // ... Alg.2 and the critical path
    uint32_t bytes;
    int rw;  // 32-bit words of a closure row: a power of two
};

__host__ __device__ inline WarpWs warp_carve(int vc, int ec) {
    WarpWs w;
    uint32_t off = 0;
    auto take = [&](int bytes) {
        const uint32_t p = off;
        off += (uint32_t)(bytes + 15) / 16 * 16;
        return p;
    };
    w.rw = vc <= 32 ? 1 : vc <= 64 ? 2 : vc <= 128 ? 4 : 8;
    w.load = take(4 * vc);
    w.srp = take(2 * (vc + 1));
    w.scol = take(ec > 0 ? ec : 1);
    w.kk = take(vc);
    w.indeg = take(vc);
    w.lpred = take(vc);
    const uint32_t y = off;
    w.wanc = take(8 * vc);
    const uint32_t yend = off;
    off = y;
    w.rank = take(vc);
    w.byrank = take(vc);
    w.blk = take(vc);
    w.gmem = take(vc);
    w.group_of = take(vc);
    w.gstart = take(2 * (vc + 2));
    off = off > yend ? off : yend;
    const uint32_t x = off;
    uint32_t end = off;
    auto mark = [&]() {
        end = off > end ? off : end;
        off = x;
    };
    w.anc = take(4 * w.rw * vc);
    w.topo = take(vc);
    w.cnt = take(vc);
    w.planes = take(4 * 32 * w.rw);
    mark();
    w.bigk = take(8 * vc);
    w.nround = take(2 * vc);
    w.fcnt = take(4 * vc);
    w.rnd = take(2 * vc);
    mark();
    w.rc = take(16 * vc);
    const uint32_t e = off;
    w.acnt = take(vc);
    w.lst = take(vc);
    w.mm = take(2 * vc);
    w.rel = take(4 * 8);
    const uint32_t eend = off;
    off = e;
    w.cpT = take(8 * vc);
    w.cpM = take(8 * vc);
    off = off > eend ? off : eend;
    mark();
    w.bytes = (end + 15) / 16 * 16;
    return w;
}

// Ascending bitonic sort of 32 R keys, key e = R lane + j in x[j].
template <int R, class K>
__device__ __forceinline__ void warp_sort(K (&x)[R], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
        for (int s = k >> 1; s > 0; s >>= 1) {
            if (s >= R) {
                const bool up = k >= 32 * R || ((lane * R) & k) == 0;
                const bool keep_min = (((lane * R) & s) == 0) == up;
#pragma unroll
                for (int j = 0; j < R; j++) {
                    const K y = __shfl_xor_sync(FULL, x[j], s / R);
                    x[j] = keep_min ? (y < x[j] ? y : x[j]) : (y > x[j] ? y : x[j]);
                }
            } else {
#pragma unroll
                for (int j = 0; j < R; j++) {
                    if (j & s) continue;
                    const bool up = k >= R ? (k >= 32 * R || ((lane * R) & k) == 0) : (j & k) == 0;
                    const K a = x[j], b = x[j | s];
                    const bool sw = (b < a) == up;
                    x[j] = sw ? b : a;
                    x[j | s] = sw ? a : b;
                }
            }
        }
    }
}

constexpr uint32_t kNone = 0xffffu;  // no round yet
constexpr int kSoloNodes = 32;

// Alg.1 on one block of n nodes by the warp: sets its nodes' rounds (kNone before) and returns their
// number. A lane keeps its nodes 32 c + lane as bit masks over c and their in-block predecessors as
// bytes in two registers, so a round of Rule 2 costs two warp reductions, a look at the lane's own
// heads and a byte comparison, however many nodes wait. A forest with loads above M has a round per
// node: rounds that scan all nodes, with one 64-bit atomic maximum per head, took 10,000 cycles each
// for 256 isolated nodes (600 binary trees of 256 nodes, loads up to 10,000: 1,245 -> 300 us).
// `mask`: 8 words, zero before and after.
__device__ __forceinline__ uint32_t peel_solo(uint32_t b, uint32_t n, uint32_t M, int V, int NC, const uint32_t *load,
                                           const uint8_t *rank, const uint8_t *byrank, const uint8_t *blk,
                                           const uint8_t *lpred, uint16_t *rnd, uint32_t *mask, int lane) {
    uint32_t open = 0, head = 0;  // the block's nodes that are not selected yet, and the heads among them
    uint32_t plo = 0, phi = 0;    // in-block predecessors (a head at the start: the node itself)
    for (int c = 0; c < NC; c++) {
        const int v = 32 * c + lane;
        if (v >= V || blk[v] != b) continue;
        const uint32_t p = lpred[v];
        open |= 1u << c;
        head |= (uint32_t)(p == (uint32_t)v) << c;
        if (c < 4) plo |= p << (8 * c);
        else phi |= p << (8 * (c - 4));
    }
    auto equal = [](uint32_t x, uint32_t y) {  // bit i: byte i of x is that of y
        return (((__vcmpeq4(x, y) & 0x01010101u) * 0x01020408u) >> 24) & 0xfu;
    };
    uint32_t round = 0;
    for (; __any_sync(FULL, head != 0); round++) {
        uint32_t top = head;
        if (n > M && __reduce_add_sync(FULL, (uint32_t)__popc(head)) > M) {
            // Top_M: heads up to the rank of the M-th, from a bit mask over the ranks
            for (uint32_t m = head; m; m &= m - 1) {
                const uint32_t r = rank[32 * (__ffs(m) - 1) + lane];
                atomicOr(&mask[r >> 5], 1u << (r & 31));
            }
            __syncwarp();
            const uint32_t word = lane < 8 ? mask[lane] : 0u;
            uint32_t upto = __popc(word);  // heads in words 0 .. lane
            for (int o = 1; o < 8; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL, upto, o);
                if (lane >= o) upto += y;
            }
            const int w = __ffs(__ballot_sync(FULL, upto >= M)) - 1;
            const uint32_t bits = __shfl_sync(FULL, word, w), last = __shfl_sync(FULL, upto, w);
            const uint32_t at = __popc(bits) - (last - M);  // the M-th head is this word's at-th
            const uint32_t it = __ballot_sync(FULL, (bits >> lane & 1u) && (uint32_t)__popc(bits << (31 - lane)) == at);
            const uint32_t th = 32 * w + __ffs(it) - 1;
            __syncwarp();
            if (lane < 8) mask[lane] = 0;
            for (uint32_t m = head; m; m &= m - 1)
                if (rank[32 * (__ffs(m) - 1) + lane] > th) top &= ~(m & (0u - m));
            __syncwarp();
        }
        uint32_t x = 0, r = ~0u;  // the largest load of at least M, then the lowest rank
        for (uint32_t m = top; m; m &= m - 1) {
            const int v = 32 * (__ffs(m) - 1) + lane;
            const uint32_t xv = load[v], rv = rank[v];
            if (xv >= M && (xv > x || (xv == x && rv < r))) {
                x = xv;
                r = rv;
            }
        }
        const uint32_t big = __reduce_max_sync(FULL, x);
        if (big) {  // it runs alone
            const uint32_t v = byrank[__reduce_min_sync(FULL, x == big ? r : ~0u)];
            if ((v & 31u) == (uint32_t)lane) {
                rnd[v] = (uint16_t)round;
                open &= ~(1u << (v >> 5));
                head &= open;
            }
            head |= (equal(plo, v * 0x01010101u) | equal(phi, v * 0x01010101u) << 4) & open;
        } else {
            for (uint32_t m = top; m; m &= m - 1) rnd[32 * (__ffs(m) - 1) + lane] = (uint16_t)round;
            open &= ~top;
            head &= open;
            __syncwarp();
            for (uint32_t m = open & ~head; m; m &= m - 1) {
                const int c = __ffs(m) - 1;
                const uint32_t p = (c < 4 ? plo >> (8 * c) : phi >> (8 * (c - 4))) & 0xffu;
                if (rnd[p] != kNone) head |= 1u << c;
            }
            __syncwarp();
        }
    }
    return round;
}

template <bool FULL_OUT>
__device__ __forceinline__ void schedule_warp(const WarpWs &ws, uint32_t base, const SchedArgs &a, int d, int lane) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int64_t n0 = a.node_off[d];
    const int V = (int)(a.node_off[d + 1] - n0);
    const int64_t e0 = a.edge_off[d];
    const int64_t E64 = a.edge_off[d + 1] - e0;
    const uint32_t M = (uint32_t)a.M, lt = (1u << lane) - 1;
    if (V < 0 || E64 < 0 || V > a.vcap || E64 > a.ecap) {  // does not fit this workspace
        if (lane == 0) write_failure(a, d, a.oversize_status);
        return;
    }
    const int E = (int)E64, NC = (V + 31) >> 5;  // chunks of 32 nodes
    const int32_t *__restrict__ grp = a.row_ptr + n0 + d;
    const int32_t *__restrict__ gcol = a.col + e0;
    uint32_t *load = (uint32_t *)(smem + base + ws.load);
    uint16_t *srp = (uint16_t *)(smem + base + ws.srp);
    uint8_t *scol = smem + base + ws.scol, *kk = smem + base + ws.kk, *indeg = smem + base + ws.indeg;
    uint8_t *lpred = smem + base + ws.lpred;
    uint64_t *wanc = (uint64_t *)(smem + base + ws.wanc);
    uint8_t *rank = smem + base + ws.rank, *byrank = smem + base + ws.byrank, *blk = smem + base + ws.blk;
    uint8_t *gmem = smem + base + ws.gmem, *group_of = smem + base + ws.group_of;
    uint16_t *gstart = (uint16_t *)(smem + base + ws.gstart);
    uint32_t *anc = (uint32_t *)(smem + base + ws.anc);
    uint8_t *topo = smem + base + ws.topo, *cnt = smem + base + ws.cnt;

    // ---- validation: row_ptr shape, then loads and fractions, then successor ids; the CSR is
    //      staged on the way
    bool bad = false;
    if (lane == 0) bad = grp[0] != 0 || (int64_t)grp[V] != E64;
    for (int v = lane; v <= V; v += 32) {
        const int x = grp[v];
        if (v < V && grp[v + 1] < x) bad = true;
        srp[v] = (uint16_t)x;
    }
    if (__any_sync(FULL, bad)) {
        if (lane == 0) write_failure(a, d, DAGRT_E_INVAL);
        return;
    }
    bool badv = false, badc = false;
    for (int e = lane; e < E; e += 32) {
        const int c = gcol[e];
        if (c < 0 || c >= V) badc = true;
        scol[e] = (uint8_t)c;
    }
    uint32_t mx = 0;
    uint64_t vol = 0;
    for (int v = lane; v < V; v += 32) {
        const int64_t w = a.wcet[n0 + v];
        const uint8_t k = a.k64[n0 + v];
        if (w < 1 || w > 0xffffffffll || k > 64) badv = true;
        load[v] = (uint32_t)w;
        kk[v] = k;
        mx = max(mx, (uint32_t)w);
        vol += (uint32_t)w;
    }
    for (int i = lane; i < (V + 3) / 4; i += 32) ((uint32_t *)cnt)[i] = 0;
    bool inorder = true;  // every edge leads to a larger id
    __syncwarp();
    if (!__any_sync(FULL, badc)) {  // self loops, unsorted or repeated successors (ids are in range)
        for (int v = lane; v < V; v += 32) {
            int prev = -1;
            for (int e = srp[v]; e < (int)srp[v + 1]; e++) {
                const int c = scol[e];
                if (c == v || c <= prev) badc = true;
                inorder &= c > v;
                prev = c;
            }
        }
    } else {
        badc = true;
    }
    if (__any_sync(FULL, badv)) {
        if (lane == 0) write_failure(a, d, DAGRT_E_INVAL);
        return;
    }
    if (__any_sync(FULL, badc)) {
        if (lane == 0) write_failure(a, d, DAGRT_E_RANGE);
        return;
    }
    if (V == 0) {
        if (lane == 0) write_empty(a, d);
        return;
    }
    mx = __reduce_max_sync(FULL, mx);
    for (int o = 16; o > 0; o >>= 1) vol += __shfl_xor_sync(FULL, vol, o);

    // ---- in-degrees (four counters a word; at most 255 each), sources, an empty closure
    for (int e = lane; e < E; e += 32) {
        const uint32_t s = scol[e];
        atomicAdd((uint32_t *)cnt + (s >> 2), 1u << (8 * (s & 3)));
    }
    const int rw = ws.rw;
    for (int i = lane; i < V * rw; i += 32) anc[i] = i % rw == i / rw >> 5 ? 1u << (i / rw & 31) : 0u;
    __syncwarp();
    int tail = 0;
    for (int c = 0; c < NC; c++) {
        const int v = 32 * c + lane;
        const bool src = v < V && cnt[v] == 0;
        if (v < V) indeg[v] = cnt[v];
        const uint32_t sb = __ballot_sync(FULL, src);
        if (src) {
            topo[tail + __popc(sb & lt)] = (uint8_t)v;
        }
        tail += __popc(sb);
    }
    const int nsrc = tail;
    __syncwarp();

    // ---- levels and the ancestor closure (with the node itself): nodes in topological order, so
    //      a node's row is complete when its turn comes and goes to its successors, a lane per
    //      successor and 128 bits (they are distinct: plain loads and stores). Where every edge
    //      leads to a larger id, ids are the order and levels are pushed along; else Kahn's queue
    //      gives both.
    auto closure = [&](auto rwc) -> int {  // the number of levels, 0 with a cycle
        constexpr int RW = decltype(rwc)::value;
        constexpr int LPE = RW == 8 ? 2 : 1;  // lanes per edge
        using T = typename std::conditional<(RW >= 4), uint4, typename std::conditional<RW == 2, uint2, uint32_t>::type>::type;
        T *rows = (T *)anc;
        const int part = lane & (LPE - 1), el = lane / LPE;
        auto merge = [](T &x, const T &y) {
            if constexpr (RW >= 4) x.z |= y.z, x.w |= y.w;
            if constexpr (RW >= 2) x.x |= y.x, x.y |= y.y;
            else x |= y;
        };
        if (__all_sync(FULL, inorder)) {
            uint8_t *lev = cnt;  // the counts are kept as indeg
            for (int i = lane; i < (V + 3) / 4; i += 32) ((uint32_t *)lev)[i] = 0;
            __syncwarp();
            int end = 0, top = 0;
            for (int u = 0; u < V; u++) {
                const int eb = end;
                end = srp[u + 1];
                const uint32_t l = lev[u] + 1u;
                const T row = rows[u * LPE + part];
                for (int e = eb + el; e < end; e += 32 / LPE) {
                    const uint32_t s = scol[e];
                    const uint32_t ls = lev[s];
                    T x = rows[s * LPE + part];
                    merge(x, row);
                    rows[s * LPE + part] = x;
                    lev[s] = (uint8_t)max(ls, l);
                    lpred[s] = (uint8_t)u;
                }
                top = max(top, (int)l);
                __syncwarp();
            }
            if (a.o.level)
                for (int v = lane; v < V; v += 32) a.o.level[n0 + v] = lev[v];
            return top;
        }
        int head = 0, lend = tail, L = 0;
        while (head < tail) {
            if (head == lend) {
                L++;
                lend = tail;
            }
            const uint32_t u = topo[head++];
            const int eb = srp[u], end = srp[u + 1];
            const T row = rows[u * LPE + part];
            for (int e0 = eb; e0 < end; e0 += 32 / LPE) {
                const bool act = e0 + el < end;
                uint32_t s = 0, c = 1;
                if (act) {
                    s = scol[e0 + el];
                    T x = rows[s * LPE + part];
                    merge(x, row);
                    rows[s * LPE + part] = x;
                    c = cnt[s] - 1u;
                }
                __syncwarp();  // both lanes of an edge have read its count
                if (act) cnt[s] = (uint8_t)c;
                const bool z = c == 0 && part == 0;
                const uint32_t zb = __ballot_sync(FULL, z);
                if (z) {
                    topo[tail + __popc(zb & lt)] = (uint8_t)s;
                    lpred[s] = (uint8_t)u;
                    if (a.o.level) a.o.level[n0 + s] = L + 1;
                }
                tail += __popc(zb);
            }
            __syncwarp();
        }
        if (a.o.level)  // sources
            for (int v = lane; v < V; v += 32)
                if (indeg[v] == 0) a.o.level[n0 + v] = 0;
        return tail == V ? L + 1 : 0;
    };
    const int nlev = rw == 8   ? closure(std::integral_constant<int, 8>())
                     : rw == 4 ? closure(std::integral_constant<int, 4>())
                     : rw == 2 ? closure(std::integral_constant<int, 2>())
                               : closure(std::integral_constant<int, 1>());
    if (nlev == 0) {
        if (lane == 0) write_failure(a, d, DAGRT_E_CYCLE);
        return;
    }

    // ---- Eq.2: W^anc(v) = sum of C^ over the node and its ancestors, by bit planes of C^
    uint32_t *planes = (uint32_t *)(smem + base + ws.planes);
    const int nb = 32 - __clz(mx);
    for (int c = 0; c < NC; c++) {
        const uint32_t x = 32 * c + lane < V ? load[32 * c + lane] : 0u;
        for (int b = 0; b < nb; b++) {
            const uint32_t p = __ballot_sync(FULL, (x >> b) & 1u);
            if (lane == 0) planes[b * rw + c] = p;
        }
    }
    for (int i = lane; i < nb * (rw - NC); i += 32) planes[i / (rw - NC) * rw + NC + i % (rw - NC)] = 0;
    __syncwarp();
    auto weigh = [&](auto rwc) {
        constexpr int RW = decltype(rwc)::value;
        for (int v = lane; v < V; v += 32) {
            uint32_t x[RW];
#pragma unroll
            for (int i = 0; i < RW; i++) x[i] = anc[v * RW + i];
            uint64_t W = 0;
            for (int b = 0; b < nb; b++) {
                uint32_t n = 0;
#pragma unroll
                for (int i = 0; i < RW; i++) n += __popc(x[i] & planes[b * RW + i]);
                W += (uint64_t)n << b;
            }
            anc[v * RW + (v >> 5)] &= ~(1u << (v & 31));  // the blocks are about other nodes
            wanc[v] = W;
            if (a.o.wanc) a.o.wanc[n0 + v] = (int64_t)W;
        }
    };
    if (rw == 8) weigh(std::integral_constant<int, 8>());
    else if (rw == 4) weigh(std::integral_constant<int, 4>());
    else if (rw == 2) weigh(std::integral_constant<int, 2>());
    else weigh(std::integral_constant<int, 1>());
    __syncwarp();

    // ---- order by (W^anc descending, id ascending); Theta (W^anc ascending, id ascending) is
    //      that order backwards but for nodes of equal W^anc. topo now lists nodes in Theta's
    //      order, cnt marks ranks whose W^anc equals that of the rank before.
    auto order = [&](auto rc, auto kc) {
        constexpr int R = decltype(rc)::value;
        using K = decltype(kc);
        constexpr int kWBits = 8 * sizeof(K) - 8;
        K x[R];
#pragma unroll
        for (int j = 0; j < R; j++) {
            const int v = lane * R + j;
            x[j] = v < V ? (K)((((K)1 << kWBits) - 1 - (K)wanc[v]) << 8 | (K)v) : ~(K)0;
        }
        __syncwarp();
        warp_sort<R, K>(x, lane);
        const K before = __shfl_up_sync(FULL, x[R - 1], 1);
        bool any = false;
#pragma unroll
        for (int j = 0; j < R; j++) {
            const int r = lane * R + j;
            if (r >= V) break;
            const K p = j ? x[j - 1] : before;
            const bool tie = r > 0 && (p >> 8) == (x[j] >> 8);
            any |= tie;
            const uint32_t v = (uint32_t)x[j] & 0xffu;
            rank[v] = (uint8_t)r;
            byrank[r] = (uint8_t)v;
            cnt[r] = tie;
            topo[V - 1 - r] = (uint8_t)v;
        }
        any = __any_sync(FULL, any);
        __syncwarp();
        if (any) {
            for (int r = lane; r < V; r += 32) {
                int f = r, t = r;  // the run of equal W^anc
                while (cnt[f]) f--;
                while (t + 1 < V && cnt[t + 1]) t++;
                if (f < t) topo[V - 1 - t + (r - f)] = byrank[r];
            }
            __syncwarp();
        }
    };
    if (vol < (1ull << 24) - 1) {
        if (V <= 128) order(std::integral_constant<int, 4>(), uint32_t());
        else order(std::integral_constant<int, 8>(), uint32_t());
    } else {
        order(std::integral_constant<int, 8>(), (unsigned long long)0);
    }

    // ---- Eq.3 blocks: block t is what the t-th join of Theta has as ancestors and no earlier
    //      join has; without a join below it, a node is in the residual block N. A lane owns rw
    //      nodes, bits q rw .. of word wi, and takes the joins backwards: the last one that
    //      finds a node's bit set is the first join. Nothing waits for anything but the row.
    uint8_t *joins = cnt;  // the joins in Theta's order
    int N = 0;
    for (int c = 0; c < NC; c++) {
        const int p = 32 * c + lane;
        const uint32_t u = p < V ? topo[p] : 0u;
        const bool join = p < V && indeg[u] >= 2;
        const uint32_t jb = __ballot_sync(FULL, join);
        if (join) joins[N + __popc(jb & lt)] = (uint8_t)u;
        N += __popc(jb);
    }
    __syncwarp();
    auto blocks = [&](auto rwc) {
        constexpr int RW = decltype(rwc)::value;
        const int wi = lane & (RW - 1), q = lane / RW;
        uint32_t b[RW];
#pragma unroll
        for (int i = 0; i < RW; i++) b[i] = (uint32_t)N;
#pragma unroll 4
        for (int t = N - 1; t >= 0; t--) {
            const uint32_t row = anc[joins[t] * RW + wi] >> (q * RW);
#pragma unroll
            for (int i = 0; i < RW; i++)
                if (row & (1u << i)) b[i] = (uint32_t)t;
        }
#pragma unroll
        for (int i = 0; i < RW; i++)
            if (32 * wi + q * RW + i < V) blk[32 * wi + q * RW + i] = (uint8_t)b[i];
    };
    if (rw == 8) blocks(std::integral_constant<int, 8>());
    else if (rw == 4) blocks(std::integral_constant<int, 4>());
    else if (rw == 2) blocks(std::integral_constant<int, 2>());
    else blocks(std::integral_constant<int, 1>());
    __syncwarp();

    // ---- Alg.1: peel every block's out-forest round by round; a round of a block takes Top_M
    //      of its heads by W^anc (Rule 1), or a single head with C^ >= M (Rule 2). Blocks of more
    //      than kSoloNodes nodes (they may have a round per node) or than M (more than M heads) are
    //      peeled one after another, then all others advance together. A node has an in-block
    //      predecessor only if it has a single predecessor (a join's ancestors are in blocks up to
    //      its own, it is in a later one).
    uint16_t *rnd = (uint16_t *)(smem + base + ws.rnd), *nround = (uint16_t *)(smem + base + ws.nround);
    unsigned long long *bigk = (unsigned long long *)(smem + base + ws.bigk);
    uint32_t *fcnt = (uint32_t *)(smem + base + ws.fcnt);
    for (int v = lane; v < V; v += 32) {
        rnd[v] = (uint16_t)kNone;
        nround[v] = 0;
        bigk[v] = 0;
        fcnt[v] = 0;
        // (the byte of) the in-block predecessor, or the node itself
        const uint32_t p = indeg[v] == 1 ? lpred[v] : (uint32_t)v;
        lpred[v] = (uint8_t)(blk[p] == blk[v] ? p : (uint32_t)v);
    }
    __syncwarp();
    if (V > kSoloNodes || V > (int)M) {
        for (int v = lane; v < V; v += 32) atomicAdd(&fcnt[blk[v]], 1u);
        __syncwarp();
        for (int c = 0; c < NC; c++) {
            const uint32_t n = 32 * c + lane < V ? fcnt[32 * c + lane] : 0u;  // the block's nodes
            for (uint32_t m = __ballot_sync(FULL, n > min((uint32_t)kSoloNodes, M)); m; m &= m - 1) {
                const int b = 32 * c + __ffs(m) - 1;
                const uint32_t rounds = peel_solo(b, __shfl_sync(FULL, n, __ffs(m) - 1), M, V, NC, load, rank, byrank, blk,
                                                  lpred, rnd, (uint32_t *)bigk, lane);
                if (lane == 0) nround[b] = (uint16_t)rounds;
            }
        }
        __syncwarp();
    }
    // the key of a head that Rule 2 may take alone: the largest load, then the lowest rank
    auto big_key = [&](uint32_t v) { return ((unsigned long long)load[v] << 16) | (0xffffu - rank[v]); };
    for (uint32_t round = 0;; round++) {
        uint32_t hm = 0;  // this lane's heads by chunk: all of them are in Top_M
        for (int c = 0; c < NC; c++) {
            const int v = 32 * c + lane;
            if (v < V && rnd[v] == kNone) {
                const uint32_t p = lpred[v];
                if (p == (uint32_t)v || rnd[p] < round) {
                    hm |= 1u << c;
                    if (load[v] >= M) atomicMax(&bigk[blk[v]], big_key(v));
                }
            }
        }
        if (!__any_sync(FULL, hm != 0)) break;
        __syncwarp();
        for (int c = 0; c < NC; c++) {
            const int v = 32 * c + lane;
            if (!((hm >> c) & 1u)) continue;
            const unsigned long long bg = bigk[blk[v]];
            if (bg == 0 || (uint32_t)(bg & 0xffffu) == 0xffffu - rank[v]) {
                rnd[v] = (uint16_t)round;
                nround[blk[v]] = (uint16_t)(round + 1);
            }
        }
        __syncwarp();
        for (int c = 0; c < NC; c++)
            if ((hm >> c) & 1u) bigk[blk[32 * c + lane]] = 0;
        __syncwarp();
    }

    // ---- group index = groups of earlier blocks + round within the block
    uint32_t G = 0;
    for (int b0 = 0; b0 <= N; b0 += 32) {
        const int b = b0 + lane;
        const uint32_t n = b <= N && b < V ? nround[b] : 0u;
        uint32_t x = n;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        if (b <= N && b < V) fcnt[b] = G + x - n;
        G += __shfl_sync(FULL, x, 31);
    }
    __syncwarp();
    // ---- member lists of each group, ordered by id, as ranks: nodes are met in id order, so a
    //      node's place in its group is the group's count so far and the lanes before it
    for (int g = lane; g < V; g += 32) nround[g] = 0;  // now the members counted, by group
    for (int v = lane; v < V; v += 32) group_of[v] = (uint8_t)(fcnt[blk[v]] + rnd[v]);
    __syncwarp();
    for (int c = 0; c < NC; c++) {
        const int v = 32 * c + lane;
        const uint32_t g = v < V ? group_of[v] : 0x100u;
        const uint32_t same = __match_any_sync(FULL, g);
        uint32_t at = 0;
        if (v < V) at = nround[g];
        __syncwarp();
        if (v < V) {
            rnd[v] = (uint16_t)(at + __popc(same & lt));
            if ((same & lt) == 0) nround[g] = (uint16_t)(at + __popc(same));
        }
        __syncwarp();
    }
    uint32_t off = 0;
    for (int g0 = 0; g0 < (int)G; g0 += 32) {
        const int g = g0 + lane;
        const uint32_t n = g < (int)G ? nround[g] : 0u;
        uint32_t x = n;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        if (g < (int)G) gstart[g] = (uint16_t)(off + x - n);
        off += __shfl_sync(FULL, x, 31);
    }
    if (lane == 0) gstart[G] = (uint16_t)V;
    __syncwarp();
    for (int v = lane; v < V; v += 32) gmem[gstart[group_of[v]] + rnd[v]] = rank[v];
    __syncwarp();

    // ---- Alg.2's records (they overlay Alg.1's arrays)
    A2<true, uint8_t> w2;
    w2.base = nullptr;
    w2.o_rc = base + ws.rc;
    w2.o_col = base + ws.scol;
    w2.o_cnt = base + ws.acnt;
    w2.o_gstart = base + ws.gstart;
    w2.o_gmem = base + ws.gmem;
    w2.o_byrank = base + ws.byrank;
    w2.o_lst = base + ws.lst;
    w2.o_mm = base + ws.mm;
    w2.o_rel = base + ws.rel;
    w2.o_sum = 0;
    if (lane < 8) w2.rel()[lane] = 0;
    __syncwarp();
    const bool want_base = a.o.greedy || a.o.greedy_unaware || a.o.graham_para;
    uint64_t b_greedy = 0, b_unaware = 0;  // baseline sums (Evaluation section)
    for (int v = lane; v < V; v += 32) {
        const uint32_t x = load[v], k = kk[v], r = rank[v];
        const uint32_t cf = (uint32_t)exec_time(x, k, x < M ? x : M, M);
        if (want_base) {
            b_greedy += cf;
            b_unaware = sat_add(b_unaware, exec_time_unaware(x, k, M));
        }
        w2.rc(r) = make_uint4(x, cf, srp[v], (uint32_t)(srp[v + 1] - srp[v]) | (k << 16));
        w2.cnt(r) = indeg[v];
        if (indeg[v] == 0) atomicOr(w2.rel() + (r >> 5), 1u << (r & 31));
        if (a.o.block_of) a.o.block_of[n0 + v] = blk[v];
        if (a.o.group_of) a.o.group_of[n0 + v] = group_of[v];
    }
    for (int e = lane; e < E; e += 32) scol[e] = rank[scol[e]];
    if (want_base)
        for (int o = 16; o > 0; o >>= 1) {
            b_greedy += __shfl_xor_sync(FULL, b_greedy, o);
            b_unaware = sat_add(b_unaware, __shfl_xor_sync(FULL, b_unaware, o));
        }
    __syncwarp();
    Dag g;
    g.n0 = n0;
    g.rbase = 2 * n0;
    g.V = V;
    g.W = (V + 63) >> 6;
    g.M = M;
    g.variant = a.variant;
    g.want_edges = a.o.extra_off != nullptr;
    g.ebase = g.want_edges ? a.o.extra_off[d] : 0;
    g.ecap = g.want_edges ? a.o.extra_off[d + 1] - g.ebase : 0;
    Acc acc;
    acc.nrel = nsrc;
    if (64ull * M * mx < (1ull << 32)) alg2_warp<false, true, FULL_OUT>(w2, a, g, (int)G, acc, lane);
    else alg2_warp<false, false, FULL_OUT>(w2, a, g, (int)G, acc, lane);
    if (lane == 0) write_totals(a, g, d, acc, Totals{mx, b_greedy, b_unaware, vol, (int)G, nlev});
    if (!a.o.crit_path) return;

    // ---- critical-path lower bound: the longest chain of the schedule's parts in G (a node's
    //      parts run one after another, every edge waits for its tail's last part), or the work
    //      bound ceil(sum m C / M). Edges lead to smaller ranks: nodes in descending rank.
    uint64_t cp = 0;
    if (a.plan) {
        uint64_t *cpT = (uint64_t *)(smem + base + ws.cpT), *cpM = (uint64_t *)(smem + base + ws.cpM);
        __syncwarp();
        for (int r = lane; r < V; r += 32) cpT[r] = cpM[r] = 0;
        __threadfence_block();  // the plan rows written by other lanes
        __syncwarp();
        uint64_t work = 0;
        for (int r = lane; r < acc.nrows; r += 32) {
            const uint4 x = a.plan[g.rbase + r];
            atomicAdd((unsigned long long *)&cpT[rank[x.w]], (unsigned long long)x.y);
            work += (uint64_t)(x.z & 0xffffu) * x.y;
        }
        for (int o = 16; o > 0; o >>= 1) work += __shfl_xor_sync(FULL, work, o);
        __syncwarp();
        for (int r = V - 1; r >= 0; r--) {
            const uint64_t dv = cpT[r] + cpM[r];
            cp = dv > cp ? dv : cp;
            const uint32_t eb = w2.rc(r).z, deg = w2.rc(r).w & 0xffffu;
            for (uint32_t e = lane; e < deg; e += 32) {
                const uint32_t s = w2.col(eb + e);
                if (dv > cpM[s]) cpM[s] = dv;
            }
            __syncwarp();
        }
        const uint64_t wb = (work + M - 1) / M;
        cp = cp > wb ? cp : wb;
    }
    if (lane == 0) write_crit_path(a, g, d, acc, cp);
}

}  // namespace dagrt
