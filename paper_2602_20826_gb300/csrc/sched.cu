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
#include <utility>

#include "alg2.cuh"
#include "dagrt_internal.cuh"
#include "sched.cuh"
#include "sched_warp.cuh"

namespace dagrt {

constexpr uint16_t NONE16 = 0xffff;
constexpr int kRelWords = (DAGRT_MAX_V + 63) / 64;  // words of the largest released-set mask
constexpr int kRelBytes = 8 * (kRelWords + kRelWords / 64);  // ... and of its summary
// dynamic shared memory of teams with a global workspace: the released set and the bit planes
// of the loads while they fit
constexpr int kPlaneWords = 4096;
constexpr int kGlobalSmem = kRelBytes + 8 * kPlaneWords;
constexpr int kSumWords = 16;  // released-set masks longer than this keep a summary of non-empty words

// ------------------------------------------------------------------ workspace layout
// Persistent arrays live for the whole DAG; the region after them is overlaid by the
// arrays of one phase at a time (A closure, B ordering, C peeling, D member lists, E Alg.2).
struct Ws {
    // persistent
    uint32_t *load;
    uint8_t *kk;
    int32_t *cnt;  // atomic counters: in-degree, Kahn count, open preds
    uint32_t *srp;  // the DAG's successor CSR, staged: offsets ...
    uint16_t *scol; // ... and successor ids
    uint16_t *indeg, *lvl_off, *topo, *rank, *byrank, *blk, *group_of, *gstart, *gmem;
    uint64_t *relmask;
    uint64_t *relsum;  // bit w: relmask[w] may be non-zero (cleared lazily by the scan)
    // phases A and B
    uint64_t *wanc;  // W^anc, then the sort keys in its place
    uint64_t *anc;   // shared memory: word w of node v at w * V + v, kept until the blocks are read off it
    uint64_t *planes;
    int32_t *poff;  // global workspaces: predecessor lists by node (inclusive offsets) ...
    uint16_t *pid;  // ... and their entries
    // phase B
    uint16_t *bk, *pos, *jcnt, *rs, *re;
    // phase C (Alg.1): groups of each block, nodes by block, blocks of two nodes or more, and
    // per node its round and its in-block predecessor (itself: none)
    int32_t *nround, *boff;
    uint16_t *bnode, *blist, *rnd, *par;
    uint32_t *tC;  // per warp: loads and ranks of Top_M, and the block's other heads by rank
    uint16_t *tR;
    uint64_t *hmask;
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

// Top_M and one batch of a selected node's successors
__host__ __device__ inline int top_cap(int vc) { return (vc < DAGRT_MAX_M ? vc : DAGRT_MAX_M) + 32; }

// Carve a workspace for DAGs of up to vc nodes and ec edges out of `base`; returns the
// bytes used. `sh`: for a team of kCtaThreads in shared memory, else kCtaThreadsGlobal.
__host__ __device__ inline int64_t ws_carve(unsigned char *base, int vc, int ec, Ws *ws, bool sh) {
    const int W = ceil_div(vc, 64) > 0 ? ceil_div(vc, 64) : 1;
    const int P = pow2_ceil(vc > 0 ? vc : 1);
    const int warps = (sh ? kCtaThreads : kCtaThreadsGlobal) / 32;
    int64_t off = 0;
    auto take = [&](int64_t bytes) {
        unsigned char *p = base + off;
        off = align_up(off + bytes, 16);
        return p;
    };
    Ws w;
    w.load = (uint32_t *)take(4ll * vc);
    w.kk = (uint8_t *)take(vc);
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
    const int64_t x0 = off;
    int64_t end = off;
    auto mark = [&]() { end = off > end ? off : end; };
    w.wanc = (uint64_t *)take(8ll * P);
    const int64_t xa = off;
    w.anc = (uint64_t *)take(8ll * vc * W);
    const int64_t xb = off;
    w.planes = (uint64_t *)take(8ll * 32 * W);
    w.poff = sh ? nullptr : (int32_t *)take(4ll * (vc + 1));
    w.pid = sh ? nullptr : (uint16_t *)take(2ll * (ec > 0 ? ec : 1));
    mark();
    off = sh ? xb : xa;
    w.jcnt = (uint16_t *)take(2ll * vc);
    w.rs = (uint16_t *)take(2ll * vc);
    w.re = (uint16_t *)take(2ll * vc);
    w.bk = w.rs;  // (the runs are read before the blocks are computed)
    w.pos = w.re;
    mark();
    off = x0;
    w.nround = (int32_t *)take(4ll * (vc + 1));
    w.boff = (int32_t *)take(4ll * (vc + 2));
    w.bnode = (uint16_t *)take(2ll * vc);
    w.blist = (uint16_t *)take(2ll * vc);
    w.rnd = (uint16_t *)take(2ll * vc);
    w.par = (uint16_t *)take(2ll * vc);
    w.tC = (uint32_t *)take(4ll * top_cap(vc) * warps);
    w.tR = (uint16_t *)take(2ll * top_cap(vc) * warps);
    w.hmask = (uint64_t *)take(8ll * W * warps);
    mark();
    off = align_up(x0 + 4ll * (vc + 1), 16);  // nround is still read
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

int64_t sched_ws_bytes(int vc, int ec) { return ws_carve(nullptr, vc, ec, nullptr, false); }
int64_t sched_smem_ws_bytes(int vc, int ec) { return ws_carve(nullptr, vc, ec, nullptr, true); }

// ------------------------------------------------------------------ Alg.1, one block
// One warp peels the out-forest of a block of n >= 2 nodes: a round takes Top_M of its heads
// by W^anc (Rule 1), or the head among them with the largest C^ >= M alone (Rule 2). Sets the
// nodes' rounds and returns their number.
//
// A successor has a larger W^anc than its predecessor, so a smaller rank: the successors of a
// selected node belong to the new Top_M. So Top_M is kept as a list (tC, tR: load and rank),
// the heads behind it as a bit mask over ranks whose lowest bits are the next to move up, and
// a round costs a pass over at most M entries, however many heads the block has. Rounds over
// all heads of all blocks cost 39,000 cycles each on 10,000-node layered DAGs, of which there
// are 900; this one 3,500 with Top_M of 148. Blocks of at most 32 nodes (most of them) keep a node per lane.
__device__ int peel_block(const Ws &ws, uint32_t M, int b, int n, uint32_t *tC, uint16_t *tR, uint64_t *mask, int W,
                          int *wcnt, int lane) {
    const uint16_t *node = ws.bnode + ws.boff[b];
    const uint32_t *__restrict__ rp = ws.srp;
    if (n <= 32 && n <= (int)M) {  // every head is in Top_M
        const int v = lane < n ? node[lane] : 0;
        const uint32_t x = lane < n ? ws.load[v] : 0u, r = lane < n ? ws.rank[v] : 0u;
        const int p = lane < n ? ws.par[v] : -1;
        bool head = lane < n && p == v, open = lane < n;  // open: not selected yet
        int round = 0;
        for (; __any_sync(FULL, open); round++) {
            const uint32_t big = __reduce_max_sync(FULL, head && x >= M ? x : 0u);
            bool sel = head;
            if (big) {
                const uint32_t lo = __reduce_min_sync(FULL, head && x == big ? r : ~0u);
                sel = head && x == big && r == lo;
            }
            if (sel) {
                ws.rnd[v] = (uint16_t)round;
                head = open = false;
            }
            __syncwarp();
            if (open && !head) head = ws.rnd[p] != NONE16;
        }
        return round;
    }
    for (int w = lane; w < W; w += 32) mask[w] = 0;
    __syncwarp();
    for (int i = lane; i < n; i += 32) {  // the first heads
        const int v = node[i];
        if (ws.par[v] == v) atomicOr((uint32_t *)mask + (ws.rank[v] >> 5), 1u << (ws.rank[v] & 31));
    }
    __syncwarp();
    int cnt = 0, cur = 0, round = 0;  // entries of Top_M, first mask word that may have bits, round
    auto refill = [&]() {             // the lowest heads of the mask move up
        while (cnt < (int)M && cur < W) {
            const uint64_t x = cur + lane < W ? mask[cur + lane] : 0ull;
            const uint32_t any = __ballot_sync(FULL, x != 0);
            if (!any) {
                cur += 32;
                continue;
            }
            const int l = __ffs(any) - 1;
            cur += l;
            const uint64_t bits = __shfl_sync(FULL, x, l);
            const int room = (int)M - cnt, have = __popcll(bits);
#pragma unroll
            for (int h = 0; h < 2; h++) {  // this lane's two bits of the word
                const int bit = lane + 32 * h;
                const int at = __popcll(bits & ((1ull << bit) - 1));
                if ((bits >> bit & 1ull) && at < room) {
                    const int r = cur * 64 + bit;
                    tC[cnt + at] = ws.load[ws.byrank[r]];
                    tR[cnt + at] = (uint16_t)r;
                }
            }
            uint64_t rest = 0;
            if (have > room) {  // keep the highest have - room bits
                rest = bits;
                for (int i = 0; i < room; i++) rest &= rest - 1;
            }
            if (lane == 0) mask[cur] = rest;
            cnt += min(have, room);
            __syncwarp();
        }
    };
    refill();
    while (cnt > 0) {
        // the largest load of at least M, then the lowest rank
        uint32_t bc = 0, br = 0xffffffffu;
        int bi = 0;
        for (int i = lane; i < cnt; i += 32) {
            const uint32_t c = tC[i], r = tR[i];
            if (c >= M && (c > bc || (c == bc && r < br))) {
                bc = c;
                br = r;
                bi = i;
            }
        }
        const uint32_t mc = __reduce_max_sync(FULL, bc);
        if (mc) {  // it runs alone; its in-block successors take part in the next round
            const uint32_t mr = __reduce_min_sync(FULL, bc == mc ? br : 0xffffffffu);
            const int at = __shfl_sync(FULL, bi, __ffs(__ballot_sync(FULL, bc == mc && br == mr)) - 1);
            const int v = ws.byrank[mr];
            const int eb = (int)rp[v], end = (int)rp[v + 1];
            const uint32_t lc = tC[cnt - 1], lr = tR[cnt - 1];
            __syncwarp();
            if (lane == 0) {
                ws.rnd[v] = (uint16_t)round;
                tC[at] = lc;
                tR[at] = (uint16_t)lr;
            }
            cnt--;
            __syncwarp();
            for (int e0 = eb; e0 < end; e0 += 32) {
                const int s = e0 + lane < end ? ws.scol[e0 + lane] : -1;
                const bool kid = s >= 0 && ws.par[s] == v && ws.blk[s] == b;
                const uint32_t kb = __ballot_sync(FULL, kid);
                if (kid) {
                    const int i = cnt + __popc(kb & ((1u << lane) - 1));
                    tC[i] = ws.load[s];
                    tR[i] = ws.rank[s];
                }
                cnt += __popc(kb);
                __syncwarp();
                while (cnt > (int)M) {  // the largest rank goes back behind Top_M
                    uint32_t hr = 0;
                    int hi = 0;
                    for (int i = lane; i < cnt; i += 32)
                        if ((uint32_t)tR[i] + 1u > hr) {
                            hr = (uint32_t)tR[i] + 1u;
                            hi = i;
                        }
                    const uint32_t mx = __reduce_max_sync(FULL, hr);
                    const int o = __shfl_sync(FULL, hi, __ffs(__ballot_sync(FULL, hr == mx)) - 1);
                    const uint32_t c1 = tC[cnt - 1], r1 = tR[cnt - 1];
                    __syncwarp();
                    if (lane == 0) {
                        mask[(mx - 1) >> 6] |= 1ull << ((mx - 1) & 63);
                        tC[o] = c1;
                        tR[o] = (uint16_t)r1;
                    }
                    cur = min(cur, (int)((mx - 1) >> 6));
                    cnt--;
                    __syncwarp();
                }
            }
        } else {  // all of Top_M; the successors join the heads, the lowest move up
            if (lane == 0) *wcnt = 0x7fffffff;
            __syncwarp();
            for (int i = lane; i < cnt; i += 32) {
                const int v = ws.byrank[tR[i]];
                ws.rnd[v] = (uint16_t)round;
                for (int e = (int)rp[v]; e < (int)rp[v + 1]; e++) {
                    const int s = ws.scol[e];
                    if (ws.par[s] != v || ws.blk[s] != b) continue;
                    const uint32_t r = ws.rank[s];
                    atomicOr((uint32_t *)mask + (r >> 5), 1u << (r & 31));
                    atomicMin(wcnt, (int)(r >> 6));
                }
            }
            __syncwarp();
            cur = min(cur, *wcnt);
            cnt = 0;
        }
        refill();
        round++;
    }
    return round;
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
    __shared__ int32_t sc_s[16];  // counters of the team
    volatile int32_t *sc = sc_s;
    const bool lead = tm.t == 0;
    extern __shared__ __align__(16) unsigned char dyn[];

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
    bool order = true;  // every edge leads to a larger id
    tm.sync();
    const uint32_t *__restrict__ rp = ws.srp;
    const uint16_t *__restrict__ col = ws.scol;
    if (!badc) {  // self loops, unsorted or repeated successors (ids are in range here)
        for (int v = tm.t; v < V; v += NT) {
            int prev = -1;
            for (int e = rp[v]; e < (int)rp[v + 1]; e++) {
                const int c = col[e];
                if (c == v || c <= prev) badc = true;
                order &= c > v;
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
        if (lead) write_empty(a, d);
        return;
    }
    tm.sync();

    // ---- in-degrees (a join has at least two predecessors), one edge per thread
    for (int e = tm.t; e < (int)E; e += NT) atomicAdd(&ws.cnt[col[e]], 1);
    const int W = (V + 63) >> 6;
    if (lead) sc[0] = 0;
    tm.sync();

    for (int v = tm.t; v < V; v += NT) {
        const int dg = ws.cnt[v];
        ws.indeg[v] = (uint16_t)dg;
        if (dg == 0) ws.topo[atomicAdd((int *)&sc[0], 1)] = (uint16_t)v;
    }
    int nlev = 0;
    uint64_t mx = 0;
    for (int v = tm.t; v < V; v += NT) mx = mx > ws.load[v] ? mx : ws.load[v];
    mx = tm.maxu(mx);  // (and a barrier)
    const int nb = 64 - __clzll((long long)mx);
    if constexpr (SH) {
        // ---- Shared memory: levels by one warp, node by node in topological order -- the ids,
        //      where every edge leads to a larger one, else Kahn's queue; nodes without successors
        //      are left out (1,000 isolated ones waited for 1,000 steps). Then (with the ids as
        //      order: meanwhile) the closure: its 64-bit columns are independent, so every warp
        //      carries its own columns through all nodes, a lane per successor (they are
        //      distinct: no atomics), without a barrier between levels. Column by column in
        //      memory, so that the successors' words spread over the banks (row by row, 25
        //      successors of a 1,000-node DAG met in one bank: 1,160 instead of 660 cycles a node).
        const int lane = tm.lane(), wp = tm.warp(), NWP = NT / 32;
        const bool ids = !tm.any(!order);
        for (int w = 0; w < W; w++)
            for (int v = tm.t; v < V; v += NT) ws.anc[w * V + v] = v >> 6 == w ? 1ull << (v & 63) : 0ull;
        if (ids)
            for (int v = tm.t; v < V; v += NT) ws.lvl_off[v] = 0;  // levels, until they are written out
        uint16_t *list = ws.byrank;  // the nodes with successors, in topological order
        auto collect = [&](auto ith) {  // one warp; their number in sc[4]
            int n = 0;
            for (int i0 = 0; i0 < V; i0 += 32) {
                const int u = i0 + lane < V ? ith(i0 + lane) : 0;
                const bool has = i0 + lane < V && rp[u + 1] > rp[u];
                const uint32_t hb = __ballot_sync(FULL, has);
                if (has) list[n + __popc(hb & ((1u << lane) - 1))] = (uint16_t)u;
                n += __popc(hb);
            }
            if (lane == 0) sc[4] = n;
        };
        if (ids && wp == 0) collect([](int i) { return i; });
        tm.sync();
        const int cw = (W + NWP - 1) / NWP;
        int w0 = min(W, wp * cw);  // this warp's columns, w0 .. w1 - 1
        const int w1 = min(W, w0 + cw);
        if (!ids) {
            if (wp == 0) {
                int head = 0, tail = sc[0], lend = tail, L = 0;
                for (int i = lane; i < tail; i += 32)
                    if (a.o.level) a.o.level[n0 + ws.topo[i]] = 0;
                while (head < tail) {
                    if (head == lend) {
                        L++;
                        lend = tail;
                    }
                    const int u = ws.topo[head++];
                    const int end = (int)rp[u + 1];
                    for (int e0 = (int)rp[u]; e0 < end; e0 += 32) {
                        int s = 0, c = 1;
                        if (e0 + lane < end) {
                            s = col[e0 + lane];
                            c = ws.cnt[s] - 1;
                            ws.cnt[s] = c;
                        }
                        const uint32_t zb = __ballot_sync(FULL, c == 0);
                        if (c == 0) {
                            ws.topo[tail + __popc(zb & ((1u << lane) - 1))] = (uint16_t)s;
                            if (a.o.level) a.o.level[n0 + s] = L + 1;
                        }
                        tail += __popc(zb);
                    }
                    __syncwarp();
                }
                if (lane == 0) sc[1] = tail == V ? L + 1 : 0;
                if (tail == V) collect([&](int i) { return (int)ws.topo[i]; });
            }
            tm.sync();
            nlev = sc[1];
            if (nlev == 0) {
                if (lead) write_failure(a, d, DAGRT_E_CYCLE);
                return;
            }
        }
        uint16_t *lev = ws.lvl_off;
        const int nlist = sc[4];
        // the warp's columns w0 .. w0 + CW - 1 of the closure. A node takes one load's latency:
        // its edges' bounds are loaded two nodes ahead, its first 32 successors one node ahead,
        // and all rows before any is stored (440 -> 300 cycles a node at 500 nodes)
        auto columns = [&](auto cwc, auto lvc) {
            constexpr int CW = decltype(cwc)::value;
            constexpr bool LV = decltype(lvc)::value;
            auto node = [&](int i) { return (int)list[min(i, nlist - 1)]; };
            uint64_t *anc = ws.anc + w0 * V;
            if (nlist == 0) return;
            int u = node(0), u1 = node(1);
            int eb = (int)rp[u], end = (int)rp[u + 1], eb1 = (int)rp[u1], end1 = (int)rp[u1 + 1];
            int s = eb + lane < end ? col[eb + lane] : 0;
            for (int i = 0; i < nlist; i++) {
                const int u2 = node(i + 2);
                const int eb2 = (int)rp[u2], end2 = (int)rp[u2 + 1];
                const int s1 = eb1 + lane < end1 ? col[eb1 + lane] : 0;
                uint64_t row[CW > 0 ? CW : 1];
#pragma unroll
                for (int c = 0; c < CW; c++) row[c] = anc[c * V + u];
                uint32_t l = 0;
                if constexpr (LV) l = lev[u] + 1u;
                for (int e = eb; e < end; e += 32) {
                    if (e > eb && e + lane < end) s = col[e + lane];
                    if (e + lane < end) {
                        uint64_t x[CW > 0 ? CW : 1];
                        uint32_t ls = 0;
#pragma unroll
                        for (int c = 0; c < CW; c++) x[c] = anc[c * V + s];
                        if constexpr (LV) ls = lev[s];
#pragma unroll
                        for (int c = 0; c < CW; c++) anc[c * V + s] = x[c] | row[c];
                        if constexpr (LV) lev[s] = (uint16_t)max(ls, l);
                    }
                }
                __syncwarp();
                u = u1;
                u1 = u2;
                eb = eb1;
                end = end1;
                eb1 = eb2;
                end1 = end2;
                s = s1;
            }
        };
        // (every warp has cw columns but for the last ones; the last warp also pushes levels)
        const bool levels = ids && wp == NWP - 1;
        for (int c = w1 - w0, at = w0;; ) {
            w0 = at;
            const int n = min(c, 4);
            auto with = [&](auto lvc) {
                if (n == 4) columns(std::integral_constant<int, 4>(), lvc);
                else if (n == 3) columns(std::integral_constant<int, 3>(), lvc);
                else if (n == 2) columns(std::integral_constant<int, 2>(), lvc);
                else if (n == 1) columns(std::integral_constant<int, 1>(), lvc);
                else if constexpr (decltype(lvc)::value) columns(std::integral_constant<int, 0>(), lvc);
            };
            if (levels && at + n == w1) with(std::true_type());
            else with(std::false_type());
            c -= n;
            at += n;
            if (c == 0) break;
        }
        if (ids) {
            tm.sync();
            uint64_t top = 0;
            for (int v = tm.t; v < V; v += NT) {
                top = max(top, (uint64_t)lev[v]);
                if (a.o.level) a.o.level[n0 + v] = lev[v];
                ws.topo[v] = (uint16_t)v;
            }
            nlev = (int)tm.maxu(top) + 1;
        }
        tm.sync();
        // ---- Eq.2: W^anc(v) = sum of C^ over v and its ancestors, by bit planes of C^
        for (int i = tm.t; i < nb * W; i += NT) {
            const int b = i / W, w = i - b * W;
            const int vb = w * 64, ve = min(V, vb + 64);
            uint64_t word = 0;
            for (int v = vb; v < ve; v++) word |= (uint64_t)((ws.load[v] >> b) & 1u) << (v - vb);
            ws.planes[i] = word;
        }
        tm.sync();
        for (int v = tm.t; v < V; v += NT) {
            uint64_t acc = 0;
            for (int w = 0; w < W; w++) {
                const uint64_t x = ws.anc[w * V + v];
                for (int b = 0; b < nb; b++) acc += (uint64_t)__popcll(x & ws.planes[b * W + w]) << b;
            }
            ws.wanc[v] = acc;
            ws.anc[(v >> 6) * V + v] &= ~(1ull << (v & 63));  // the blocks are about other nodes
            if (a.o.wanc) a.o.wanc[n0 + v] = (int64_t)acc;
        }
    } else {
    // ---- Global memory: Kahn levels by the whole team
    const int n_src = sc[0];
    for (int i = tm.t; a.o.level && i < n_src; i += NT) a.o.level[n0 + ws.topo[i]] = 0;
    tm.sync();  // read by everyone before it moves on
    int ls = 0, le = n_src, L = 0;
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
    nlev = L;
    if (le != V) {
        if (lead) write_failure(a, d, DAGRT_E_CYCLE);
        return;
    }

    // ---- ... then the ancestor closure and Eq.2 level by level, a warp per node: the rows of
    //      the predecessors and the predecessors themselves, 64-bit words over the lanes, and
    //      W^anc as one predecessor's plus the loads of the ancestors that only others have, by
    //      bit planes of C^ (in shared memory while they fit). Most words add nothing: counting
    //      the bits of every word took 19.3 M cycles at 20,000 nodes, this takes 17.4 M.
    uint64_t *planes = nb * W <= kPlaneWords ? (uint64_t *)(dyn + kRelBytes) : ws.planes;
    for (int i = tm.t; i < nb * W; i += NT) {
        const int b = i / W, w = i - b * W;
        const int vb = w * 64, ve = min(V, vb + 64);
        uint64_t word = 0;
        for (int v = vb; v < ve; v++) word |= (uint64_t)((ws.load[v] >> b) & 1u) << (v - vb);
        planes[i] = word;
    }
    for (int v = tm.t; v < V; v += NT) ws.poff[v] = ws.indeg[v];
    tm.sync();
    team_scan_inplace(tm, ws.poff, V, [](uint64_t x, uint64_t y) { return x + y; }, false);
    for (int u = tm.t; u < V; u += NT)  // ws.cnt is zero again after Kahn's pass
        for (int e = rp[u]; e < (int)rp[u + 1]; e++) {
            const int s = col[e];
            ws.pid[ws.poff[s] - ws.indeg[s] + atomicAdd(&ws.cnt[s], 1)] = (uint16_t)u;
        }
    tm.sync();
    // the bits of word w of a row that `planes` weigh
    auto weigh = [&](uint64_t x, int w) {
        uint64_t s = 0;
        if (nb <= 24) {  // 64 * 2^24 fits: the word's sum in 32 bits
            uint32_t t = 0;
            for (int b = 0; b < nb; b++) t += (uint32_t)__popcll(x & planes[b * W + w]) << b;
            s = t;
        } else {
            for (int b = 0; b < nb; b++) s += (uint64_t)__popcll(x & planes[b * W + w]) << b;
        }
        return s;
    };
    // Rows of up to 32 words (2,048 nodes), and any node of more than 16 predecessors: what takes
    // the time is the latency of their rows, so a warp reads 32 / LW rows at once, one or two words
    // per lane, and eight deep. (Dense graphs, whose levels are narrow: 100 DAGs of 300-900 nodes with
    // 35% of the edges 10 ms, 10 of 1,500-2,500 with 30% 81; with the rows one after another 18
    // and 121.)
    const int LW = W <= 4 ? 4 : W <= 8 ? 8 : W <= 16 ? 16 : 32;
    auto store_wanc = [&](int v, uint64_t w) {
        if (tm.lane() == 0) {
            ws.wanc[v] = w;
            if (a.o.wanc) a.o.wanc[n0 + v] = (int64_t)w;
        }
    };
    auto wide = [&](auto twoc, int v, int pb, int np) {
        constexpr bool TWO = decltype(twoc)::value;  // rows of more than 32 words
        const int ln = tm.lane(), step = 32 / LW;
        uint64_t acc = 0;
        for (int c = 0; c < W; c += 64) {
            const int wi = c + (ln & (LW - 1)), w2 = c + 32 + ln;
            uint64_t x = 0, x2 = 0;
            for (int k0 = ln / LW; k0 < np; k0 += 8 * step) {
                int p[8];
                uint64_t z[8], z2[8];
#pragma unroll
                for (int j = 0; j < 8; j++) p[j] = k0 + j * step < np ? (int)ws.pid[pb + k0 + j * step] : -1;
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    z[j] = p[j] >= 0 && wi < W ? ws.anc[(int64_t)p[j] * W + wi] : 0ull;
                    if constexpr (TWO) z2[j] = p[j] >= 0 && w2 < W ? ws.anc[(int64_t)p[j] * W + w2] : 0ull;
                }
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    x |= z[j] | (p[j] >= 0 && wi == p[j] >> 6 ? 1ull << (p[j] & 63) : 0ull);
                    if constexpr (TWO) x2 |= z2[j] | (p[j] >= 0 && w2 == p[j] >> 6 ? 1ull << (p[j] & 63) : 0ull);
                }
            }
            __syncwarp();
            for (int o = LW; o < 32; o <<= 1) x |= __shfl_xor_sync(FULL, x, o);
            if (c + ln < W) {  // (LW < 32: the lanes of the first row)
                ws.anc[(int64_t)v * W + c + ln] = x;
                acc += weigh(x, c + ln);
            }
            if (TWO && w2 < W) {
                ws.anc[(int64_t)v * W + w2] = x2;
                acc += weigh(x2, w2);
            }
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
        store_wanc(v, acc + ws.load[v]);
    };
    for (int l = 0; l < nlev; l++) {
        const int lb = ws.lvl_off[l], lend = (l + 1 < nlev) ? ws.lvl_off[l + 1] : V;
        const int ln = tm.lane(), stride = NT / 32;
        if (W <= 32) {
            for (int i = lb + tm.warp(); i < lend; i += stride) {
                const int v = ws.topo[i], np = ws.indeg[v];
                wide(std::false_type(), v, ws.poff[v] - np, np);
            }
            tm.sync();
            continue;
        }
        for (int i0 = lb + tm.warp(); i0 < lend; i0 += 32 * stride) {
            // the warp's next 32 nodes, one per lane; their predecessor lists are fetched two
            // nodes ahead and the predecessors' W^anc one node ahead
            const int mine = i0 + ln * stride, nq = min(32, (lend - i0 + stride - 1) / stride);
            const int vq = mine < lend ? ws.topo[mine] : 0;
            const int peq = mine < lend ? ws.poff[vq] : 0, npq = mine < lend ? ws.indeg[vq] : 0;
            auto preds = [&](int q) {  // the q-th node's first 32 predecessors, one per lane
                const int n = __shfl_sync(FULL, npq, q), b = __shfl_sync(FULL, peq, q) - n;
                return q < nq && ln < n ? (int)ws.pid[b + ln] : -1;
            };
            auto weight = [&](int p) { return p >= 0 ? ws.wanc[p] : 0ull; };
            int p0 = preds(0), p1 = preds(1);
            uint64_t w0 = weight(p0);
            for (int q = 0; q < nq; q++) {
                const int v = __shfl_sync(FULL, vq, q), np = __shfl_sync(FULL, npq, q);
                const int pb = __shfl_sync(FULL, peq, q) - np;
                const int p2 = preds(min(q + 2, 31));
                const uint64_t w1 = weight(p1);
                if (np > 16) {
                    wide(std::true_type(), v, pb, np);
                    p0 = p1;
                    p1 = p2;
                    w0 = w1;
                    continue;
                }
                // the predecessor of largest W^anc (about: any would do) and two others
                const uint32_t key = p0 >= 0 ? __float_as_uint((float)w0) : 0u;
                const int kb = __ffs(__ballot_sync(FULL, key == __reduce_max_sync(FULL, key))) - 1;
                uint32_t rest = ((1u << np) - 1u) & ~(1u << kb);
                const int pa = __shfl_sync(FULL, p0, kb);
                const int pc = __shfl_sync(FULL, p0, (__ffs(rest) - 1) & 31);
                rest &= rest - 1;
                const int pd = __shfl_sync(FULL, p0, (__ffs(rest) - 1) & 31);
                rest &= rest - 1;
                uint64_t acc = 0;
                for (int c = 0; c < W; c += 4 * 32) {  // four words of three rows per lane in flight
                    uint64_t x0[4] = {0, 0, 0, 0}, x[4] = {0, 0, 0, 0}, y[4] = {0, 0, 0, 0};
                    auto load = [&](uint64_t(&r)[4], int p) {
                        const uint64_t *row = ws.anc + (int64_t)p * W;
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            if (c + 32 * j + ln < W) r[j] = row[c + 32 * j + ln];
                    };
                    auto self = [&](uint64_t(&r)[4], int p) {
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            if (c + 32 * j + ln == p >> 6) r[j] |= 1ull << (p & 63);
                    };
                    if (np > 0) load(x0, pa);
                    if (np > 1) load(x, pc);
                    if (np > 2) load(y, pd);
                    if (np > 0) self(x0, pa);
                    if (np > 1) self(x, pc);
                    if (np > 2) self(y, pd);
                    uint32_t more = rest;
                    auto other = [&]() {
                        const int p = __shfl_sync(FULL, p0, (__ffs(more) - 1) & 31);
                        more &= more - 1;
                        return p;
                    };
                    for (int k = 3; k < np; k += 2) {
                        uint64_t z[4] = {0, 0, 0, 0}, z2[4] = {0, 0, 0, 0};
                        const int p = other(), p3 = k + 1 < np ? other() : -1;
                        load(z, p);
                        if (p3 >= 0) load(z2, p3);
                        self(z, p);
                        if (p3 >= 0) self(z2, p3);
#pragma unroll
                        for (int j = 0; j < 4; j++) x[j] |= z[j] | z2[j];
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const int w = c + 32 * j + ln;
                        x[j] |= y[j];
                        if (w < W) ws.anc[(int64_t)v * W + w] = x0[j] | x[j];
                        const uint64_t add = x[j] & ~x0[j];  // zero beyond W
                        if (add) acc += weigh(add, w);
                    }
                }
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
                store_wanc(v, acc + ws.load[v] + __shfl_sync(FULL, w0, kb));  // (no predecessor: 0)
                p0 = p1;
                p1 = p2;
                w0 = w1;
            }
        }
        tm.sync();
    }
    }
    tm.sync();

    // ---- order nodes by (W^anc, id): Theta uses it ascending, Top_M and para(pi_j)
    //      descending with ties broken by lower id
    const int P = pow2_ceil(V);
    uint64_t *skey = ws.wanc;  // the keys take the weights' place
    for (int i = tm.t; i < P; i += NT) skey[i] = i < V ? ((ws.wanc[i] << 16) | (uint64_t)i) : KEY_INF;
    tm.sync();
    team_bitonic_sort(tm, skey, P, SH ? nullptr : (uint64_t *)(dyn + kRelBytes), SH ? 0 : kPlaneWords);
    // per sorted position: join flag (-> Theta index), start and end of its W^anc run
    for (int i = tm.t; i < V; i += NT) {
        const int v = (int)(skey[i] & 0xffff);
        const uint64_t wv = skey[i] >> 16;
        ws.jcnt[i] = ws.indeg[v] >= 2 ? 1 : 0;
        ws.rs[i] = (uint16_t)((i == 0 || (skey[i - 1] >> 16) != wv) ? i : 0);
        ws.re[i] = (uint16_t)((i == V - 1 || (skey[i + 1] >> 16) != wv) ? i : NONE16);
    }
    tm.sync();
    team_scan_inplace(tm, ws.jcnt, V, [](uint64_t x, uint64_t y) { return x + y; }, false);
    team_scan_inplace(tm, ws.rs, V, [](uint64_t x, uint64_t y) { return x > y ? x : y; }, false);
    team_scan_inplace(tm, ws.re, V, [](uint64_t x, uint64_t y) { return x < y ? x : y; }, true);
    const int N = ws.jcnt[V - 1];  // number of join nodes
    for (int i = tm.t; i < V; i += NT) {
        const int v = (int)(skey[i] & 0xffff);
        const int r = (V - 1 - ws.re[i]) + (i - ws.rs[i]);
        ws.rank[v] = (uint16_t)r;
        ws.byrank[r] = (uint16_t)v;
    }
    tm.sync();

    // ---- Eq.3 blocks: a node belongs to the first join (in Theta order) it is an ancestor of;
    //      no such join: the residual block N
    if constexpr (SH) {
        // read off the closure: a thread owns a node and takes the joins backwards, so the last
        // row with its bit is the first join's (the row's word is the same for a warp's nodes)
        uint16_t *joins = ws.rs;
        for (int i = tm.t; i < V; i += NT)
            if (ws.indeg[skey[i] & 0xffff] >= 2) joins[ws.jcnt[i] - 1] = (uint16_t)(skey[i] & 0xffff);
        tm.sync();
        for (int v = tm.t; v < V; v += NT) {
            const int w = v >> 6;
            const uint64_t bit = 1ull << (v & 63);
            int b = N;
#pragma unroll 4
            for (int t = N - 1; t >= 0; t--)
                if (ws.anc[w * V + joins[t]] & bit) b = t;
            ws.blk[v] = (uint16_t)b;
        }
    } else {
        // the smallest sorted position among the joins reachable, by a min over successors in
        // reverse level order
        for (int i = tm.t; i < V; i += NT) {
            const int v = (int)(skey[i] & 0xffff);
            ws.pos[v] = (uint16_t)i;
            ws.bk[v] = NONE16;
        }
        tm.sync();
        for (int l = nlev - 1; l >= 0; l--) {
            const int lb = ws.lvl_off[l], lend = (l + 1 < nlev) ? ws.lvl_off[l + 1] : V;
            for (int i = lb + tm.t; i < lend; i += NT) {
                const int v = ws.topo[i];
                int b = NONE16;
                for (int e = rp[v]; e < rp[v + 1]; e++) {
                    const int s = col[e];
                    if (ws.indeg[s] >= 2) b = min(b, (int)ws.pos[s]);
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
    }
    tm.sync();

    // ---- Alg.1: peel every block's out-forest, a warp per block (peel_block); a node has an
    //      in-block predecessor only if it has a single predecessor (a join's ancestors are in
    //      blocks up to its own, it is in a later one). Round r of block k becomes the group
    //      after block k's earlier rounds and after every group of blocks 0..k-1.
    for (int v = tm.t; v < V; v += NT) {
        ws.par[v] = (uint16_t)v;
        ws.rnd[v] = NONE16;
    }
    for (int b = tm.t; b <= N + 1; b += NT) ws.boff[b] = 0;
    for (int b = tm.t; b <= N; b += NT) ws.nround[b] = 0;
    if (lead) {
        sc[2] = 0;  // blocks of two nodes or more: listed, and taken
        sc[3] = 0;
    }
    tm.sync();
    for (int u = tm.t; u < V; u += NT) {
        const int b = ws.blk[u];
        atomicAdd(&ws.boff[b + 1], 1);
        for (int e = rp[u]; e < (int)rp[u + 1]; e++) {
            const int s = col[e];
            if (ws.indeg[s] == 1 && ws.blk[s] == b) ws.par[s] = (uint16_t)u;
        }
    }
    tm.sync();
    team_scan_inplace(tm, ws.boff, N + 2, [](uint64_t x, uint64_t y) { return x + y; }, false);
    for (int v = tm.t; v < V; v += NT) {  // nround counts the nodes placed so far
        const int b = ws.blk[v];
        ws.bnode[ws.boff[b] + atomicAdd(&ws.nround[b], 1)] = (uint16_t)v;
    }
    tm.sync();
    for (int b = tm.t; b <= N; b += NT) {
        const int n = ws.boff[b + 1] - ws.boff[b];
        ws.nround[b] = n ? 1 : 0;
        if (n == 1) ws.rnd[ws.bnode[ws.boff[b]]] = 0;
        if (n > 1) ws.blist[atomicAdd((int *)&sc[2], 1)] = (uint16_t)b;
    }
    tm.sync();
    {
        const int nblk = sc[2], cap = top_cap(vc), wcap = ceil_div(vc, 64);
        __shared__ int s_wcnt[NT / 32];
        for (;;) {
            int i = 0;
            if (tm.lane() == 0) i = atomicAdd((int *)&sc[3], 1);
            i = __shfl_sync(FULL, i, 0);
            if (i >= nblk) break;
            const int b = ws.blist[i];
            const int n = peel_block(ws, M, b, ws.boff[b + 1] - ws.boff[b], ws.tC + (int64_t)tm.warp() * cap,
                                     ws.tR + (int64_t)tm.warp() * cap, ws.hmask + (int64_t)tm.warp() * wcap, W,
                                     &s_wcnt[tm.warp()], tm.lane());
            if (tm.lane() == 0) ws.nround[b] = n;
            __syncwarp();
        }
    }
    tm.sync();
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
        A2<SH, uint16_t> w2;
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
        if (W > kSumWords) {
            if (narrow) alg2_warp<true, true, FULL_OUT>(w2, a, g, G, acc, tm.t);
            else alg2_warp<true, false, FULL_OUT>(w2, a, g, G, acc, tm.t);
        } else {
            if (narrow) alg2_warp<false, true, FULL_OUT>(w2, a, g, G, acc, tm.t);
            else alg2_warp<false, false, FULL_OUT>(w2, a, g, G, acc, tm.t);
        }
    }
    tm.sync();

    // ---- per-DAG and per-node outputs
    if (lead) write_totals(a, g, d, acc, Totals{mx, b_greedy, b_unaware, b_vol, G, nlev});
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
        if constexpr (SH) {  // one warp in topological order: a node's successors are distinct
            for (int i = 0; tm.warp() == 0 && i < V; i++) {
                const int v = ws.topo[i];
                const uint64_t dv = ws.cpT[v] + ws.cpM[v];
                __syncwarp();  // every lane has read cpT[v]
                ws.cpT[v] = dv;
                for (int e = (int)rp[v] + tm.lane(); e < (int)rp[v + 1]; e += 32) {
                    const int s = ws.byrank[col[e]];
                    if (dv > ws.cpM[s]) ws.cpM[s] = dv;
                }
                __syncwarp();
            }
            tm.sync();
        } else {
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
        }
        uint64_t path = 0;
        for (int v = tm.t; v < V; v += NT) path = ws.cpT[v] > path ? ws.cpT[v] : path;
        path = tm.maxu(path);
        const uint64_t wb = (work + M - 1) / M;
        cp = path > wb ? path : wb;
    }

    if (lead && a.o.crit_path) write_crit_path(a, g, d, acc, cp);
    tm.sync();
}

// ------------------------------------------------------------------ kernels
// Warp teams for small DAGs: kWarpsPerCta teams per CTA, each with a shared-memory workspace
// sized for (a.vcap, a.ecap), the largest V and E of the launch's size class.
// Five CTAs an SM (96 registers): at four (128) the 10,000-DAG batch is latency-bound on 16 warps.
// The variants with every output keep four: at 96 registers they spill (1,000 DAGs of 50-500 nodes
// with the plan written out: 1.27 ms at four, 1.35 ms at five).
template <bool FULL_OUT>
__global__ void __launch_bounds__(32 * kWarpsPerCta, FULL_OUT ? 4 : 5) k_sched_warp(SchedArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const WarpWs ws = warp_carve(a.vcap, a.ecap);
    const uint32_t base = (threadIdx.x >> 5) * ws.bytes;
    for (int idx = blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);;) {
        if (a.counter) {
            if (lane == 0) idx = atomicAdd(a.counter, 1);
            idx = __shfl_sync(FULL, idx, 0);
        }
        if (idx >= a.n_list) break;
        schedule_warp<FULL_OUT>(ws, base, a, a.list[idx], lane);
        if (!a.counter) break;
        __syncwarp();
    }
}

// CTA teams for large DAGs: the workspace sized for (a.vcap, a.ecap) lives in dynamic shared
// memory (SMEM) or in the global block a.gws + blockIdx.x * a.gws_stride.
template <int NT, bool SMEM, bool FULL_OUT>
__global__ void __launch_bounds__(NT, SMEM ? 512 / NT : 1) k_sched_cta(SchedArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t red[NT / 32];
    __shared__ int idx_s;
    Ws ws;
    ws_carve(SMEM ? smem : a.gws + (int64_t)blockIdx.x * a.gws_stride, a.vcap, a.ecap, &ws, SMEM);
    if constexpr (!SMEM) {  // the released set changes with every group: always in shared memory
        ws.relmask = (uint64_t *)smem;
        ws.relsum = ws.relmask + kRelWords;
    }
    Team<NT> tm{(int)threadIdx.x, red};
    for (;;) {
        if (threadIdx.x == 0) idx_s = a.counter ? atomicAdd(a.counter, 1) : (int)blockIdx.x;
        __syncthreads();
        const int idx = idx_s;
        __syncthreads();
        if (idx >= a.n_list) break;
        schedule_one<NT, SMEM, FULL_OUT>(tm, ws, a, a.list ? a.list[idx] : idx, a.vcap, a.ecap);
        if (!a.counter) break;
        __syncthreads();
    }
}

// ------------------------------------------------------------------ launchers
// Does the call need the FULL_OUT kernels?
static bool full_out(const SchedArgs &a) {
    const dagrt_schedule_out &o = a.o;
    return a.variant != DAGRT_VAR_PAPER || !a.plan || o.n_extra || o.extra_off || o.group_R || o.seg_parent ||
           o.row_id || o.row_group || o.row_m0 || o.row_load;
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
    const int64_t bytes = (int64_t)warp_carve(a.vcap, a.ecap).bytes * kWarpsPerCta;
    const bool full = full_out(a);
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
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCtaThreadsGlobal, kGlobalSmem);
        if (e == cudaSuccess && per_sm > best) best = per_sm;
    }
    return n_sm * best;
}

cudaError_t sched_launch_cta(const SchedArgs &a, int grid, cudaStream_t st) {
    if (grid < 1 || a.n_list < 1) return cudaSuccess;
    const auto kern = full_out(a) ? k_sched_cta<kCtaThreadsGlobal, false, true> : k_sched_cta<kCtaThreadsGlobal, false, false>;
    kern<<<grid, kCtaThreadsGlobal, kGlobalSmem, st>>>(a);
    return cudaGetLastError();
}

int64_t sched_smem_limit() {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    return optin - 512;  // the kernels' static shared memory
}

cudaError_t sched_launch_cta_smem(const SchedArgs &a, int n_sm, cudaStream_t st) {
    if (a.n_list < 1) return cudaSuccess;
    const int64_t bytes = sched_smem_ws_bytes(a.vcap, a.ecap);
    const auto kern = full_out(a) ? k_sched_cta<kCtaThreads, true, true> : k_sched_cta<kCtaThreads, true, false>;
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
