// gnn.cu -- learned proposer: message-passing network forward/backward on the tensor
// cores (tcgen05 + TMEM), Adam, and top-k decoding of per-kernel SM-level distributions.
//
// GEMM tiles are 128 node rows. Operands are staged by the CTA's threads into shared memory
// in the K-major no-swizzle layout (umma.cuh). A layer's input is [h | mean over predecessors |
// mean over successors]: a kernel of its own gathers the two means into `agg` (512 bytes a node
// and 128-wide layer, written and read once more by the weight gradients), the product reads
// them beside h. Reductions over nodes (weight gradients) run in a fixed order (per-CTA partials in TMEM, then a fixed-order sum), so training is
// deterministic for a given GPU.
#include <cuda_bf16.h>

#include <cfloat>

#include "dagrt_internal.cuh"
#include "gnn.cuh"
#include "umma.cuh"

namespace dagrt {

constexpr uint32_t kWaitLimit = 1u << 24;

__device__ __forceinline__ float bf2f(uint16_t x) { return __uint_as_float((uint32_t)x << 16); }
__device__ __forceinline__ uint16_t f2bf(float f) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}

// ------------------------------------------------------------------ graph
constexpr int kGraphThreads = 256;
constexpr int kGraphWarps = kGraphThreads / 32;
constexpr int kGraphSmemV = 2048;  // DAGs up to this many nodes build in shared memory

// shared memory of k_gnn_graph for DAGs of up to v nodes: a cursor per warp and node, row
// pointers and offsets
static int graph_smem(int v) { return 4 * ((kGraphWarps + 2) * v + 1); }

// One CTA per DAG: global successor CSR, in-degrees, then predecessor lists with every list
// in increasing predecessor id (deterministic). DAGs of at most vcap nodes: a stable counting
// sort of the edges (CSR order: increasing source) by target. Each warp counts the targets of
// its eighth of the edges, the counts of the warps before it and the scan over the nodes give
// its cursors, and it fills 32 edges at a time; lanes with the same target rank themselves
// with a match. Larger DAGs: counts and fill in global memory with atomics, then an insertion
// sort per list. Bound by the latency of a DAG's passes: eight warps a DAG instead of one
// take 300 DAGs of 100-1,000 nodes from 725 to 110 us.
__global__ void __launch_bounds__(kGraphThreads)
    k_gnn_graph(int32_t n_dags, const int64_t *node_off, const int64_t *edge_off, const int32_t *row_ptr,
                const int32_t *col, const int32_t *status, int2 *pred, int32_t *pred_idx, int2 *succ,
                int32_t *succ_idx, int32_t *cursor, int vcap) {
    extern __shared__ int32_t s_graph[];
    __shared__ uint64_t red[kGraphWarps];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const Team<kGraphThreads> tm{tid, red};
    int32_t *rps = s_graph;           // [V + 1]: the DAG's row pointers
    int32_t *off = rps + vcap + 1;    // [V]: in-degrees, then the end of each list
    int32_t *cur = off + vcap;        // [warps][V]: counts, then next free slot
    for (int d = blockIdx.x; d < n_dags; d += gridDim.x) {
        const int64_t n0 = node_off[d], e0 = edge_off[d];
        const int V = (int)(node_off[d + 1] - n0);
        if (status[d] != DAGRT_OK) {  // a DAG the scheduler rejected: its CSR is not trusted
            for (int v = tid; v < V; v += kGraphThreads)
                succ[n0 + v] = pred[n0 + v] = make_int2((int32_t)e0, (int32_t)e0);
            continue;
        }
        const int32_t *rp = row_ptr + n0 + d;
        const int32_t *cl = col + e0;
        const int E = rp[V];
        if (V <= vcap) {
            for (int v = tid; v <= V; v += kGraphThreads) {
                const int x = rp[v];
                rps[v] = x;
                if (v < V) succ[n0 + v] = make_int2((int32_t)(e0 + x), (int32_t)(e0 + rp[v + 1]));
            }
            for (int i = tid; i < kGraphWarps * V; i += kGraphThreads) cur[i] = 0;
            __syncthreads();
            const int seg = ((E + kGraphWarps - 1) / kGraphWarps + 31) & ~31;
            const int s0 = min(E, w * seg), s1 = min(E, s0 + seg);
            int32_t *mine = cur + w * V;
            for (int e = s0 + lane; e < s1; e += 32) {
                const int t = cl[e];
                succ_idx[e0 + e] = (int32_t)(n0 + t);
                atomicAdd(&mine[t], 1);
            }
            __syncthreads();
            for (int v = tid; v < V; v += kGraphThreads) {
                int x = 0;
                for (int i = 0; i < kGraphWarps; i++) {
                    const int c = cur[i * V + v];
                    cur[i * V + v] = x;
                    x += c;
                }
                off[v] = x;
            }
            __syncthreads();
            team_scan_inplace(tm, off, V, [](uint64_t x, uint64_t y) { return x + y; }, false);
            for (int v = tid; v < V; v += kGraphThreads) {
                const int x = v ? off[v - 1] : 0;
                pred[n0 + v] = make_int2((int32_t)(e0 + x), (int32_t)(e0 + off[v]));
                for (int i = 0; i < kGraphWarps; i++) cur[i * V + v] += x;
            }
            __syncthreads();
            int u = 0;  // source row of the segment's first edge: the last row starting at or before it
            if (s0 < s1) {
                int hi = V;
                while (hi - u > 1) {
                    const int mid = (u + hi) >> 1;
                    if (rps[mid] <= s0) u = mid;
                    else hi = mid;
                }
            }
            for (int base = s0; base < s1; base += 32) {
                const int e = base + lane;
                const bool act = e < s1;
                const int t = act ? cl[e] : -1;
                int r = u;
                if (act)
                    while (rps[r + 1] <= e) r++;
                const uint32_t same = __match_any_sync(FULL, t);  // lanes of this chunk with target t
                const int rank = __popc(same & ((1u << lane) - 1));
                const int slot = act ? mine[t] + rank : 0;
                __syncwarp();
                if (act) {
                    if (rank == __popc(same) - 1) mine[t] = slot + 1;  // the set's last lane moves the cursor
                    pred_idx[e0 + slot] = (int32_t)(n0 + r);
                }
                u = __shfl_sync(FULL, r, 31);
                __syncwarp();
            }
            __syncthreads();
            continue;
        }
        for (int v = tid; v < V; v += kGraphThreads) {
            succ[n0 + v] = make_int2((int32_t)(e0 + rp[v]), (int32_t)(e0 + rp[v + 1]));
            cursor[n0 + v] = 0;
        }
        for (int e = tid; e < E; e += kGraphThreads) succ_idx[e0 + e] = (int32_t)(n0 + cl[e]);
        __syncthreads();
        for (int e = tid; e < E; e += kGraphThreads) atomicAdd(&cursor[n0 + cl[e]], 1);
        __syncthreads();
        team_scan_inplace(tm, cursor + n0, V, [](uint64_t x, uint64_t y) { return x + y; }, false);
        for (int v = tid; v < V; v += kGraphThreads)
            pred[n0 + v] = make_int2((int32_t)(e0 + (v ? cursor[n0 + v - 1] : 0)), (int32_t)(e0 + cursor[n0 + v]));
        __syncthreads();
        for (int v = tid; v < V; v += kGraphThreads) cursor[n0 + v] = 0;
        __syncthreads();
        for (int u = tid; u < V; u += kGraphThreads)  // fill in any order ...
            for (int e = rp[u]; e < rp[u + 1]; e++) {
                const int s = cl[e];
                pred_idx[pred[n0 + s].x + atomicAdd(&cursor[n0 + s], 1)] = (int32_t)(n0 + u);
            }
        __syncthreads();
        for (int v = tid; v < V; v += kGraphThreads) {  // ... then sort each list (increasing predecessor id)
            int32_t *p = pred_idx + pred[n0 + v].x;
            const int n = cursor[n0 + v];
            for (int i = 1; i < n; i++) {
                const int32_t x = p[i];
                int j = i - 1;
                while (j >= 0 && p[j] > x) {
                    p[j + 1] = p[j];
                    j--;
                }
                p[j + 1] = x;
            }
        }
        __syncthreads();
    }
}

cudaError_t gnn_build_graph(int32_t n_dags, const int64_t *node_off, const int64_t *edge_off, const int32_t *row_ptr,
                            const int32_t *col, const int32_t *status, int2 *pred, int32_t *pred_idx,
                            int2 *succ, int32_t *succ_idx, int32_t *cursor, int max_v, int n_sm,
                            cudaStream_t st) {
    if (n_dags == 0) return cudaSuccess;
    const int vcap = max_v < kGraphSmemV ? max_v : kGraphSmemV;
    cudaError_t e = cudaFuncSetAttribute(k_gnn_graph, cudaFuncAttributeMaxDynamicSharedMemorySize, graph_smem(kGraphSmemV));
    if (e != cudaSuccess) return e;
    const int grid = n_dags < 32 * n_sm ? n_dags : 32 * n_sm;
    k_gnn_graph<<<grid, kGraphThreads, graph_smem(vcap), st>>>(n_dags, node_off, edge_off, row_ptr, col, status,
                                                               pred, pred_idx, succ, succ_idx, cursor, vcap);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ features
// x = [log2 C^ / 32, k / 64, log2(1 + indeg) / 8, log2(1 + outdeg) / 8, level / depth,
//      W^anc / sum C^, log2 m / 12 (the paper schedule's SMs), 1, 0 ...] (16 bf16)
constexpr int kFeatThreads = 256;
__global__ void __launch_bounds__(kFeatThreads) k_gnn_features(int32_t n_dags, const int64_t *node_off, const int64_t *wcet, const uint8_t *k64,
                               const int32_t *level, const int64_t *wanc, const int32_t *m, const int32_t *status,
                               GnnGraph g, uint16_t *x) {
    __shared__ double s_tot[kFeatThreads / 32];
    __shared__ int s_depth[kFeatThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    for (int d = blockIdx.x; d < n_dags; d += gridDim.x) {  // a CTA per DAG
        const int64_t n0 = node_off[d];
        const int V = (int)(node_off[d + 1] - n0);
        if (status[d] != DAGRT_OK) {  // no schedule outputs: zero features
            for (int v = tid; v < V; v += kFeatThreads) {
                uint4 *dst = (uint4 *)(x + (n0 + v) * kFeat);
                dst[0] = make_uint4(0, 0, 0, 0);
                dst[1] = make_uint4(0, 0, 0, 0);
            }
            continue;
        }
        double tot = 0;  // whole ticks: exact in any order
        int depth = 0;
        for (int v = tid; v < V; v += kFeatThreads) {
            tot += (double)wcet[n0 + v];
            depth = max(depth, level[n0 + v]);
        }
        for (int o = 16; o > 0; o >>= 1) {
            tot += __shfl_xor_sync(FULL, tot, o);
            depth = max(depth, __shfl_xor_sync(FULL, depth, o));
        }
        __syncthreads();  // the DAG before is read
        if (lane == 0) {
            s_tot[tid >> 5] = tot;
            s_depth[tid >> 5] = depth;
        }
        __syncthreads();
        tot = 0;
        for (int i = 0; i < kFeatThreads / 32; i++) {
            tot += s_tot[i];
            depth = max(depth, s_depth[i]);
        }
        for (int v = tid; v < V; v += kFeatThreads) {
            const int64_t i = n0 + v;
            float f[kFeat];
#pragma unroll
            for (int q = 0; q < kFeat; q++) f[q] = 0.f;
            f[0] = log2f((float)wcet[i]) / 32.f;
            f[1] = (float)k64[i] / 64.f;
            const int2 pl = g.pred[i], sl = g.succ[i];
            f[2] = log2f(1.f + (float)(pl.y - pl.x)) / 8.f;
            f[3] = log2f(1.f + (float)(sl.y - sl.x)) / 8.f;
            f[4] = depth > 0 ? (float)level[i] / (float)depth : 0.f;
            f[5] = tot > 0 ? (float)((double)wanc[i] / tot) : 0.f;
            f[6] = log2f((float)max(m[i], 1)) / 12.f;
            f[7] = 1.f;
            uint32_t w[kFeat / 2];
#pragma unroll
            for (int q = 0; q < kFeat / 2; q++) w[q] = (uint32_t)f2bf(f[2 * q]) | ((uint32_t)f2bf(f[2 * q + 1]) << 16);
            uint4 *dst = (uint4 *)(x + i * kFeat);
            dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
            dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
    }
}

cudaError_t gnn_features(int32_t n_dags, const int64_t *node_off, const int64_t *wcet, const uint8_t *k64,
                         const int32_t *level, const int64_t *wanc, const int32_t *m, const int32_t *status, GnnGraph g,
                         uint16_t *x, int n_sm, cudaStream_t st) {
    if (n_dags == 0) return cudaSuccess;
    const int grid = n_dags < 32 * n_sm ? n_dags : 32 * n_sm;
    k_gnn_features<<<grid, kFeatThreads, 0, st>>>(n_dags, node_off, wcet, k64, level, wanc, m, status, g, x);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ aggregation
__device__ __forceinline__ uint4 pack8(const float *f) {
    return make_uint4((uint32_t)f2bf(f[0]) | ((uint32_t)f2bf(f[1]) << 16), (uint32_t)f2bf(f[2]) | ((uint32_t)f2bf(f[3]) << 16),
                      (uint32_t)f2bf(f[4]) | ((uint32_t)f2bf(f[5]) << 16), (uint32_t)f2bf(f[6]) | ((uint32_t)f2bf(f[7]) << 16));
}

// acc[2i], acc[2i + 1] += the two bf16 of word i (fp32 additions, two to an instruction)
__device__ __forceinline__ void acc8(uint64_t *acc, uint4 u) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; i++) {
        uint64_t x;
        asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(w[i] << 16), "r"(w[i] & 0xffff0000u));
        asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[i]) : "l"(x));
    }
}

// bf16 mean over the rows idx[list.x .. list.y) of h, features [8 sub, 8 sub + 8): fp32 sums in list
// order, one rounding; four rows in flight. OVERLAP: the launch may start while the kernel that
// writes h still runs, so h is not read-only for its whole life (what ld.global.nc asks for).
template <int KIN, bool OVERLAP>
__device__ __forceinline__ uint4 mean_rows(const uint16_t *h, const int32_t *__restrict__ idx, int2 list, int sub) {
    auto ld = [](const uint4 *p) {
        if constexpr (OVERLAP) return *p;
        else return __ldg(p);
    };
    const int b = list.x, e = list.y;
    uint64_t acc[4] = {0, 0, 0, 0};
    const uint4 *hs = (const uint4 *)h + sub;
    int i = b;
    for (; i + 4 <= e; i += 4) {
        const int32_t j0 = __ldg(idx + i), j1 = __ldg(idx + i + 1), j2 = __ldg(idx + i + 2), j3 = __ldg(idx + i + 3);
        const uint4 u0 = ld(hs + (int64_t)j0 * (KIN / 8)), u1 = ld(hs + (int64_t)j1 * (KIN / 8));
        const uint4 u2 = ld(hs + (int64_t)j2 * (KIN / 8)), u3 = ld(hs + (int64_t)j3 * (KIN / 8));
        acc8(acc, u0);
        acc8(acc, u1);
        acc8(acc, u2);
        acc8(acc, u3);
    }
    for (; i < e; i++) acc8(acc, ld(hs + (int64_t)__ldg(idx + i) * (KIN / 8)));
    const float inv = e > b ? 1.f / (float)(e - b) : 0.f;
    float m[8];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        float x, y;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(acc[q]));
        m[2 * q] = x * inv;
        m[2 * q + 1] = y * inv;
    }
    return pack8(m);
}

// agg[v] = [mean over predecessors of h | mean over successors of h], bf16 [N x 2 KIN]. A
// group of KIN/8 lanes owns a node (16 bytes = 8 features per lane). A CTA's nodes are
// neighbours in the batch, so mostly of one DAG, whose rows (140 KB for 550 nodes) stay in
// the L1 cache: the kernel uses no shared memory, and that is why it is apart from the
// matrix product, whose operands fill it. Bound by latency: 42 warps an SM issue in 63% of the
// cycles, and 10 of the 17 cycles between a warp's instructions are waits for indices and rows
// (13 TB/s of rows; L1 at 58% of its rate, L2 25%, DRAM 12%).
// 165,000 nodes, 2.8 M edges, 128 features: 110 us, and the product 52, where one kernel for
// both took 190 (the rows of a CTA's nodes from a chunk next to its SM's other CTAs: 127, the
// chunks' degrees then differ by SM); 16 features: 97 -> 31 and 24.
//
// SMALL (up to four 128-node tiles of the product per SM): latency is what counts, so a warp
// takes the predecessors or the successors of its nodes, a CTA one pass of them, and the
// layer's kernels start early (programmatic launches). Three layers and the head, in this form
// and in the other: 9,000 nodes of degree 55 58 and 85 us, 25,000 of degree 20 81 and 101,
// 42,000 of degree 70 150 and 175. On 165,000 nodes the two kinds of lists apart cost the L1
// cache more than they gain (447 -> 473).
constexpr int kAggThreads = 512;
template <int KIN, bool SMALL>
__global__ void __launch_bounds__(kAggThreads, 3) k_gnn_agg(GnnGraph g, const uint16_t *h, uint16_t *agg) {
    constexpr int LPN = KIN / 8;  // lanes per node
    if constexpr (SMALL) {
        griddep_wait();
        griddep_launch_dependents();
        constexpr int NODES = kAggThreads / 2 / LPN;
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane % LPN, succ = w & 1;
        const int2 *list = succ ? g.succ : g.pred;
        const int32_t *idx = succ ? g.succ_idx : g.pred_idx;
        for (int64_t v = (int64_t)blockIdx.x * NODES + (w >> 1) * (32 / LPN) + lane / LPN; v < g.n_nodes;
             v += (int64_t)gridDim.x * NODES)
            ((uint4 *)(agg + v * 2 * KIN))[succ * LPN + sub] = mean_rows<KIN, true>(h, idx, list[v], sub);
    } else {
        constexpr int NODES = kAggThreads / LPN;          // nodes per CTA pass
        constexpr int CHUNK = NODES < 128 ? 128 : NODES;  // neighbouring nodes that a CTA takes together
        const int sub = threadIdx.x % LPN;
        for (int64_t c0 = (int64_t)blockIdx.x * CHUNK; c0 < g.n_nodes; c0 += (int64_t)gridDim.x * CHUNK)
            for (int i = 0; i < CHUNK / NODES; i++) {
                const int64_t v = c0 + i * NODES + threadIdx.x / LPN;
                if (v >= g.n_nodes) break;
                uint4 *dst = (uint4 *)(agg + v * 2 * KIN);
                dst[sub] = mean_rows<KIN, false>(h, g.pred_idx, g.pred[v], sub);
                dst[LPN + sub] = mean_rows<KIN, false>(h, g.succ_idx, g.succ[v], sub);
            }
    }
}

// 16-byte piece i of warp w's share of a [128 rows x 8 C columns] tile in the layout of
// kmajor_off. A warp takes RW rows of CL pieces: whole 128-byte lines of four rows (C a
// multiple of 8; two lanes then store to the same banks) or 32 bytes of 16 rows.
template <int C>
__device__ __forceinline__ void tile_piece(int i, int warps, int w, int lane, int &r, int &c) {
    constexpr int CL = C % 8 == 0 ? 8 : 2, RW = 32 / CL;
    const int p = i * warps + w;
    c = p % (C / CL) * CL + lane / RW;
    r = p / (C / CL) * RW + lane % RW;
}

// 32 bytes in one store (an aligned sector)
__device__ __forceinline__ void st32(void *p, const uint32_t *x) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(x[0]), "r"(x[1]), "r"(x[2]),
                 "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7])
                 : "memory");
}

// ------------------------------------------------------------------ forward layer
// h_out = ReLU([h | agg] W + b). Persistent CTAs over 128-row tiles: the A tile (K = 3 KIN) is
// copied to shared memory through registers, the next tile's loads issued before the wait for
// this one's MMA; one thread issues the tcgen05 chain against the resident W^T; the epilogue
// (bias, ReLU, bf16) reads TMEM: warp w takes TMEM lanes 32 (w % 4) .. + 31 and columns
// 32 (w / 4) .. + 31. Bound by reading A.
constexpr int kFwdThreads = 512;

template <int KIN>
__global__ void __launch_bounds__(kFwdThreads) k_gnn_fwd(GnnGraph g, const uint16_t *h_in, const uint16_t *agg,
                                                         const uint16_t *__restrict__ wt,
                                                         const float *__restrict__ bias, uint16_t *h_out,
                                                         int32_t *err, bool early) {
    constexpr int K = 3 * KIN, C = K / 8, N_IT = (128 * C + kFwdThreads - 1) / kFwdThreads;
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    __shared__ float sbias[kHidden];
    unsigned char *sA = sm, *sB = sm + 128 * K * 2;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    uint4 x[N_IT];  // this thread's 16-byte pieces of the next A tile
    auto load = [&](int64_t tile) {
#pragma unroll
        for (int i = 0; i < N_IT; i++) {
            int r, c;
            tile_piece<C>(i, kFwdThreads / 32, w, lane, r, c);
            const int64_t v = tile * 128 + r;
            x[i] = make_uint4(0, 0, 0, 0);
            if (r < 128 && v < g.n_nodes)
                x[i] = c < KIN / 8 ? *((const uint4 *)(h_in + v * KIN) + c)
                                   : *((const uint4 *)(agg + v * 2 * KIN) + c - KIN / 8);
        }
    };
    if (!early) load(blockIdx.x);
    for (int i = t; i < kHidden * (K / 8); i += blockDim.x) {  // W^T [H x K] -> K-major B operand
        const int r = i / (K / 8), kc = (i % (K / 8)) * 8;
        *(uint4 *)(sB + kmajor_off(r, kc, K)) = *(const uint4 *)(wt + (size_t)r * K + kc);
    }
    if (t < kHidden) sbias[t] = bias[t];
    if (w == 0) tmem_alloc(&tslot, 128);
    if (t == 0) mbar_init1(&bar);
    if (early) {  // the weights are older than the aggregation that this launch may overlap
        griddep_wait();
        griddep_launch_dependents();
        load(blockIdx.x);
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t taddr = tslot;
    const int64_t n_tiles = (g.n_nodes + 127) / 128;
    const int lq = w & 3, c0 = 32 * (w >> 2);  // epilogue: TMEM lane quarter and 32-column block
    uint32_t phase = 0;
    bool ok = true;
    for (int64_t tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
#pragma unroll
        for (int i = 0; i < N_IT; i++) {
            int r, c;
            tile_piece<C>(i, kFwdThreads / 32, w, lane, r, c);
            if (r < 128) *(uint4 *)(sA + kmajor_off(r, 8 * c, K)) = x[i];
        }
        fence_async_smem();
        __syncthreads();
        if (t == 0) {
            tmem_fence_after();
            umma_gemm(taddr, sA, sB, K, kHidden, false);
            umma_commit(&bar);
        }
        load(tile + gridDim.x);  // (rows past the end read as zero)
        ok = __syncthreads_and(mbar_wait_parity(&bar, phase, kWaitLimit)) != 0;  // uniform across the CTA
        phase ^= 1;
        tmem_fence_after();
        if (ok) {
            const int64_t v = tile * 128 + 32 * lq + lane;  // this thread's TMEM lane = row 32 lq + lane
            float acc[32];
            tmem_ld32(taddr + ((uint32_t)(32 * lq) << 16) + c0, acc);
            if (v < g.n_nodes) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    const float a0 = fmaxf(acc[2 * i] + sbias[c0 + 2 * i], 0.f);
                    const float a1 = fmaxf(acc[2 * i + 1] + sbias[c0 + 2 * i + 1], 0.f);
                    pk[i] = (uint32_t)f2bf(a0) | ((uint32_t)f2bf(a1) << 16);
                }
                st32(h_out + v * kHidden + c0, pk);
                st32(h_out + v * kHidden + c0 + 16, pk + 8);
            }
        } else if (t == 0 && err) {
            atomicExch(err, DAGRT_E_TIMEOUT);
        }
        // no barrier here: the MMA that read the A tile has completed, and the barrier after the
        // next copy orders this epilogue's TMEM reads before the next MMA writes the accumulator
        tmem_fence_before();
    }
    __syncthreads();  // every epilogue has read TMEM before it is released
    if (w == 0) tmem_dealloc(taddr, 128);
}

// one launch of the forward chain, early: it may start before the kernel before it has ended
template <class... P, class... A>
static cudaError_t launch_chain(bool early, void (*kern)(P...), int64_t grid, int block, int smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// a batch of at most four 128-node tiles per SM (see k_gnn_agg)
static bool small_batch(int64_t n_nodes, int n_sm) { return n_nodes <= 512ll * n_sm; }

template <int KIN>
static cudaError_t launch_fwd(GnnGraph g, const uint16_t *h_in, const uint16_t *wt, const float *bias,
                              uint16_t *h_out, uint16_t *agg, int32_t *err, int n_sm, cudaStream_t st) {
    constexpr int K = 3 * KIN;
    const int64_t n_tiles = (g.n_nodes + 127) / 128;
    if (n_tiles < 1) return cudaSuccess;
    const bool small = small_batch(g.n_nodes, n_sm);
    const auto agg_kern = small ? k_gnn_agg<KIN, true> : k_gnn_agg<KIN, false>;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, agg_kern, kAggThreads, 0);
    if (e != cudaSuccess) return e;
    constexpr int pass = kAggThreads * 8 / KIN, chunk = pass < 128 ? 128 : pass;
    const int64_t per_cta = small ? pass / 2 : chunk;
    const int64_t n_chunks = (g.n_nodes + per_cta - 1) / per_cta, most = (int64_t)n_sm * (per_sm < 1 ? 1 : per_sm);
    e = launch_chain(small, agg_kern, n_chunks < most ? n_chunks : most, kAggThreads, 0, st, g, h_in, agg);
    if (e != cudaSuccess) return e;
    const int smem = 2 * 128 * K * 2;
    e = cudaFuncSetAttribute(k_gnn_fwd<KIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gnn_fwd<KIN>, kFwdThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    if (per_sm > 4) per_sm = 4;  // 4 x 128 TMEM columns per SM
    const int64_t grid = n_tiles < (int64_t)n_sm * per_sm ? n_tiles : (int64_t)n_sm * per_sm;
    return launch_chain(small, k_gnn_fwd<KIN>, grid, kFwdThreads, smem, st, g, h_in, (const uint16_t *)agg, wt, bias, h_out,
                        err, small);
}

cudaError_t gnn_layer_fwd(int kin, GnnGraph g, const uint16_t *h_in, const uint16_t *wt, const float *bias,
                          uint16_t *h_out, uint16_t *agg, int32_t *err, int n_sm, cudaStream_t st) {
    if (kin == kFeat) return launch_fwd<kFeat>(g, h_in, wt, bias, h_out, agg, err, n_sm, st);
    if (kin == kHidden) return launch_fwd<kHidden>(g, h_in, wt, bias, h_out, agg, err, n_sm, st);
    return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------ head
// logits = h3 Wh + bh; with labels: softmax cross-entropy (mean over labelled nodes, via
// `scale` = 1 / count), dlogits and dh3 = dlogits Wh^T. One thread per node up to the
// logits; the 32 nodes of a warp are then written together: logits and dlogits through
// shared memory, dh3 with four outputs per lane (their weights in registers), so every store
// is a whole line. The loss is reduced per CTA in a fixed order. Bound by the FMAs of the two
// products; with one node's row per thread for the stores too, and one CTA an SM, 110,000
// nodes took 285 us (now 89), 165,000 without labels 77 (now 39).
constexpr int kHeadThreads = 128;
constexpr int kHeadMaxCtas = 1024;  // partial losses
template <bool OVERLAP>
__global__ void __launch_bounds__(kHeadThreads) k_gnn_head(GnnGraph g, const uint16_t *h3,
                                                  const float *__restrict__ wh, const float *__restrict__ bh,
                                                  int L, const int8_t *__restrict__ labels, float scale,
                                                  float *logits, float *dlogits, float *dh3, float *loss_part) {
    __shared__ __align__(16) float swh[kHidden * kMaxLevels];
    __shared__ float sbh[kMaxLevels];
    __shared__ float sloss[kHeadThreads];
    __shared__ float sout[kHeadThreads / 32][32 * kMaxLevels];
    for (int i = threadIdx.x; i < kHidden * kMaxLevels; i += blockDim.x) swh[i] = wh[i];
    if (threadIdx.x < kMaxLevels) sbh[threadIdx.x] = bh[threadIdx.x];
    if constexpr (OVERLAP) griddep_wait();  // (in a small batch this launch overlaps the last layer's)
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float *so = sout[w];
    float my_loss = 0.f;
    for (int64_t v0 = ((int64_t)blockIdx.x * kHeadThreads + 32 * w); v0 < g.n_nodes;
         v0 += (int64_t)gridDim.x * kHeadThreads) {
        const int64_t v = v0 + lane;
        const int n = (int)min((int64_t)32, g.n_nodes - v0);  // nodes of this warp
        float z[kMaxLevels];
#pragma unroll
        for (int l = 0; l < kMaxLevels; l++) z[l] = l < L ? sbh[l] : 0.f;
        if (lane < n) {
            const uint4 *row = (const uint4 *)(h3 + v * kHidden);
#pragma unroll 2
            for (int c = 0; c < kHidden / 8; c++) {
                uint4 q;
                if constexpr (OVERLAP) q = row[c];
                else q = __ldg(row + c);
                const uint32_t wd[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const float hv = bf2f((uint16_t)(wd[j >> 1] >> (16 * (j & 1))));
                    const float4 *wr = (const float4 *)(swh + (8 * c + j) * kMaxLevels);
#pragma unroll
                    for (int l4 = 0; l4 < kMaxLevels / 4; l4++) {
                        if (4 * l4 >= L) break;
                        const float4 x = wr[l4];
                        z[4 * l4] = fmaf(hv, x.x, z[4 * l4]);
                        z[4 * l4 + 1] = fmaf(hv, x.y, z[4 * l4 + 1]);
                        z[4 * l4 + 2] = fmaf(hv, x.z, z[4 * l4 + 2]);
                        z[4 * l4 + 3] = fmaf(hv, x.w, z[4 * l4 + 3]);
                    }
                }
            }
        }
        auto put = [&](float *dst, const float *x) {  // 32 rows of L values, in order
#pragma unroll
            for (int l = 0; l < kMaxLevels; l++)
                if (l < L) so[lane * L + l] = x[l];
            __syncwarp();
            for (int i = lane; i < n * L; i += 32) dst[v0 * L + i] = so[i];
            __syncwarp();
        };
        if (logits) put(logits, z);
        if (!labels) continue;
        const int y = lane < n ? labels[v] : -1;
        float gz[kMaxLevels];
#pragma unroll
        for (int l = 0; l < kMaxLevels; l++) gz[l] = 0.f;
        if (y >= 0 && y < L) {
            float mx = z[0], zy = 0.f;
#pragma unroll
            for (int l = 0; l < kMaxLevels; l++)
                if (l < L) {
                    mx = fmaxf(mx, z[l]);
                    zy = l == y ? z[l] : zy;
                }
            float se = 0.f;
#pragma unroll
            for (int l = 0; l < kMaxLevels; l++)
                if (l < L) se += __expf(z[l] - mx);
            const float lse = mx + __logf(se);
            my_loss += (lse - zy) * scale;
#pragma unroll
            for (int l = 0; l < kMaxLevels; l++)
                if (l < L) gz[l] = (__expf(z[l] - lse) - (l == y ? 1.f : 0.f)) * scale;
        }
        put(dlogits, gz);
        // dh3: lane owns outputs 4 lane .. + 3 of every node; gz of node i from lane i
        float4 acc[4];
        for (int i0 = 0; i0 < n; i0 += 4) {
#pragma unroll
            for (int i = 0; i < 4; i++) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int l = 0; l < kMaxLevels; l++) {
                if (l >= L) break;
                const float *wl = swh + 4 * lane * kMaxLevels + l;
                const float w0 = wl[0], w1 = wl[kMaxLevels], w2 = wl[2 * kMaxLevels], w3 = wl[3 * kMaxLevels];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const float gv = __shfl_sync(FULL, gz[l], (i0 + i) & 31);
                    acc[i].x = fmaf(gv, w0, acc[i].x);
                    acc[i].y = fmaf(gv, w1, acc[i].y);
                    acc[i].z = fmaf(gv, w2, acc[i].z);
                    acc[i].w = fmaf(gv, w3, acc[i].w);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (i0 + i < n) *(float4 *)(dh3 + (v0 + i0 + i) * kHidden + 4 * lane) = acc[i];
        }
    }
    if (labels && loss_part) {
        sloss[threadIdx.x] = my_loss;
        __syncthreads();
        if (threadIdx.x == 0) {
            float s = 0.f;
            for (int i = 0; i < (int)blockDim.x; i++) s += sloss[i];
            loss_part[blockIdx.x] = s;
        }
    }
}

// CTAs of gnn_head, and partial losses it writes
int gnn_head_ctas(int64_t n_nodes, int n_sm) {
    int64_t grid = (n_nodes + kHeadThreads - 1) / kHeadThreads;
    const int64_t most = 6 * n_sm < kHeadMaxCtas ? 6 * n_sm : kHeadMaxCtas;
    return (int)(grid < 1 ? 1 : grid < most ? grid : most);
}

cudaError_t gnn_head(GnnGraph g, const uint16_t *h3, const float *wh, const float *bh, int n_levels,
                     const int8_t *labels, float scale, float *logits, float *dlogits, float *dh3,
                     float *loss_part, int n_sm, cudaStream_t st) {
    if (g.n_nodes == 0) return cudaSuccess;
    // the loss is reduced per CTA: a fixed grid keeps the summation order fixed
    const bool small = small_batch(g.n_nodes, n_sm);
    return launch_chain(small, small ? k_gnn_head<true> : k_gnn_head<false>, gnn_head_ctas(g.n_nodes, n_sm), kHeadThreads, 0,
                        st, g, h3, wh, bh, n_levels, labels, scale, logits, dlogits, dh3, loss_part);
}

// dWh = h3^T dlogits, dbh = sum dlogits: CTA c reduces a fixed node range in tiles of
// kHgTile nodes whose dlogits are staged; thread (o, p) adds output row o over every 8th
// node from p, and the parts are added in order. Bound by the loads of h3 (one line per node
// and warp); with one node after another per CTA it took 395 us for 110,000 nodes (now 44).
constexpr int kHgParts = 8, kHgTile = 64;
__global__ void __launch_bounds__(kHidden * kHgParts) k_gnn_head_grad(GnnGraph g, const uint16_t *__restrict__ h3,
                                                                     const float *__restrict__ dlogits, int L,
                                                                     float *part) {
    extern __shared__ __align__(16) float s_hg[];  // [tile][16] dlogits, then the parts' sums
    const int tid = threadIdx.x, o = tid & (kHidden - 1), p = tid >> 7;
    const int64_t per = (g.n_nodes + gridDim.x - 1) / gridDim.x;
    const int64_t v0 = blockIdx.x * per, v1 = min(g.n_nodes, v0 + per);
    float acc[kMaxLevels];
#pragma unroll
    for (int l = 0; l < kMaxLevels; l++) acc[l] = 0.f;
    float bacc = 0.f;  // threads 0 .. 15: dbh
    for (int64_t t0 = v0; t0 < v1; t0 += kHgTile) {
        const int n = (int)min((int64_t)kHgTile, v1 - t0);
        __syncthreads();
        for (int i = tid; i < n * kMaxLevels; i += kHidden * kHgParts) {
            const int v = i / kMaxLevels, l = i % kMaxLevels;
            s_hg[i] = l < L ? dlogits[(t0 + v) * L + l] : 0.f;
        }
        __syncthreads();
        float hv[kHgTile / kHgParts];
#pragma unroll
        for (int i = 0; i < kHgTile / kHgParts; i++) {
            const int v = p + i * kHgParts;
            hv[i] = v < n ? bf2f(h3[(t0 + v) * kHidden + o]) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < kHgTile / kHgParts; i++) {
            const int v = p + i * kHgParts;
            if (v >= n) break;
#pragma unroll
            for (int l4 = 0; l4 < kMaxLevels / 4; l4++) {
                const float4 x = *(const float4 *)(s_hg + v * kMaxLevels + 4 * l4);
                acc[4 * l4] = fmaf(hv[i], x.x, acc[4 * l4]);
                acc[4 * l4 + 1] = fmaf(hv[i], x.y, acc[4 * l4 + 1]);
                acc[4 * l4 + 2] = fmaf(hv[i], x.z, acc[4 * l4 + 2]);
                acc[4 * l4 + 3] = fmaf(hv[i], x.w, acc[4 * l4 + 3]);
            }
        }
        if (tid < kMaxLevels)
            for (int v = 0; v < n; v++) bacc += s_hg[v * kMaxLevels + tid];
    }
    float *pp = part + (int64_t)blockIdx.x * ParamLayout::total;
    __syncthreads();
#pragma unroll
    for (int l = 0; l < kMaxLevels; l++) s_hg[(p * kMaxLevels + l) * kHidden + o] = acc[l];
    __syncthreads();
    for (int i = tid; i < kHidden * kMaxLevels; i += kHidden * kHgParts) {
        const int oo = i / kMaxLevels, l = i % kMaxLevels;
        float s = 0.f;
        for (int k = 0; k < kHgParts; k++) s += s_hg[(k * kMaxLevels + l) * kHidden + oo];
        pp[ParamLayout::Wh + i] = l < L ? s : 0.f;  // (beyond L, an infinite h3 times 0 is a NaN)
    }
    if (tid < kMaxLevels) pp[ParamLayout::bh + tid] = bacc;
}

cudaError_t gnn_head_grad(GnnGraph g, const uint16_t *h3, const float *dlogits, int n_levels, float *part,
                          int n_parts, cudaStream_t st) {
    constexpr int smem = kHgParts * kMaxLevels * kHidden * 4;
    static_assert(kHgTile * kMaxLevels * 4 <= smem, "the tile fits");
    cudaError_t e = cudaFuncSetAttribute(k_gnn_head_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_gnn_head_grad<<<n_parts, kHidden * kHgParts, smem, st>>>(g, h3, dlogits, n_levels, part);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ backward
// dZ = dh * [h_out > 0] in bf16 for the 128 rows of a tile, in the layout of
// kmajor_off(row, output, kHidden); thread t of kBwdThreads takes outputs dz_out(t) .. + 7 of
// rows dz_row(t) + 32 i (eight lanes store eight rows, 128 contiguous bytes), and adds its
// unrounded dZ to db[8].
constexpr int kBwdThreads = 512;
constexpr int kZBytes = 128 * kHidden * 2;
__device__ __forceinline__ int dz_out(int t) { return 8 * (((t >> 3) & 3) + 4 * ((t >> 5) & 3)); }
__device__ __forceinline__ int dz_row(int t) { return (t & 7) + 8 * (t >> 7); }
__device__ __forceinline__ void stage_dz(const GnnGraph &g, const uint16_t *__restrict__ h_out,
                                         const float *__restrict__ dh_out, int64_t tile, unsigned char *sZ, int t,
                                         float *db) {
    const int o = dz_out(t);
    float4 x[4], y[4];
    uint4 h[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int64_t v = tile * 128 + dz_row(t) + 32 * i;
        const bool in = v < g.n_nodes;
        h[i] = in ? __ldg((const uint4 *)(h_out + v * kHidden + o)) : make_uint4(0, 0, 0, 0);
        x[i] = in ? __ldg((const float4 *)(dh_out + v * kHidden + o)) : make_float4(0.f, 0.f, 0.f, 0.f);
        y[i] = in ? __ldg((const float4 *)(dh_out + v * kHidden + o + 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        float z[8] = {x[i].x, x[i].y, x[i].z, x[i].w, y[i].x, y[i].y, y[i].z, y[i].w};
        const uint32_t hw[4] = {h[i].x, h[i].y, h[i].z, h[i].w};
#pragma unroll
        for (int j = 0; j < 8; j++) {
            if (((hw[j >> 1] >> (16 * (j & 1))) & 0xffffu) == 0) z[j] = 0.f;
            db[j] += z[j];
        }
        *(uint4 *)(sZ + kmajor_off(dz_row(t) + 32 * i, o, kHidden)) = pack8(z);
    }
}

// dW: per CTA over its tiles dW_part += A^T dZ, the reduction along the nodes: both tiles are
// MMA operands as they come, node by node (MN-major), so nothing is transposed. A = [h |
// mean_pred h | mean_succ h] comes from h and from the means the forward pass kept. The
// accumulators stay in TMEM across tiles (128 columns per 128 features); db_part = column
// sums of dZ in a fixed order. Bound by reading A, dh and h_out once: 512 threads keep 24
// 16-byte loads each in flight. 110,000 nodes: 636 -> 62 us a 128-wide layer (128 threads
// gathered the means again and transposed through 2-byte stores), the first 518 -> 35.
template <int KIN>
__global__ void __launch_bounds__(kBwdThreads) k_gnn_bwd_dw(GnnGraph g, const uint16_t *__restrict__ h_in,
                                                            const uint16_t *__restrict__ agg,
                                                            const uint16_t *__restrict__ h_out,
                                                            const float *__restrict__ dh_out, float *part,
                                                            int64_t w_off, int64_t b_off, int32_t *err) {
    constexpr int K = 3 * KIN;
    constexpr int S = (K + 127) / 128, KP = S * 128;  // feature slices of 128; features padded with zeros
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    __shared__ float sdb[32][kHidden];
    unsigned char *sA = sm;                 // [128 nodes x KP features] bf16
    unsigned char *sZ = sm + 128 * KP * 2;  // [128 nodes x 128 outputs] bf16
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    if (KP > K)
        for (int i = t; i < 128 * KP * 2 / 16; i += kBwdThreads) ((uint4 *)sA)[i] = make_uint4(0, 0, 0, 0);
    if (w == 0) tmem_alloc(&tslot, S * 128 <= 128 ? 128 : 512);
    if (t == 0) mbar_init1(&bar);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t taddr = tslot;
    const int64_t n_tiles = (g.n_nodes + 127) / 128;
    uint32_t phase = 0;
    bool ok = true, first = true;
    float db[8];
#pragma unroll
    for (int j = 0; j < 8; j++) db[j] = 0.f;
    for (int64_t tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
        constexpr int C = K / 8, N_IT = (128 * C + kBwdThreads - 1) / kBwdThreads, U = N_IT < 6 ? N_IT : 6;  // 16-byte pieces
        static_assert(N_IT % U == 0, "whole batches of pieces");
        for (int i0 = 0; i0 < N_IT; i0 += U) {
            uint4 x[U];
#pragma unroll
            for (int i = 0; i < U; i++) {
                int r, c;
                tile_piece<C>(i0 + i, kBwdThreads / 32, w, lane, r, c);
                const int64_t v = tile * 128 + r;
                x[i] = make_uint4(0, 0, 0, 0);
                if (r < 128 && v < g.n_nodes)
                    x[i] = c < KIN / 8 ? __ldg((const uint4 *)(h_in + v * KIN) + c)
                                       : __ldg((const uint4 *)(agg + v * 2 * KIN) + c - KIN / 8);
            }
#pragma unroll
            for (int i = 0; i < U; i++) {
                int r, c;
                tile_piece<C>(i0 + i, kBwdThreads / 32, w, lane, r, c);
                if (r < 128) *(uint4 *)(sA + kmajor_off(r, 8 * c, KP)) = x[i];
            }
        }
        stage_dz(g, h_out, dh_out, tile, sZ, t, db);
        fence_async_smem();
        __syncthreads();
        if (t == 0) {
            tmem_fence_after();
            for (int s = 0; s < S; s++)
                umma_gemm_tn(taddr + s * 128, sA + s * 16 * 128, KP, sZ, kHidden, 128, kHidden, !first);
            umma_commit(&bar);
        }
        first = false;
        ok = __syncthreads_and(mbar_wait_parity(&bar, phase, kWaitLimit)) != 0;  // uniform across the CTA
        phase ^= 1;
        tmem_fence_after();
    }
    if (!ok && t == 0 && err) atomicExch(err, DAGRT_E_TIMEOUT);
    float *pw = part + (int64_t)blockIdx.x * ParamLayout::total;
    const int lq = w & 3, c0 = 32 * (w >> 2);  // TMEM lane quarter and 32-column block
    for (int s = 0; s < S; s++) {
        float acc[32];
        if (!first && ok) tmem_ld32(taddr + ((uint32_t)(32 * lq) << 16) + s * 128 + c0, acc);
        else
            for (int i = 0; i < 32; i++) acc[i] = 0.f;
        const int feat = s * 128 + 32 * lq + lane;  // TMEM lane = feature
        if (feat < K) {
            float4 *dst = (float4 *)(pw + w_off + (int64_t)feat * kHidden + c0);
#pragma unroll
            for (int i = 0; i < 8; i++) dst[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; j++) sdb[dz_row(t)][dz_out(t) + j] = db[j];
    tmem_fence_before();
    __syncthreads();
    if (t < kHidden) {
        float s = 0.f;
        for (int i = 0; i < 32; i++) s += sdb[i][t];
        pw[b_off + t] = s;
    }
    if (w == 0) tmem_dealloc(taddr, S * 128 <= 128 ? 128 : 512);
}

template <int KIN>
static cudaError_t launch_dw(int layer, GnnGraph g, const uint16_t *h_in, const uint16_t *agg, const uint16_t *h_out,
                             const float *dh_out, float *part, int n_parts, int32_t *err, cudaStream_t st) {
    const int64_t woff[3] = {ParamLayout::W1, ParamLayout::W2, ParamLayout::W3};
    const int64_t boff[3] = {ParamLayout::b1, ParamLayout::b2, ParamLayout::b3};
    constexpr int KP = (3 * KIN + 127) / 128 * 128;
    const int smem = 128 * KP * 2 + kZBytes;
    cudaError_t e = cudaFuncSetAttribute(k_gnn_bwd_dw<KIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_gnn_bwd_dw<KIN><<<n_parts, kBwdThreads, smem, st>>>(g, h_in, agg, h_out, dh_out, part, woff[layer], boff[layer], err);
    return cudaGetLastError();
}

cudaError_t gnn_layer_bwd_dw(int kin, int layer, GnnGraph g, const uint16_t *h_in, const uint16_t *agg,
                             const uint16_t *h_out, const float *dh_out, float *part, int n_parts, int32_t *err,
                             cudaStream_t st) {
    if (kin == kFeat) return launch_dw<kFeat>(layer, g, h_in, agg, h_out, dh_out, part, n_parts, err, st);
    return launch_dw<kHidden>(layer, g, h_in, agg, h_out, dh_out, part, n_parts, err, st);
}

// dA = dZ W^T per 128-row tile: A operand dZ [rows x H], B operand W [K x H] (resident),
// three 128-column TMEM blocks for K = 384. Bound by writing dA (1.5 KB a node): every thread
// writes 128 contiguous bytes of its row per 32 columns, and 512 threads stage the next dZ
// while others still write. 110,000 nodes: 380 -> 70 us (128 threads, 4-byte stores).
template <int KIN>
__global__ void __launch_bounds__(kBwdThreads) k_gnn_bwd_da(GnnGraph g, const uint16_t *__restrict__ h_out,
                                                            const float *__restrict__ dh_out,
                                                            const uint16_t *__restrict__ wb, float *da, int32_t *err) {
    constexpr int K = 3 * KIN;
    constexpr int S = K / 128;
    static_assert(K % 128 == 0, "whole 128-column blocks");
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    unsigned char *sB = sm;                    // W [K x H] as B operand rows
    unsigned char *sZ = sm + K * kHidden * 2;  // dZ [128 x H]
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    for (int i = t; i < K * (kHidden / 8); i += kBwdThreads) {
        const int r = i / (kHidden / 8), kc = (i % (kHidden / 8)) * 8;
        *(uint4 *)(sB + kmajor_off(r, kc, kHidden)) = *(const uint4 *)(wb + (size_t)r * kHidden + kc);
    }
    if (w == 0) tmem_alloc(&tslot, 512);
    if (t == 0) mbar_init1(&bar);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t taddr = tslot;
    const int64_t n_tiles = (g.n_nodes + 127) / 128;
    const int lq = w & 3, cb = w >> 2;  // TMEM lane quarter and 32-column block of each 128
    uint32_t phase = 0;
    bool ok = true;
    float db[8];  // not used here
#pragma unroll
    for (int j = 0; j < 8; j++) db[j] = 0.f;
    for (int64_t tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
        stage_dz(g, h_out, dh_out, tile, sZ, t, db);
        fence_async_smem();
        __syncthreads();
        if (t == 0) {
            tmem_fence_after();
            for (int s = 0; s < S; s++)
                umma_gemm(taddr + s * 128, sZ, sB + s * 128 * kHidden * 2, kHidden, 128, false);
            umma_commit(&bar);
        }
        ok = __syncthreads_and(mbar_wait_parity(&bar, phase, kWaitLimit)) != 0;  // uniform across the CTA
        phase ^= 1;
        tmem_fence_after();
        if (ok) {
            const int64_t v = tile * 128 + 32 * lq + lane;
            for (int s = 0; s < S; s++) {
                float acc[32];
                tmem_ld32(taddr + ((uint32_t)(32 * lq) << 16) + s * 128 + 32 * cb, acc);
                if (v < g.n_nodes) {
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        uint32_t x[8];
#pragma unroll
                        for (int j = 0; j < 8; j++) x[j] = __float_as_uint(acc[8 * i + j]);
                        st32(da + v * K + s * 128 + 32 * cb + 8 * i, x);
                    }
                }
            }
        } else if (t == 0 && err) {
            atomicExch(err, DAGRT_E_TIMEOUT);
        }
        // no barrier here: each thread goes on to its part of the next dZ tile (the MMA that
        // read this one has completed); the barrier after that fill orders these TMEM reads
        // before the next MMA
        tmem_fence_before();
    }
    __syncthreads();  // every thread has read TMEM before it is released
    if (w == 0) tmem_dealloc(taddr, 512);
}

cudaError_t gnn_layer_bwd_da(int kin, GnnGraph g, const uint16_t *h_out, const float *dh_out, const uint16_t *wb,
                             float *da, int32_t *err, int n_sm, cudaStream_t st) {
    if (kin != kHidden) return cudaErrorInvalidValue;  // the first layer's input needs no gradient
    const int smem = 3 * kHidden * kHidden * 2 + kZBytes;
    cudaError_t e = cudaFuncSetAttribute(k_gnn_bwd_da<kHidden>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int64_t n_tiles = (g.n_nodes + 127) / 128;
    int grid = (int)(n_tiles < n_sm ? n_tiles : n_sm);
    if (grid < 1) return cudaSuccess;
    k_gnn_bwd_da<kHidden><<<grid, kBwdThreads, smem, st>>>(g, h_out, dh_out, wb, da, err);
    return cudaGetLastError();
}

// dh_in[u] = dA_self[u] + sum_{v in succ(u)} dA_pred[v] / indeg(v)
//                       + sum_{w in pred(u)} dA_succ[w] / outdeg(w)
// One warp per node, four features (16 bytes) per lane, four neighbours' rows in flight; the
// sum keeps its order. x / n is x (1/n) with one Newton step on the remainder, which rounds
// like the division (Markstein, "Computation of elementary functions on the IBM RISC
// System/6000", 1990) for normal x and quotients. An infinite x leaves a remainder of NaN, which the
// maximum drops: x / n stays infinite. (A branch to a division for such x: a training step on 1,000
// DAGs of 20-200 nodes 982 -> 1,037 us.) Bound by the rows it gathers from L2
// (512 bytes per edge and direction). 110,000 nodes, 740,000 edges: 277 -> 105 us.
__device__ __forceinline__ void add_div(float4 &s, float4 x, float n) {
    const float r = __frcp_rn(n);
    auto div = [&](float a) {
        const float q = a * r;
        return fmaf(fmaxf(fmaf(-n, q, a), -FLT_MAX), r, q);
    };
    s.x += div(x.x);
    s.y += div(x.y);
    s.z += div(x.z);
    s.w += div(x.w);
}

template <int KIN>
__global__ void __launch_bounds__(256) k_gnn_agg_bwd(GnnGraph g, const float *__restrict__ da, float *dh_in) {
    constexpr int K = 3 * KIN;
    static_assert(KIN == 128, "four features per lane");
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < g.n_nodes; u += warps) {
        float4 s = __ldg((const float4 *)(da + u * K) + lane);
        auto gather = [&](const int2 *__restrict__ list, const int32_t *__restrict__ idx,
                          const int2 *__restrict__ nlist, int third) {
            const int b = list[u].x, e = list[u].y;
            for (int i = b; i < e; i += 4) {
                float4 x[4];
                float n[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    if (i + j >= e) break;
                    const int64_t v = __ldg(idx + i + j);
                    const int2 nl = __ldg(nlist + v);
                    n[j] = (float)(nl.y - nl.x);
                    x[j] = __ldg((const float4 *)(da + v * K + third * KIN) + lane);
                }
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    if (i + j >= e) break;
                    add_div(s, x[j], n[j]);
                }
            }
        };
        gather(g.succ, g.succ_idx, g.pred, 1);
        gather(g.pred, g.pred_idx, g.succ, 2);
        *((float4 *)(dh_in + u * KIN) + lane) = s;
    }
}

cudaError_t gnn_agg_bwd(int kin, GnnGraph g, const float *da, float *dh_in, int n_sm, cudaStream_t st) {
    if (kin != kHidden) return cudaErrorInvalidValue;
    int64_t grid = (g.n_nodes + 7) / 8;
    if (grid > 32 * n_sm) grid = 32 * n_sm;
    if (grid < 1) return cudaSuccess;
    k_gnn_agg_bwd<kHidden><<<(int)grid, 256, 0, st>>>(g, da, dh_in);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ Adam
__global__ void k_gnn_adam(float *p, float *m, float *v, const float *part, int n_parts, int64_t n, float lr,
                           float b1, float b2, float eps, float c1, float c2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float gsum = 0.f;
        for (int c = 0; c < n_parts; c++) gsum += part[(int64_t)c * n + i];
        const float mi = b1 * m[i] + (1.f - b1) * gsum;
        const float vi = b2 * v[i] + (1.f - b2) * gsum * gsum;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

cudaError_t gnn_adam(float *p, float *m, float *v, const float *part, int n_parts, int64_t n, float lr, float b1,
                     float b2, float eps, int step, cudaStream_t st) {
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_gnn_adam<<<(int)((n + 255) / 256), 256, 0, st>>>(p, m, v, part, n_parts, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

// bf16 copies: W^T [H x K] (forward B operand) and W [K x H] (backward B operand)
__global__ void k_gnn_refresh(const float *p, uint16_t *wt1, uint16_t *wt2, uint16_t *wt3, uint16_t *wb1,
                              uint16_t *wb2, uint16_t *wb3) {
    const int64_t woff[3] = {ParamLayout::W1, ParamLayout::W2, ParamLayout::W3};
    const int Ks[3] = {3 * kFeat, 3 * kHidden, 3 * kHidden};
    uint16_t *wt[3] = {wt1, wt2, wt3}, *wb[3] = {wb1, wb2, wb3};
    for (int l = 0; l < 3; l++) {
        const int K = Ks[l];
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)K * kHidden;
             i += (int64_t)gridDim.x * blockDim.x) {
            const int k = (int)(i / kHidden), o = (int)(i % kHidden);
            const uint16_t b = f2bf(p[woff[l] + i]);
            wb[l][i] = b;
            wt[l][(int64_t)o * K + k] = b;
        }
    }
}

cudaError_t gnn_refresh(const float *p, uint16_t *const *wt, uint16_t *const *wb, cudaStream_t st) {
    k_gnn_refresh<<<96, 256, 0, st>>>(p, wt[0], wt[1], wt[2], wb[0], wb[1], wb[2]);
    return cudaGetLastError();
}

}  // namespace dagrt

namespace dagrt {

// ------------------------------------------------------------------ top-k decode
// The network gives each node an independent distribution over levels. The k most likely
// joint assignments: start from every node's best level; any other assignment changes some
// nodes to other levels, costing delta = z_best - z_alt each (log-probability loss). Only
// the k-1 smallest deltas can appear among the k best (an assignment using a larger one is
// matched or beaten by the all-best assignment and the k-1 single changes), so the search
// runs over those items, grouped by node (at most one change per node). Groups are ordered
// by their smallest delta, options within a group ascending; a state (group g, option j,
// earlier groups fixed) has the successors: next option of g; keep g and take option 0 of
// g+1; and, from option 0 only, drop g and take option 0 of g+1. Every assignment has one
// parent and no successor is cheaper, so a best-first walk pops the k best in order.
// One CTA per DAG; column 0 of every row keeps the paper's allocation (0), column 1 + j
// holds the j-th best assignment.
//
// The kTopkMax - 1 smallest (delta, node, level) of a thread's nodes stay sorted in registers
// as one 64-bit key each (a delta is not negative, so its bits order like it); the CTA merges
// them by argmin over the threads' heads; one thread walks. A row is written as two 16-byte
// stores, and only rows of the few nodes that some assignment changes look at the masks.
// Bound by latency: 300 DAGs of 100-1,000 nodes, 857 -> 53 us (a warp per DAG, sorted lists in
// local memory, a test of every change for every byte).
constexpr int kTopkMax = 16;
constexpr int kTopkThreads = 128;
static_assert(kTopkMax + 1 <= 32, "a row's candidates fit its 32 bytes");

template <int K1>
__device__ __forceinline__ void topk_insert(uint64_t (&best)[K1], uint64_t x) {
#pragma unroll
    for (int i = 0; i < K1; i++) {  // x sinks to its place, the last key falls out
        const bool lt = x < best[i];
        const uint64_t y = best[i];
        best[i] = lt ? x : y;
        x = lt ? y : x;
    }
}

__global__ void __launch_bounds__(kTopkThreads) k_gnn_topk(int32_t n_dags, const int64_t *node_off, const float *logits,
                                                  int L, const uint8_t *levels, int k, const uint4 *plan,
                                                  const int32_t *nrows, uint8_t *best_level, uint8_t *m_alloc,
                                                  int64_t stride) {
    constexpr int KM = kTopkMax - 1;
    __shared__ uint64_t s_key[KM];
    __shared__ uint64_t s_red[kTopkThreads / 32];
    __shared__ float s_dv[KM];
    __shared__ int32_t s_dn[KM];
    __shared__ uint8_t s_dl[KM];
    __shared__ uint32_t s_mask[kTopkMax];
    __shared__ int s_nc;
    __shared__ float s_hc[3 * kTopkMax + 1];
    __shared__ uint32_t s_hm[3 * kTopkMax + 1];
    __shared__ uint8_t s_hg[3 * kTopkMax + 1], s_hj[3 * kTopkMax + 1], s_lev[kMaxLevels];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int K1 = k - 1;
    if (tid < L) s_lev[tid] = levels[tid];
    for (int d = blockIdx.x; d < n_dags; d += gridDim.x) {
        const int64_t n0 = node_off[d];
        const int V = (int)(node_off[d + 1] - n0);
        uint64_t best[KM];
#pragma unroll
        for (int i = 0; i < KM; i++) best[i] = KEY_INF;
        for (int v = tid; v < V; v += kTopkThreads) {
            const float *zp = logits + (n0 + v) * L;
            float z[kMaxLevels];
#pragma unroll
            for (int l = 0; l < kMaxLevels; l++) z[l] = l < L ? __ldg(zp + l) : 0.f;
            int b = 0;
            float zb = z[0];
#pragma unroll
            for (int l = 1; l < kMaxLevels; l++)
                if (l < L && z[l] > zb) {
                    b = l;
                    zb = z[l];
                }
            best_level[n0 + v] = (uint8_t)b;
            if (K1 == 0) continue;
#pragma unroll
            for (int l = 0; l < kMaxLevels; l++) {
                if (l >= L || l == b) continue;
                // (delta, node, level); a sum with +0 makes a -0 a +0
                const uint64_t key = ((uint64_t)__float_as_uint(zb - z[l] + 0.f) << 32) | ((uint32_t)v << 8) | (uint32_t)l;
                if (key < best[KM - 1]) topk_insert(best, key);
            }
        }
        // merge: the K1 smallest over all threads, an argmin over their heads at a time
        int m = 0;
        for (; m < K1; m++) {
            uint64_t x = best[0];
            for (int o = 16; o > 0; o >>= 1) {
                const uint64_t y = __shfl_xor_sync(FULL, x, o);
                x = y < x ? y : x;
            }
            if (lane == 0) s_red[w] = x;
            __syncthreads();
            x = s_red[0];
#pragma unroll
            for (int i = 1; i < kTopkThreads / 32; i++) x = s_red[i] < x ? s_red[i] : x;
            if (x == KEY_INF) break;  // every list is exhausted
            if (best[0] == x) {  // keys are distinct: one thread moves on
#pragma unroll
                for (int i = 0; i + 1 < KM; i++) best[i] = best[i + 1];
                best[KM - 1] = KEY_INF;
                s_key[m] = x;
            }
            __syncthreads();
        }
        __syncthreads();
        if (tid == 0) {
            // group-major order: groups in order of first appearance (= smallest delta)
            int gs[kTopkMax], gc[kTopkMax], G = 0, q = 0;
            uint32_t used = 0;
            for (int i = 0; i < m; i++) {
                if (used >> i & 1) continue;
                const uint32_t ni = (uint32_t)s_key[i] >> 8;
                gs[G] = q;
                gc[G] = 0;
                for (int j = i; j < m; j++)
                    if (!(used >> j & 1) && (uint32_t)s_key[j] >> 8 == ni) {
                        used |= 1u << j;
                        s_dv[q] = __uint_as_float((uint32_t)(s_key[j] >> 32));
                        s_dn[q] = (int32_t)ni;
                        s_dl[q] = (uint8_t)s_key[j];
                        q++;
                        gc[G]++;
                    }
                G++;
            }
            // best-first walk: heap entries (cost, mask of chosen items, group, option)
            int hn = 0, nc = 0;
            s_mask[nc++] = 0;  // the all-best assignment
            if (G > 0) {
                s_hc[0] = s_dv[0];
                s_hm[0] = 1u;
                s_hg[0] = 0;
                s_hj[0] = 0;
                hn = 1;
            }
            while (nc < k && hn > 0) {
                int bi = 0;
                float c = s_hc[0];
                uint32_t msk = s_hm[0];
                for (int i = 1; i < hn; i++) {
                    const float ci = s_hc[i];
                    const uint32_t mi = s_hm[i];
                    if (ci < c || (ci == c && mi < msk)) {
                        bi = i;
                        c = ci;
                        msk = mi;
                    }
                }
                const int g = s_hg[bi], j = s_hj[bi];
                hn--;
                s_hc[bi] = s_hc[hn];
                s_hm[bi] = s_hm[hn];
                s_hg[bi] = s_hg[hn];
                s_hj[bi] = s_hj[hn];
                s_mask[nc++] = msk;
                const int it = gs[g] + j;
                auto push = [&](float cost, uint32_t mask, int gg, int jj) {
                    s_hc[hn] = cost;
                    s_hm[hn] = mask;
                    s_hg[hn] = (uint8_t)gg;
                    s_hj[hn] = (uint8_t)jj;
                    hn++;
                };
                if (j + 1 < gc[g])  // next option of group g
                    push(c - s_dv[it] + s_dv[it + 1], (msk & ~(1u << it)) | (1u << (it + 1)), g, j + 1);
                if (g + 1 < G) {
                    const int nx = gs[g + 1];
                    push(c + s_dv[nx], msk | (1u << nx), g + 1, 0);  // keep g, add group g+1
                    if (j == 0) push(c - s_dv[it] + s_dv[nx], (msk & ~(1u << it)) | (1u << nx), g + 1, 0);  // swap
                }
            }
            s_nc = nc;
        }
        __syncthreads();
        const int nc = s_nc;
        const int rows = nrows[d];
        const int64_t rbase = 2 * n0;
        for (int r = tid; r < rows; r += kTopkThreads) {
            const int node = (int)plan[rbase + r].w;
            uint32_t hit = 0;  // changes of this node
            for (int i = 0; i < m; i++) hit |= (uint32_t)(s_dn[i] == node) << i;
            const uint32_t lb = s_lev[best_level[n0 + node]];
            uint32_t out[8];
#pragma unroll
            for (int i = 0; i < 8; i++) out[i] = lb * 0x01010101u;
            out[0] &= ~0xffu;
            if (hit) {
                // mostly one change: byte 1 + j of the row for every assignment that has it
#pragma unroll
                for (int j = 0; j < kTopkMax; j++) {
                    const uint32_t x = s_mask[j < nc ? j : 0] & hit;
                    if (x && j < k) {
                        const uint32_t lv = s_lev[s_dl[31 - __clz(x)]];
                        out[(1 + j) >> 2] = (out[(1 + j) >> 2] & ~(0xffu << (8 * ((1 + j) & 3)))) | (lv << (8 * ((1 + j) & 3)));
                    }
                }
            }
            uint4 *dst = (uint4 *)(m_alloc + (rbase + r) * stride);
            dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
            dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
        }
        __syncthreads();  // the DAG's lists are read
    }
}

cudaError_t gnn_topk(int32_t n_dags, const int64_t *node_off, const float *logits, int n_levels,
                     const uint8_t *levels, int k, const uint4 *plan, const int32_t *nrows, uint8_t *best_level,
                     uint8_t *m_alloc, int64_t stride, int n_sm, cudaStream_t st) {
    if (n_dags == 0) return cudaSuccess;
    if (k < 1 || k > kTopkMax || stride % 16 != 0 || stride < 32) return cudaErrorInvalidValue;
    const int grid = n_dags < 32 * n_sm ? n_dags : 32 * n_sm;
    k_gnn_topk<<<grid, kTopkThreads, 0, st>>>(n_dags, node_off, logits, n_levels, levels, k, plan, nrows, best_level,
                                              m_alloc, stride);
    return cudaGetLastError();
}

// the winning candidate's allocation, row by row (one CTA per DAG)
__global__ void k_pick_column(int32_t n_dags, const int64_t *node_off, const int32_t *nrows, const int32_t *best,
                              const uint8_t *m_alloc, int64_t stride, uint8_t *out) {
    for (int d = blockIdx.x; d < n_dags; d += gridDim.x) {
        const int c = best[d];
        const int64_t rbase = 2 * node_off[d];
        for (int r = threadIdx.x; r < nrows[d]; r += blockDim.x) out[rbase + r] = c >= 0 ? m_alloc[(rbase + r) * stride + c] : 0;
    }
}

cudaError_t gnn_pick_column(int32_t n_dags, const int64_t *node_off, const int32_t *nrows, const int32_t *best,
                            const uint8_t *m_alloc, int64_t stride, uint8_t *out, int n_sm, cudaStream_t st) {
    if (n_dags == 0) return cudaSuccess;
    const int grid = n_dags < 32 * n_sm ? n_dags : 32 * n_sm;
    k_pick_column<<<grid, 128, 0, st>>>(n_dags, node_off, nrows, best, m_alloc, stride, out);
    return cudaGetLastError();
}

}  // namespace dagrt
