// dagrt_internal.cuh -- device-side building blocks shared by the libdagrt kernels.
//
// A "team" is the set of threads that cooperates on one DAG: one warp (several independent teams
// per CTA, sched_warp.cuh) or a whole CTA, here Team<NT>: NT == blockDim.x, workspace in shared or
// global memory.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "dagrt.h"

namespace dagrt {

constexpr uint64_t KEY_INF = ~0ull;
constexpr unsigned FULL = 0xffffffffu;

__host__ __device__ constexpr int ceil_div(int a, int b) { return (a + b - 1) / b; }
__host__ __device__ constexpr int64_t align_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

// ------------------------------------------------------------------ team
template <int NT>
struct Team {
    static constexpr int NW = NT / 32;
    int t;              // rank in team
    uint64_t *red;      // NW words of shared scratch

    __device__ __forceinline__ int lane() const { return t & 31; }
    __device__ __forceinline__ int warp() const { return t >> 5; }
    __device__ __forceinline__ void sync() const { __syncthreads(); }

    template <class Op>
    __device__ __forceinline__ uint64_t reduce(uint64_t v, Op op) const {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(FULL, v, o));
        if (lane() == 0) red[warp()] = v;
        __syncthreads();
        uint64_t r = red[0];
#pragma unroll
        for (int i = 1; i < NW; i++) r = op(r, red[i]);
        __syncthreads();
        return r;
    }
    __device__ __forceinline__ uint64_t sum(uint64_t v) const {
        return reduce(v, [](uint64_t a, uint64_t b) { return a + b; });
    }
    __device__ __forceinline__ uint64_t maxu(uint64_t v) const {
        return reduce(v, [](uint64_t a, uint64_t b) { return a > b ? a : b; });
    }
    __device__ __forceinline__ bool any(bool p) const { return __syncthreads_or(p) != 0; }

    // Inclusive scan of v across the team with an associative op; *total gets the
    // reduction of all values.
    template <class Op>
    __device__ __forceinline__ uint64_t incl_scan(uint64_t v, Op op, uint64_t *total) const {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint64_t x = __shfl_up_sync(FULL, v, o);
            if (lane() >= o) v = op(v, x);
        }
        if (lane() == 31) red[warp()] = v;
        __syncthreads();
        uint64_t carry = 0, tot = 0;
        bool have = false;
        for (int i = 0; i < NW; i++) {
            if (i == warp()) { carry = tot; have = i > 0; }
            tot = i == 0 ? red[0] : op(tot, red[i]);
        }
        __syncthreads();
        *total = tot;
        return have ? op(carry, v) : v;
    }
};

// In-place inclusive scan of arr[0..n) (team-wide, chunk by chunk with a carry); with
// `reverse` the scan runs from arr[n-1] down to arr[0]. Lanes past the end take part in
// the warp scan but sit after every real lane, so they never reach a real result.
template <int NT, class T, class Op>
__device__ void team_scan_inplace(const Team<NT> &tm, T *arr, int n, Op op, bool reverse) {
    uint64_t carry = 0;
    bool have = false;
    for (int base = 0; base < n; base += NT) {
        int i = base + tm.t;
        int idx = reverse ? n - 1 - i : i;
        uint64_t v = i < n ? (uint64_t)arr[idx] : 0;
        uint64_t tot;
        uint64_t s = tm.incl_scan(v, op, &tot);
        int last = min(n - base, NT) - 1;
        if (tm.t == last) tm.red[0] = s;
        __syncthreads();
        const uint64_t chunk_tot = tm.red[0];
        __syncthreads();
        if (i < n) arr[idx] = (T)(have ? op(carry, s) : s);
        carry = have ? op(carry, chunk_tot) : chunk_tot;
        have = true;
        tm.sync();
    }
}

// Bitonic network, strides j, j / 2, ..., jmin of the merge of runs of k, over keys[0..n) (n a
// power of two), which are the keys from `base` on of the sequence that is sorted. Two strides a
// pass: a thread takes four keys through both.
template <int NT>
__device__ __forceinline__ void team_bitonic_merge(const Team<NT> &tm, uint64_t *keys, int n, int base, int k, int j, int jmin) {
    auto order = [](uint64_t &x, uint64_t &y, bool up) {
        const uint64_t lo = x < y ? x : y, hi = x < y ? y : x;
        x = up ? lo : hi;
        y = up ? hi : lo;
    };
    while (j >= jmin) {
        const int h = j >> 1;
        if (h >= jmin) {
            for (int t = tm.t; t < n >> 2; t += NT) {
                const int i = (t & ~(h - 1)) << 2 | (t & (h - 1));
                const bool up = ((base + i) & k) == 0;
                uint64_t x0 = keys[i], x1 = keys[i + h], x2 = keys[i + 2 * h], x3 = keys[i + 3 * h];
                order(x0, x2, up);
                order(x1, x3, up);
                order(x0, x1, up);
                order(x2, x3, up);
                keys[i] = x0;
                keys[i + h] = x1;
                keys[i + 2 * h] = x2;
                keys[i + 3 * h] = x3;
            }
            j >>= 2;
        } else {
            for (int t = tm.t; t < n >> 1; t += NT) {
                const int i = (t & ~(j - 1)) << 1 | (t & (j - 1));
                uint64_t x0 = keys[i], x1 = keys[i + j];
                order(x0, x1, ((base + i) & k) == 0);
                keys[i] = x0;
                keys[i + j] = x1;
            }
            j >>= 1;
        }
        tm.sync();
    }
}

// Sorts keys[0..P) ascending, P a power of two. `buf`: shared memory for C keys (C a power of
// two; 0: the keys are in shared memory themselves), which takes every stride below C: what
// bounds the sort is the barrier and the latency of a pass, so passes over global memory are
// the few strides of C and above (32,768 keys by 384 threads: 4.9 -> 1.2 M cycles).
template <int NT>
__device__ void team_bitonic_sort(const Team<NT> &tm, uint64_t *keys, int P, uint64_t *buf = nullptr, int C = 0) {
    if (C == 0) {
        for (int k = 2; k <= P; k <<= 1) team_bitonic_merge(tm, keys, P, 0, k, k >> 1, 1);
        return;
    }
    C = min(C, P);
    for (int k0 = C; k0 <= P; k0 <<= 1) {
        if (k0 > C) team_bitonic_merge(tm, keys, P, 0, k0, k0 >> 1, C);
        for (int b = 0; b < P; b += C) {
            for (int i = tm.t; i < C; i += NT) buf[i] = keys[b + i];
            tm.sync();
            if (k0 == C)
                for (int k = 2; k <= C; k <<= 1) team_bitonic_merge(tm, buf, C, b, k, k >> 1, 1);
            else
                team_bitonic_merge(tm, buf, C, b, k0, C >> 1, 1);
            for (int i = tm.t; i < C; i += NT) keys[b + i] = buf[i];
            tm.sync();
        }
    }
}

// ------------------------------------------------------------------ programmatic launches
// A kernel launched with programmatic stream serialization starts once every CTA of the kernel
// before it has called the first of these or ended; the second waits until that kernel has
// completed and its stores are visible. Both do nothing in an ordinary launch.
__device__ __forceinline__ void griddep_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------ Eq.1
// Execution time of a kernel with load x (ticks on one SM) and parallel fraction k/64 on m
// of M SMs: max(1, ceil(ceil(m/M) * x * (64m - k(m-1)) / (64m))). Products stay below
// 2^62 for x < 2^32, m <= 4096, M >= 1.
__device__ __forceinline__ uint64_t exec_time(uint64_t x, uint32_t k, uint32_t m, uint32_t M) {
    uint32_t waves = m <= M ? 1u : (m + M - 1) / M;
    uint64_t a = 64ull * m - (uint64_t)k * (m - 1);
    uint64_t num = (uint64_t)waves * x * a;
    uint64_t den = 64ull * m;
    uint64_t c;
    if ((m & (m - 1)) == 0) {
        int sh = 6 + (31 - __clz(m));
        c = (num + den - 1) >> sh;
    } else if (num < (1ull << 32)) {
        c = ((uint32_t)num - 1u) / (uint32_t)den + 1u;  // num >= 64 > 0
    } else {
        c = (num + den - 1) / den;
    }
    return c < 1 ? 1 : c;
}

__device__ __forceinline__ uint64_t udiv(uint64_t n, uint64_t d) {  // 32-bit divide when both fit
    return (n >> 32) == 0 && (d >> 32) == 0 ? (uint64_t)((uint32_t)n / (uint32_t)d) : n / d;
}

// The largest dynamic shared memory a launch of `kern` may take on the current device: the
// opt-in maximum per block less the kernel's static shared memory (0 on error). Kernels
// whose launches use different sizes set their attribute to this, not to one launch's
// size: the attribute is per function, and a captured graph node launched on its own (as
// a profiler replays it) is checked against the attribute's current value.
template <class F>
inline int max_dynamic_smem(F *kern) {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, kern) != cudaSuccess)
        return 0;
    return optin - (int)fa.sharedSizeBytes;
}

}  // namespace dagrt
