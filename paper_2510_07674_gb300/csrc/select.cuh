// ArgSort(C)[:k] of Alg. 1 on the GPU: the k smallest costs, ordered by (cost, index).
//
// One CTA of 1024 threads:  (1) costs become order-preserving 32-bit keys in shared
// memory; (2) a 4-pass radix select (8 bits per pass, shared-memory histograms with
// integer atomics) finds the k-th smallest key T and how many keys equal to T are taken;
// (3) every key < T is gathered in any order and the lowest-index keys == T by ballots; (4) a
// bitonic sort of the k selected (key << 32 | index) pairs.  Integer work only, and the sort
// orders whatever the gathering left, so the result is deterministic and equals a stable sort by
// (cost, index).
// A latency-bound single CTA: the bucket of a pass is found by one warp's scan (a thread walking
// the 256 buckets took 3.7 us a pass, most of the time at a few hundred costs), the gathering
// reads consecutive keys (a contiguous run per thread met 16-way bank conflicts), and the sort
// keeps the pairs in registers: 63 of its 78 steps at 4096 stay inside a thread or a warp, the
// other 15 take nine passes through shared memory (every step through shared memory: 27 us at
// 4096 pairs, 10 us now).  n = 16384, k = 4096: 59.5 -> 30.8 us, of which the four passes over the
// keys 11 and the launch with its latency 8; n = 4096, k = 1024: 22.6 -> 14.4 us; n = 256, k = 64:
// 16.4 -> 8.2 us.
#pragma once
#include "common.cuh"

namespace spasm {

constexpr int kSelectThreads = 1024;

// NaN sorts last; -0 and +0 compare equal (both map to the key of +0).
__device__ __forceinline__ uint32_t cost_key(float c) {
    if (c != c) return 0xFFFFFFFFu;
    c = c + 0.0f;
    const uint32_t u = __float_as_uint(c);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Bitonic sort of kp2 pairs (ascending, a power of two; kp2 <= 1024 for E = 1, else kp2 = 1024 E) by the whole
// block.  Thread t keeps pairs t E .. t E + E - 1 in registers: exchanges over distances below E stay in the
// thread, below 32 E in the warp (shuffles); the longer ones go through shared memory two distances at a
// time, a barrier per pair of distances.  Leaves the sorted pairs in v (all ones beyond kp2).
template <int E>
__device__ __forceinline__ void sort_pairs(unsigned long long* pairs, int kp2, unsigned long long (&v)[E]) {
    const int t = threadIdx.x, nt = blockDim.x, total = kp2 < 32 ? 32 : kp2;
    const bool mine = t * E < total;   // uniform over a warp
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = t * E + e < kp2 ? pairs[t * E + e] : ~0ull;
    for (int size = 2; size <= total; size <<= 1) {
        int stride = size >> 1;
        if (stride >= 32 * E) {
            if (mine)
#pragma unroll
                for (int e = 0; e < E; ++e) pairs[t * E + e] = v[e];
            __syncthreads();
            for (; stride >= 64 * E; stride >>= 2) {
                const int half = stride >> 1;
                for (int i = t; i < total / 4; i += nt) {
                    const int base = 4 * i - 3 * (i & (half - 1));
                    const bool up = (base & size) == 0;
                    unsigned long long a = pairs[base], b = pairs[base + half];
                    unsigned long long c = pairs[base + stride], d = pairs[base + stride + half], x;
                    if ((a > c) == up) { x = a; a = c; c = x; }
                    if ((b > d) == up) { x = b; b = d; d = x; }
                    if ((a > b) == up) { x = a; a = b; b = x; }
                    if ((c > d) == up) { x = c; c = d; d = x; }
                    pairs[base] = a; pairs[base + half] = b;
                    pairs[base + stride] = c; pairs[base + stride + half] = d;
                }
                __syncthreads();
            }
            if (stride == 32 * E) {
                for (int i = t; i < total / 2; i += nt) {
                    const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                    const unsigned long long a = pairs[lo], b = pairs[hi];
                    if ((a > b) == ((lo & size) == 0)) { pairs[lo] = b; pairs[hi] = a; }
                }
                __syncthreads();
                stride >>= 1;
            }
            if (mine)
#pragma unroll
                for (int e = 0; e < E; ++e) v[e] = pairs[t * E + e];
        }
        if (!mine) continue;
        for (; stride >= E; stride >>= 1) {
            const int lanes = stride / E;
            const bool keep_min = ((t & lanes) == 0) == (((t * E) & size) == 0);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const unsigned long long o = __shfl_xor_sync(0xffffffffu, v[e], lanes);
                if ((o < v[e]) == keep_min) v[e] = o;
            }
        }
#pragma unroll
        for (int st = E / 2; st > 0; st >>= 1) {
            if (st > stride) continue;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (e & st) continue;
                const unsigned long long a = v[e], b = v[e + st];
                if ((a > b) == (((t * E + e) & size) == 0)) { v[e] = b; v[e + st] = a; }
            }
        }
    }
}

template <int E>
__device__ __forceinline__ void sort_and_write(unsigned long long* pairs, int kp2, int k, const float* __restrict__ cost,
                                               int* __restrict__ out_idx, float* __restrict__ out_cost) {
    unsigned long long v[E];
    sort_pairs<E>(pairs, kp2, v);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = (int)threadIdx.x * E + e;
        if (i >= k) continue;
        const int idx = (int)(uint32_t)(v[e] & 0xffffffffull);
        out_idx[i] = idx;
        if (out_cost) out_cost[i] = cost[idx];
    }
}

// keys (n) and pairs (kp2 >= k, power of two) live in dynamic shared memory; kp2 <= 8192.
__global__ void __launch_bounds__(kSelectThreads) k_topk(const float* __restrict__ cost, int n, int k,
                                                          int* __restrict__ out_idx, float* __restrict__ out_cost,
                                                          int kp2) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long* pairs = reinterpret_cast<unsigned long long*>(smem_raw);
    uint32_t* keys = reinterpret_cast<uint32_t*>(pairs + kp2);
    __shared__ int hist[256];   // a pass's buckets; then the keys == T of each warp
    __shared__ uint32_t s_prefix;
    __shared__ int s_need, s_equal, s_less_at, s_equal_at;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w = tid >> 5;
    if (k > n) k = n;

    for (int i = tid; i < n; i += nt) keys[i] = cost_key(cost[i]);
    if (tid == 0) { s_prefix = 0; s_need = k; s_equal = 0; s_less_at = 0; s_equal_at = 0; }
    __syncthreads();

    // radix select of the k-th smallest key (1-based rank k)
    uint32_t mask = 0;
    for (int shift = 24; shift >= 0 && k > 0; shift -= 8) {
        for (int i = tid; i < 256; i += nt) hist[i] = 0;
        __syncthreads();
        const uint32_t prefix = s_prefix;
        for (int i = tid; i < n; i += nt) {
            const uint32_t key = keys[i];
            if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1);
        }
        __syncthreads();
        if (w == 0) {   // the bucket that holds rank s_need: eight buckets per lane, a scan over the lanes
            int cnt[8], sum = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) { cnt[i] = hist[8 * lane + i]; sum += cnt[i]; }
            int below = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, below, off);
                if (lane >= off) below += up;
            }
            below -= sum;
            const int need = s_need;
            __syncwarp();
            if (below < need && need <= below + sum) {
                int bkt = 8 * lane;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (below < need && need <= below + cnt[i]) {
                        s_need = need - below;
                        s_equal = cnt[i];
                        s_prefix = prefix | ((uint32_t)(bkt + i) << shift);
                    }
                    below += cnt[i];
                }
            }
        }
        mask |= 255u << shift;
        __syncthreads();
    }
    const uint32_t T = s_prefix;
    const int need_eq = s_need;   // keys == T to take (lowest indices first)

    // gather: 1024 consecutive keys at a time
    const int n_sel_less = k > 0 ? k - need_eq : 0;
    const bool ordered = s_equal > need_eq;   // not every key == T is taken: the lowest indices are
    int eq_done = 0;
    for (int base = 0; k > 0 && base < n; base += nt) {
        const int i = base + tid;
        const uint32_t key = i < n ? keys[i] : 0xFFFFFFFFu;
        const unsigned less = __ballot_sync(0xffffffffu, i < n && key < T);
        const unsigned equal = __ballot_sync(0xffffffffu, i < n && key == T);
        const unsigned before = (1u << lane) - 1u;
        int at = 0;
        if (lane == 0 && less) at = atomicAdd(&s_less_at, __popc(less));
        at = __shfl_sync(0xffffffffu, at, 0);
        if ((less >> lane) & 1u) pairs[at + __popc(less & before)] = ((unsigned long long)key << 32) | (uint32_t)i;
        int eq_at = 0;
        if (ordered && eq_done < need_eq) {   // uniform over the block
            if (lane == 0) hist[w] = __popc(equal);
            __syncthreads();
            const int c = hist[lane];
            eq_at = __reduce_add_sync(0xffffffffu, lane < w ? c : 0) + eq_done;
            eq_done += __reduce_add_sync(0xffffffffu, c);
            __syncthreads();
        } else if (ordered) {
            continue;
        } else {
            if (lane == 0 && equal) eq_at = atomicAdd(&s_equal_at, __popc(equal));
            eq_at = __shfl_sync(0xffffffffu, eq_at, 0);
        }
        if ((equal >> lane) & 1u) {
            const int pos = eq_at + __popc(equal & before);
            if (pos < need_eq) pairs[n_sel_less + pos] = ((unsigned long long)key << 32) | (uint32_t)i;
        }
    }
    for (int i = k + tid; i < kp2; i += nt) pairs[i] = ~0ull;
    __syncthreads();

    if (kp2 <= 1024) sort_and_write<1>(pairs, kp2, k, cost, out_idx, out_cost);
    else if (kp2 == 2048) sort_and_write<2>(pairs, kp2, k, cost, out_idx, out_cost);
    else if (kp2 == 4096) sort_and_write<4>(pairs, kp2, k, cost, out_idx, out_cost);
    else sort_and_write<8>(pairs, kp2, k, cost, out_idx, out_cost);   // 8192
}

}  // namespace spasm
