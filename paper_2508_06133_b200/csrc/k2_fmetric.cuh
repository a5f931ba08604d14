// K2 -- F-metric batch selection over a sorted list (Algorithm 1, Phase 1, restricted to prefixes).
//
// Section 3: F(X) = (sum of o over X) / |X|^2; the batch with the smallest F is taken next, ties go
// to the larger batch.  Candidates here are the prefixes of the not-yet-selected requests in
// ascending (s+o, o, index) order (the order Algorithm 3 builds its first batch from), subject to
// Algorithms 2/3/4's memory test  sum (s_i + o_i) <= M.  With inclusive prefix sums P (of s+o) and
// O (of o) over the sorted list, the batch that starts at offset a is
//     k_max = max { k : P[a+k] - P[a] <= M },    k* = argmin_{1 <= k <= k_max} (O[a+k] - O[a]) / k^2,
// and the next batch starts at a + k*.  F values are compared exactly: A/ka^2 < B/kb^2 iff
// A*kb^2 < B*ka^2, evaluated on 128-bit products (on 64-bit ones
// where sum(o) n^2 < 2^63 says that they cannot overflow).
//
// One CTA: the batches depend on each other, so what counts is the latency of one batch.  Up to about
// 14,000 requests the prefix sums stay in shared memory; k_max is found by 32-way votes (3 turns for
// 10,000 requests, a binary search takes 14); a batch of up to 256 candidates is chosen by every warp
// for itself, without a barrier.
#pragma once

#include "common.cuh"

// true iff batch (sumA, kA) is strictly preferred to (sumB, kB); kB == 0 means "no batch yet".
__device__ __forceinline__ bool k2_f_better(u64 sumA, u64 kA, u64 sumB, u64 kB) {
    if (kA == 0) return false;
    if (kB == 0) return true;
    const u64 a2 = kA * kA, b2 = kB * kB;
    const u64 l_hi = __umul64hi(sumA, b2), l_lo = sumA * b2;
    const u64 r_hi = __umul64hi(sumB, a2), r_lo = sumB * a2;
    if (l_hi != r_hi) return l_hi < r_hi;
    if (l_lo != r_lo) return l_lo < r_lo;
    return kA > kB;
}

template <bool kWide>
__device__ __forceinline__ bool k2_better(u64 sumA, u64 kA, u64 sumB, u64 kB) {
    if (kWide) return k2_f_better(sumA, kA, sumB, kB);
    if (kA == 0) return false;
    if (kB == 0) return true;
    const u64 l = sumA * kB * kB, r = sumB * kA * kA;
    return l != r ? l < r : kA > kB;
}

#define K2_THREADS 512
#define K2_PER_THREAD 4
#define K2_SOLO 256                        // candidates up to which every warp decides for itself

// P[0] = O[0] = 0, P[q+1] = P[q] + (s+o of ids[q]), O[q+1] = O[q] + weight; the weight is o, or
// a_num * s + a_den * o with Section 7's prefill weight alpha = a_num / a_den.
__device__ void k2_prefix_sums(const int* __restrict__ s, const int* __restrict__ o, const int* __restrict__ ids, int n,
                               i64* P, i64* O, i64* sh_warp /* [2 * 32] */, i64 a_num, i64 a_den) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int W = K2_THREADS / 32, E = K2_PER_THREAD, TILE = K2_THREADS * E;
    i64 ct = 0, co = 0;
    if (tid == 0) { P[0] = 0; O[0] = 0; }
    int id[E];
#pragma unroll
    for (int e = 0; e < E; ++e) id[e] = tid * E + e < n ? ids[tid * E + e] : -1;
    for (int base = 0; base < n; base += TILE) {
        i64 vt[E], vo[E], it = 0, io = 0;
        int next[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int q = base + TILE + tid * E + e;
            next[e] = q < n ? ids[q] : -1;
            const int si = id[e] >= 0 ? s[id[e]] : 0, oi = id[e] >= 0 ? o[id[e]] : 0;
            it += (i64)si + oi; io += a_num * si + a_den * oi;
            vt[e] = it; vo[e] = io;
        }
        i64 st = it, so = io;
        for (int d = 1; d < 32; d <<= 1) {
            const i64 yt = __shfl_up_sync(KV_FULL, st, d), yo = __shfl_up_sync(KV_FULL, so, d);
            if (lane >= d) { st += yt; so += yo; }
        }
        if (lane == 31) { sh_warp[w] = st; sh_warp[32 + w] = so; }
        __syncthreads();
        i64 bt = ct + st - it, bo = co + so - io;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const i64 x = sh_warp[k], y = sh_warp[32 + k];
            if (k < w) { bt += x; bo += y; }
            ct += x; co += y;
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int q = base + tid * E + e;
            if (q < n) { P[q + 1] = bt + vt[e]; O[q + 1] = bo + vo[e]; }
            id[e] = next[e];
        }
        __syncthreads();
    }
}

template <bool kWide>
__device__ __forceinline__ void k2_reduce(u64& bs, u64& bk) {
    for (int d = 16; d >= 1; d >>= 1) {
        const u64 os = __shfl_xor_sync(KV_FULL, bs, d), ok = __shfl_xor_sync(KV_FULL, bk, d);
        if (k2_better<kWide>(os, ok, bs, bk)) { bs = os; bk = ok; }
    }
}

// Batch boundaries by the rule above.  Writes batch_off[0..nb] and returns nb (same in all
// threads).  sh_best: 2 * 32 + 1 shared 64-bit words.
template <bool kWide>
__device__ int k2_select_batches(const i64* P, const i64* O, int n, i64 M, int* batch_off, u64* sh_best) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int W = K2_THREADS / 32;
    int a = 0, nb = 0;
    if (tid == 0) batch_off[0] = 0;
    while (a < n) {
        // k_max: P is ascending; every warp narrows [lo, hi] to a 32nd per turn
        int lo = 1, hi = n - a;                     // P[a + lo] - P[a] <= M: every request fits on its own
        const i64 Pa = P[a], Oa = O[a];
        while (lo < hi) {
            const int step = (hi - lo + 31) >> 5, k = lo + (lane + 1) * step;
            const unsigned fits = __ballot_sync(KV_FULL, k <= hi && P[a + k] - Pa <= M);
            const int c = __popc(fits);             // a prefix of the lanes
            hi = min(hi, lo + (c + 1) * step - 1);
            lo = lo + c * step;
        }
        const int kmax = lo;
        u64 bs = 0, bk = 0;
        const bool solo = kmax <= K2_SOLO;
        for (int k = 1 + (solo ? lane : tid); k <= kmax; k += solo ? 32 : K2_THREADS) {
            const u64 sum = (u64)(O[a + k] - Oa);
            if (k2_better<kWide>(sum, (u64)k, bs, bk)) { bs = sum; bk = (u64)k; }
        }
        k2_reduce<kWide>(bs, bk);
        if (!solo) {
            if (lane == 0) { sh_best[w] = bs; sh_best[32 + w] = bk; }
            __syncthreads();
            bs = lane < W ? sh_best[lane] : 0; bk = lane < W ? sh_best[32 + lane] : 0;
            k2_reduce<kWide>(bs, bk);
            __syncthreads();                        // sh_best may be written again
        }
        a += (int)bk;
        ++nb;
        if (tid == 0) batch_off[KV_IDX(nb, n + 1, 801)] = a;
    }
    return nb;
}

// One CTA: prefix sums over the sorted ids, then the batch loop.  P, O: global int64[n+1], or nullptr:
// in dynamic shared memory.
__global__ void __launch_bounds__(K2_THREADS)
k2_prefix_f(const int* __restrict__ s, const int* __restrict__ o, const int* __restrict__ sorted_ids,
            int n, i64 M, i64* P, i64* O,
            int* __restrict__ batch_off, int* __restrict__ num_batches, i64 a_num, i64 a_den) {
    extern __shared__ __align__(16) i64 k2_smem[];
    __shared__ i64 sh_warp[64];
    __shared__ u64 sh_best[64];
    if (!P) { P = k2_smem; O = k2_smem + n + 1; }
    k2_prefix_sums(s, o, sorted_ids, n, P, O, sh_warp, a_num, a_den);
    __syncthreads();
    const bool wide = (double)O[n] * (double)n * (double)n >= 9.0e18;
    const int nb = wide ? k2_select_batches<true>(P, O, n, M, batch_off, sh_best)
                        : k2_select_batches<false>(P, O, n, M, batch_off, sh_best);
    if (threadIdx.x == 0) *num_batches = nb;
}
