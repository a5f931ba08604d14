// K2b -- Phase 1 of Sorted-F with Algorithm 3 (Local Swap Search, Section 5.2 / the supplement to Section 5) as the
// batch solver, all batches in one launch of one CTA (the batches depend on each other: each one
// is built from what the previous ones left).
//
// Algorithm 3 on the remaining requests, sorted by ascending s+o (ties: lower index):
//   first fit  -- in that order a request is taken iff it still fits; because the sizes ascend,
//                 the result is the longest prefix whose sum(s+o) <= M;
//   improvement -- walk r_out over X (insertion order, a swapped-in request keeps the place of the
//                 one it replaces) and r_in over the requests outside X (sorted order); the first
//                 pair with  mem + (s+o)_in - (s+o)_out <= M  and  F(X') < F(X)  is swapped and the
//                 walk starts over; |X| never changes, so F drops iff o_in < o_out (with Section 7's
//                 prefill weight alpha = a_num / a_den: iff a_num s_in + a_den o_in is smaller).
// The pair walk is not executed cell by cell.  For one r_out the admissible r_in are the outside
// requests among the first ub positions (sizes ascend: (s+o)_in <= cap is a prefix), and it has a
// partner iff the smallest weight outside X among those is below its own; all members are asked at
// once, the lowest one that has a partner wins (that is the pair the printed loops reach first), and
// its partner is the first outside position with a smaller weight.
//
// What bounds it: a chain of swaps (1,425 for the 2,000-request backlog of the paper's lengths), each
// of which needs the one before it, so the latency of one swap.  Hence:
//   - prefix minima in two levels, 32-position blocks (pin, written by one warp's shuffle scan) and
//     block totals (bpre): a swap changes two blocks, which warp 0 scans again, instead of the list;
//   - ub of every member is kept from the last turn and moved a few positions (the free memory changes
//     little from swap to swap) instead of searched for;
//   - the partner is found with two votes; two barriers per swap; every array in shared memory where
//     it fits.
#pragma once

#include "common.cuh"

#define K2L_THREADS 512
#define K2L_IN (1 << 30)                      // in id[]: the position belongs to X

// Scratch of one solver: the remaining list by position (ascending (s+o, index)) and what the swaps
// need.  IX: 16-bit where the positions fit.
template <typename IX>
struct K2lArrays {
    int *T, *O, *id;                          // size, weight, request id (| K2L_IN) by position
    int *pin;                                 // min weight outside X over the position's block, up to it
    int *bmin, *bpre;                         // per block: min weight outside X; bpre[b] = min over blocks < b
    IX *ub, *xpos;                            // per member in walking order: partners lie below ub; position
};

__host__ __device__ inline size_t k2l_blocks(int n) { return (size_t)((n + 31) / 32); }
template <typename IX>
__host__ __device__ inline size_t k2l_bytes(int n) {
    return (size_t)n * (4 * sizeof(int) + 2 * sizeof(IX)) + (2 * k2l_blocks(n) + 4) * sizeof(int) + 16;
}
template <typename IX>
__device__ __forceinline__ K2lArrays<IX> k2l_arrays(void* base, int n) {
    K2lArrays<IX> a;
    int* p = (int*)base;
    a.T = p; a.O = p + n; a.id = p + 2 * (size_t)n; a.pin = p + 3 * (size_t)n;
    a.bmin = p + 4 * (size_t)n; a.bpre = a.bmin + k2l_blocks(n) + 1;
    a.ub = (IX*)(a.bpre + k2l_blocks(n) + 2); a.xpos = a.ub + n;
    return a;
}

template <int THREADS>
struct K2lShared {
    static constexpr int W = THREADS / 32;
    i64 sum64[W];
    int cnt[W];
    int pick[2];
    int mem;
};

template <int THREADS>
__device__ __forceinline__ void k2l_sync() { if (THREADS == 32) __syncwarp(); else __syncthreads(); }

// min-scan of one 32-position block by one warp
template <typename IX>
__device__ __forceinline__ void k2l_scan_block(const K2lArrays<IX>& a, int m, int b, int lane) {
    const int p = 32 * b + lane;
    int v = (p < m && !(a.id[p] & K2L_IN)) ? a.O[p] : INT_MAX;
    for (int d = 1; d < 32; d <<= 1) { const int y = __shfl_up_sync(KV_FULL, v, d); if (lane >= d) v = min(v, y); }
    if (p < m) a.pin[p] = v;
    if (lane == 31) a.bmin[b] = v;
}

// bpre[b + 1] = min(bmin[0 .. b]) for the blocks from the 32-group of `first` on, by one warp
template <typename IX>
__device__ __forceinline__ void k2l_scan_totals(const K2lArrays<IX>& a, int nblocks, int first, int lane) {
    int carry = a.bpre[first & ~31];
    for (int b0 = first & ~31; b0 < nblocks; b0 += 32) {
        int v = b0 + lane < nblocks ? a.bmin[b0 + lane] : INT_MAX;
        for (int d = 1; d < 32; d <<= 1) { const int y = __shfl_up_sync(KV_FULL, v, d); if (lane >= d) v = min(v, y); }
        v = min(v, carry);
        if (b0 + lane < nblocks) a.bpre[b0 + lane + 1] = v;
        carry = __shfl_sync(KV_FULL, v, 31);
    }
}

// One batch of Algorithm 3 out of the list at positions 0 .. m-1 (no K2L_IN set).  Called by all
// THREADS threads of a CTA.  Sets K2L_IN on the members, leaves their positions in walking order in
// xpos[0 .. k0) and returns k0 (the same value in every thread).
template <int THREADS, typename IX>
__device__ int k2l_batch(const K2lArrays<IX>& a, int m, i64 M, int* status, K2lShared<THREADS>& sh) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int W = THREADS / 32;
    // first fit = longest prefix with sum(s+o) <= M
    int k0 = 0;
    i64 run = 0;
    for (int base = 0; base < m; base += THREADS) {
        const int p = base + tid;
        i64 incl = p < m ? (i64)a.T[p] : 0;
        for (int d = 1; d < 32; d <<= 1) { const i64 y = __shfl_up_sync(KV_FULL, incl, d); if (lane >= d) incl += y; }
        if (W > 1) {
            if (lane == 31) sh.sum64[w] = incl;
            __syncthreads();
            i64 total = 0;
            for (int k = 0; k < W; ++k) { if (k == w) incl += total; total += sh.sum64[k]; }
            incl += run;
            run += total;
        } else {
            incl += run;
            run = __shfl_sync(KV_FULL, incl, 31);
        }
        const bool ok = p < m && incl <= M;
        const int cnt = W > 1 ? __syncthreads_count(ok) : __popc(__ballot_sync(KV_FULL, ok));
        if (ok) {
            a.id[p] |= K2L_IN; a.xpos[p] = (IX)p; a.ub[p] = (IX)p;
            if (p + 1 == m || p + 1 == base + cnt) sh.mem = (int)incl;     // the last one taken so far
        }
        k0 += cnt;
        if (cnt < min(THREADS, m - base)) break;
    }
    if (tid == 0) { sh.pick[0] = INT_MAX; sh.pick[1] = INT_MAX; a.bpre[0] = INT_MAX; }
    k2l_sync<THREADS>();
    const int nblocks = (m + 31) >> 5;
    for (int b = w; b < nblocks; b += W) k2l_scan_block(a, m, b, lane);
    k2l_sync<THREADS>();
    if (w == 0) k2l_scan_totals(a, nblocks, 0, lane);
    // improving swaps; every swap lowers the weights' sum over X by at least 1
    const i64 step_cap = kv_loop_cap(((i64)k0 << 30) + 16);
    for (i64 step = 0;; ++step) {
        k2l_sync<THREADS>();
        const int slack = (int)M - sh.mem, par = (int)(step & 1);
        int hit = INT_MAX;
        for (int k = tid; k < k0; k += THREADS) {
            const int pos = a.xpos[k], cap = slack + a.T[pos];
            int u = a.ub[k];                                  // first position with T > cap: from where it was
            if (u < m && a.T[u] <= cap) {
                int hop = 1;
                while (u + hop < m && a.T[u + hop] <= cap) { u += hop; hop <<= 1; }
                for (; hop; hop >>= 1) if (u + hop < m && a.T[u + hop] <= cap) u += hop;
                ++u;
            } else if (u > 0 && a.T[u - 1] > cap) {
                int hop = 1;
                --u;                                          // T[u] > cap
                while (u - hop >= 0 && a.T[u - hop] > cap) { u -= hop; hop <<= 1; }
                for (; hop; hop >>= 1) if (u - hop >= 0 && a.T[u - hop] > cap) u -= hop;
            }
            a.ub[k] = (IX)u;
            if (u > 0 && min(a.bpre[(u - 1) >> 5], a.pin[u - 1]) < a.O[pos]) { hit = k; break; }
        }
        hit = kv_warp_min(hit);
        if (lane == 0 && hit != INT_MAX) atomicMin(&sh.pick[par], hit);
        k2l_sync<THREADS>();
        const int kstar = sh.pick[par];
        if (kstar == INT_MAX) break;
        if (step > step_cap) { if (tid == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }
        if (w == 0) {
            // the first outside position with a smaller weight: its block, then its place in the block
            const int pos = a.xpos[kstar], thr = a.O[pos];
            int b = 0;
            for (int b0 = 0; b0 < nblocks; b0 += 32) {
                const unsigned v = __ballot_sync(KV_FULL, b0 + lane < nblocks && a.bpre[b0 + lane + 1] < thr);
                if (v) { b = b0 + __ffs(v) - 1; break; }
            }
            const int p = 32 * b + lane;
            const unsigned v = __ballot_sync(KV_FULL, p < m && a.pin[p] < thr);
            const int j = (int)KV_IDX(32 * b + __ffs(v) - 1, m, 811);
            if (lane == 0) {
                a.id[pos] &= ~K2L_IN; a.id[j] |= K2L_IN;
                a.xpos[kstar] = (IX)j;
                sh.mem += a.T[j] - a.T[pos];
                sh.pick[par ^ 1] = INT_MAX;
            }
            __syncwarp();
            k2l_scan_block(a, m, pos >> 5, lane);
            if ((j >> 5) != (pos >> 5)) k2l_scan_block(a, m, j >> 5, lane);
            __syncwarp();
            k2l_scan_totals(a, nblocks, min(pos, j) >> 5, lane);
        }
    }
    return k0;
}

// Takes the members of the batch just built out of the list (the order of the others is kept);
// returns the new length.
template <int THREADS, typename IX>
__device__ int k2l_compact(const K2lArrays<IX>& a, int m, K2lShared<THREADS>& sh) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int W = THREADS / 32;
    int left = 0;
    for (int base = 0; base < m; base += THREADS) {
        const int p = base + tid;
        const int id = p < m ? a.id[p] : K2L_IN, T = p < m ? a.T[p] : 0, O = p < m ? a.O[p] : 0;
        const bool keep = !(id & K2L_IN);
        const unsigned v = __ballot_sync(KV_FULL, keep);
        int before = __popc(v & ((1u << lane) - 1u)), total = __popc(v);
        if (W > 1) {
            if (lane == 0) sh.cnt[w] = total;
            __syncthreads();                                  // also: everyone has read its position
            total = 0;
            for (int k = 0; k < W; ++k) { if (k == w) before += total; total += sh.cnt[k]; }
        }
        if (keep) { a.id[left + before] = id; a.T[left + before] = T; a.O[left + before] = O; }
        left += total;
        k2l_sync<THREADS>();
    }
    return left;
}

// sorted_ids: request ids by ascending (s+o, index).  `scratch`: k2l_bytes(n) bytes of global memory,
// or nullptr when the arrays are in dynamic shared memory.  order_out receives every batch in X's
// walking order (the caller sorts each batch by (o, index)).
template <typename IX>
__global__ void __launch_bounds__(K2L_THREADS)
k2_local_swap(const int* __restrict__ s, const int* __restrict__ o, const int* __restrict__ sorted_ids,
              int n, i64 M, int a_num, int a_den, int* scratch,
              int* __restrict__ order_out, int* __restrict__ batch_off, int* __restrict__ num_batches,
              int* status) {
    extern __shared__ __align__(16) int k2l_smem[];
    __shared__ K2lShared<K2L_THREADS> sh;
    const int tid = threadIdx.x;
    const K2lArrays<IX> a = k2l_arrays<IX>(scratch ? (void*)scratch : (void*)k2l_smem, n);
    for (int p = tid; p < n; p += K2L_THREADS) {
        const int id = sorted_ids[p];
        a.id[p] = id; a.T[p] = s[id] + o[id]; a.O[p] = a_num * s[id] + a_den * o[id];      // weight: o when alpha = 0
    }
    if (tid == 0) batch_off[0] = 0;
    __syncthreads();
    int done = 0, nb = 0, m = n;
    while (m > 0) {
        const int k0 = k2l_batch<K2L_THREADS, IX>(a, m, M, status, sh);
        if (k0 < 1) { if (tid == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }          // every batch places a request
        for (int k = tid; k < k0; k += K2L_THREADS) order_out[KV_IDX(done + k, n, 812)] = a.id[a.xpos[k]] & ~K2L_IN;
        done += k0;
        ++nb;
        if (tid == 0) batch_off[KV_IDX(nb, n + 1, 813)] = done;
        __syncthreads();
        m = k2l_compact<K2L_THREADS, IX>(a, m, sh);
    }
    if (tid == 0) *num_batches = nb;
}
