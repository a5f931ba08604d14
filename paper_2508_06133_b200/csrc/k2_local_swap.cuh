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
// of which needs the one before it, so the latency of one swap; a dependent shared-memory load takes 39
// cycles here, a step of a shuffle scan 40, a branch on a vote 80.  Sizes and the weights outside X are
// therefore kept as trees of four children per node (largest size; smallest weight), one 16-byte load per
// level: a member goes down once and has its ub and the smallest weight below it, the partner is one
// descent, a swap changes two paths.  Two barriers per swap; every array in shared memory where it fits.
#pragma once

#include "common.cuh"

#define K2L_THREADS 512
#define K2L_IN (1 << 30)                      // in id[]: the position belongs to X
#define K2L_LEVELS 16

// Scratch of one solver: the remaining list by position (ascending (s+o, index)), the trees over it and
// the members.  IX: 16-bit where the positions fit.
template <typename IX>
struct K2lArrays {
    int *O, *id;                              // weight, request id (| K2L_IN) by position
    int *T, *U;                               // trees: size; weight outside X (INT_MAX: in X or no position).  Level 0 by position
    IX* xpos;                                 // position of every member in walking order
    int n;
};

// entries of level l of a tree over n positions and at least one INT_MAX behind them, a multiple of 4
__host__ __device__ inline size_t k2l_level(int n, int l) {
    const size_t c = ((size_t)n >> (2 * l)) + 1;
    return (c + 3) & ~(size_t)3;
}
__host__ __device__ inline size_t k2l_tree(int n) {
    size_t c = 0;
    for (int l = 0;; ++l) { c += k2l_level(n, l); if ((n >> (2 * l)) < 4) return c; }
}
template <typename IX>
__host__ __device__ inline size_t k2l_bytes(int n) {
    return (2 * k2l_tree(n) + 2 * (size_t)n) * sizeof(int) + (size_t)n * sizeof(IX) + 32;
}
template <typename IX>
__device__ __forceinline__ K2lArrays<IX> k2l_arrays(void* base /* 16-byte aligned */, int n) {
    K2lArrays<IX> a;
    const size_t tree = k2l_tree(n);
    int* p = (int*)base;
    a.T = p; a.U = p + tree; a.O = p + 2 * tree; a.id = a.O + n; a.xpos = (IX*)(a.id + n); a.n = n;
    return a;
}

template <int THREADS>
struct K2lShared {
    static constexpr int W = THREADS / 32;
    i64 sum64[W];
    int cnt[W];
    int off[K2L_LEVELS];                      // where a level begins in its tree
    int pick[2];
    int mem;
};

#define K2L_TOP 6                             // lists of up to 4^7 - 1: their walks through the trees are unrolled

template <int THREADS>
__device__ __forceinline__ void k2l_sync() { if (THREADS == 32) __syncwarp(); else __syncthreads(); }

// The improving swaps of one batch; TOP: the trees' highest level, -1: `top`, whatever it is.
template <int THREADS, typename IX, int TOP>
__device__ void k2l_improve(const K2lArrays<IX>& a, int m, int k0, i64 M, int top, int* status, K2lShared<THREADS>& sh) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int LEVELS = TOP < 0 ? 1 : TOP + 1;
    int off[LEVELS];                                          // where the levels begin
    off[0] = 0;
#pragma unroll
    for (int l = 1; l < LEVELS; ++l) off[l] = off[l - 1] + (int)k2l_level(a.n, l - 1);
    // every swap lowers the weights' sum over X by at least 1
    const i64 step_cap = kv_loop_cap(((i64)k0 << 30) + 16);
    for (i64 step = 0;; ++step) {
        const int slack = (int)M - sh.mem, par = (int)(step & 1);
        int hit = INT_MAX;
        for (int k = tid; k < k0; k += THREADS) {
            const int pos = a.xpos[k], cap = slack + a.T[pos], mine = a.O[pos];
            int idx = 0, least = INT_MAX;                     // down to the first position with T > cap
            auto down = [&](int from) {
                // sizes ascend and an INT_MAX follows the last, so at most three of the four are passed
                const int4 t = *reinterpret_cast<const int4*>(a.T + from + 4 * idx), u = *reinterpret_cast<const int4*>(a.U + from + 4 * idx);
                const bool p0 = t.x <= cap, p1 = t.y <= cap, p2 = t.z <= cap;
                least = min(least, min(p0 ? u.x : INT_MAX, min(p1 ? u.y : INT_MAX, p2 ? u.z : INT_MAX)));
                idx = 4 * idx + (p0 ? 1 : 0) + (p1 ? 1 : 0) + (p2 ? 1 : 0);
            };
            if constexpr (TOP >= 0) {
#pragma unroll
                for (int l = TOP; l >= 0; --l) down(off[l]);
            } else {
                for (int l = top; l >= 0; --l) down(sh.off[l]);
            }
            if (least < mine) { hit = k; break; }
        }
        hit = kv_warp_min(hit);
        if (lane == 0 && hit != INT_MAX) atomicMin(&sh.pick[par], hit);
        k2l_sync<THREADS>();
        const int kstar = sh.pick[par];
        if (kstar == INT_MAX) break;
        if (step > step_cap) { if (tid == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }
        if (w == 0) {
            // the first outside position with a smaller weight
            const int pos = a.xpos[kstar], thr = a.O[pos];
            int j = 0;
            auto down = [&](int from) {
                const int4 u = *reinterpret_cast<const int4*>(a.U + from + 4 * j);
                j = 4 * j + (u.x < thr ? 0 : u.y < thr ? 1 : u.z < thr ? 2 : 3);
            };
            if constexpr (TOP >= 0) {
#pragma unroll
                for (int l = TOP; l >= 0; --l) down(off[l]);
            } else {
                for (int l = top; l >= 0; --l) down(sh.off[l]);
            }
            j = (int)KV_IDX(j, m, 811);
            // lane 0 goes up from the one that leaves X, the others all from the one that enters it
            int node = lane == 0 ? pos : j;
            a.U[node] = lane == 0 ? thr : INT_MAX;
            auto up = [&](int from, int to) {
                __syncwarp();
                node >>= 2;
                const int4 u = *reinterpret_cast<const int4*>(a.U + from + 4 * node);
                a.U[to + node] = min(min(u.x, u.y), min(u.z, u.w));
            };
            if constexpr (TOP >= 0) {
#pragma unroll
                for (int l = 1; l <= TOP; ++l) up(off[l - 1], off[l]);
            } else {
                for (int l = 1; l <= top; ++l) up(sh.off[l - 1], sh.off[l]);
            }
            if (lane == 0) {
                a.id[pos] &= ~K2L_IN; a.id[j] |= K2L_IN;
                a.xpos[kstar] = (IX)j;
                sh.mem += a.T[j] - a.T[pos];
                sh.pick[par ^ 1] = INT_MAX;
            }
        }
        k2l_sync<THREADS>();
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
            a.id[p] |= K2L_IN; a.xpos[p] = (IX)p;
            if (p + 1 == m || p + 1 == base + cnt) sh.mem = (int)incl;     // the last one taken so far
        }
        k0 += cnt;
        if (cnt < min(THREADS, m - base)) break;
    }
    // the trees over m positions
    int top = 0;                                              // the level of at most 4 entries
    while ((m >> (2 * top)) >= 4) ++top;
    if (tid == 0) {
        sh.pick[0] = INT_MAX; sh.pick[1] = INT_MAX;
        int off = 0;
        for (int l = 0; l <= top; ++l) { sh.off[l] = off; off += (int)k2l_level(a.n, l); }
    }
    k2l_sync<THREADS>();
    for (int p = tid; p < (int)k2l_level(m, 0); p += THREADS) {
        if (p >= m) a.T[p] = INT_MAX;
        a.U[p] = p >= k0 && p < m ? a.O[p] : INT_MAX;
    }
    k2l_sync<THREADS>();
    for (int l = 1; l <= top; ++l) {
        const int below = sh.off[l - 1], at = sh.off[l], nodes = (int)k2l_level(m, l), children = (int)k2l_level(m, l - 1) >> 2;
        for (int i = tid; i < nodes; i += THREADS) {
            int tv = INT_MAX, uv = INT_MAX;
            if (i < children) {
                const int4 u = *reinterpret_cast<const int4*>(a.U + below + 4 * i);
                tv = a.T[below + 4 * i + 3];
                uv = min(min(u.x, u.y), min(u.z, u.w));
            }
            a.T[at + i] = tv; a.U[at + i] = uv;
        }
        k2l_sync<THREADS>();
    }
    switch (top) {
        case 0: k2l_improve<THREADS, IX, 0>(a, m, k0, M, top, status, sh); break;
        case 1: k2l_improve<THREADS, IX, 1>(a, m, k0, M, top, status, sh); break;
        case 2: k2l_improve<THREADS, IX, 2>(a, m, k0, M, top, status, sh); break;
        case 3: k2l_improve<THREADS, IX, 3>(a, m, k0, M, top, status, sh); break;
        case 4: k2l_improve<THREADS, IX, 4>(a, m, k0, M, top, status, sh); break;
        case 5: k2l_improve<THREADS, IX, 5>(a, m, k0, M, top, status, sh); break;
        case K2L_TOP: k2l_improve<THREADS, IX, K2L_TOP>(a, m, k0, M, top, status, sh); break;
        default: k2l_improve<THREADS, IX, -1>(a, m, k0, M, top, status, sh); break;
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
template <typename IX, bool kShared>
__global__ void __launch_bounds__(K2L_THREADS)
k2_local_swap(const int* __restrict__ s, const int* __restrict__ o, const int* __restrict__ sorted_ids,
              int n, i64 M, int a_num, int a_den, int* scratch,
              int* __restrict__ order_out, int* __restrict__ batch_off, int* __restrict__ num_batches,
              int* status) {
    extern __shared__ __align__(16) int k2l_smem[];
    __shared__ K2lShared<K2L_THREADS> sh;
    const int tid = threadIdx.x;
    const K2lArrays<IX> a = k2l_arrays<IX>(kShared ? (void*)k2l_smem : (void*)scratch, n);
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
