// K1 -- sorting of (64-bit key, 32-bit value) pairs in ascending (key, value) order, in independent rows
// of n entries; the keys are made on the fly from what they are a function of.
//
// Used for the request orderings the method needs: ascending (s+o, o, index) over the whole backlog
// (the order Algorithm 3 starts from), ascending (o, index) inside every selected batch (Algorithm 1,
// Phase 1: "sort requests in X* in nondecreasing order of o_i"), and the requests of explicit schedules
// by start time.  Values are distinct within a row (request ids), so the result does not depend on
// anything but the pairs.
//
//   k1_tile_sort    one CTA sorts a tile of up to 1,024 pairs: a bitonic network, exchanges within a
//                   warp by shuffles, the others through shared memory.
//   k1_tile_merge   merges up to K1_MERGE_RUNS sorted runs: the place of a pair in the merged run is its
//                   place in its own plus, for every other one, the pairs there that come before it: a
//                   binary search each, four runs at a time.  Neighbouring lanes hold neighbouring pairs,
//                   so their searches read the same lines.
// One launch up to 1,024 entries, two up to 32,768, three up to 2^20, and 11 to 15 search steps per pair, run
// and merge.  All tiles in one merge took n / 1024 * 11 steps per pair: sorted_f of 1,000,000 requests 71.6 -> 55.8
// ms, of 10,000,000 2,390 -> 679.  The radix sort in front of that, one CTA per row and a chain of 6 to 8 passes
// over it, was bounded by latency.
#pragma once

#include "common.cuh"

#define K1_TILE 1024
#define K1_MERGE_THREADS 256
#define K1_MERGE_RUNS 32

__device__ __forceinline__ bool k1_less(u64 ka, int va, u64 kb, int vb) { return ka < kb || (ka == kb && va < vb); }

// KEY: a struct with  __device__ u64 key(row, i, n, val&)  for entry i of a row.  blockDim.x: the tile,
// a power of two of 32 .. K1_TILE; grid: rows * tiles per row.
template <class KEY>
__global__ void __launch_bounds__(K1_TILE)
k1_tile_sort(const KEY src, int n, int tiles, u64* __restrict__ keys, int* __restrict__ vals) {
    __shared__ u64 sk[K1_TILE];
    __shared__ int sv[K1_TILE];
    const int tid = threadIdx.x, size_max = blockDim.x;
    const int row = blockIdx.x / tiles, i = (blockIdx.x % tiles) * K1_TILE + tid;
    u64 key = ~0ull;                                     // the padding sorts to the end of a row's last tile
    int val = 0x7fffffff;
    if (i < n) key = src.key(row, i, n, val);
    for (int size = 2; size <= size_max; size <<= 1) {
        const bool up = (tid & size) == 0 || size == size_max;
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            u64 ok; int ov;
            if (stride >= 32) {
                __syncthreads();
                sk[tid] = key; sv[tid] = val;
                __syncthreads();
                ok = sk[tid ^ stride]; ov = sv[tid ^ stride];
            } else {
                ok = __shfl_xor_sync(KV_FULL, key, stride); ov = __shfl_xor_sync(KV_FULL, val, stride);
            }
            const bool low = (tid & stride) == 0;
            if (k1_less(ok, ov, key, val) == (low == up)) { key = ok; val = ov; }
        }
    }
    if (i < n) {
        const size_t at = (size_t)row * n + i;
        if (keys) keys[at] = key;
        vals[at] = val;
    }
}

// Merges every `group` runs of `run` sorted pairs.  keys_out: nullptr at the last merge of a row.  grid: total entries / K1_MERGE_THREADS
static __global__ void __launch_bounds__(K1_MERGE_THREADS)
k1_tile_merge(const u64* __restrict__ keys_all, const int* __restrict__ vals_all, int n, i64 total, int run, int group, int steps,
              u64* __restrict__ keys_out, int* __restrict__ vals_out) {
    const i64 at = (i64)blockIdx.x * K1_MERGE_THREADS + threadIdx.x;
    if (at >= total) return;
    const i64 row0 = at / n * n;
    const u64* keys = keys_all + row0;
    const int* vals = vals_all + row0;
    const int i = (int)(at - row0);
    const u64 key = keys[i];
    const int val = vals[i];
    const int mine = i / run, first = mine / group * group;
    const int runs = min(group, (n - first * run + run - 1) / run);           // of this group
    int rank = i - mine * run;
    for (int t0 = 0; t0 < runs; t0 += 4) {
        int lo[4], hi[4], from[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int t = t0 + q;
            const bool other = t < runs && first + t != mine;
            lo[q] = from[q] = other ? (first + t) * run : 0;
            hi[q] = other ? (int)min((i64)n, (i64)from[q] + run) : 0;
        }
        for (int step = 0; step < steps; ++step) {       // `run` entries: run + 1 answers
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (lo[q] < hi[q]) {
                    const int mid = lo[q] + ((hi[q] - lo[q]) >> 1);
                    const u64 k = keys[mid];
                    if (k < key || (k == key && vals[mid] < val)) lo[q] = mid + 1; else hi[q] = mid;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) rank += lo[q] - from[q];
    }
    const i64 to = row0 + KV_IDX(first * run + rank, n, 701);
    if (keys_out) keys_out[to] = key;
    vals_out[to] = val;
}

// Whole-backlog orders: ascending (s+o, o, index) / (s+o, index) / (o, index).
struct K1RequestKey {
    const int *s, *o;
    int policy;
    __device__ __forceinline__ u64 key(int, int i, int, int& val) const {
        val = i;
        const u64 T = (u64)(s[i] + o[i]), O = (u64)o[i];
        return policy == SCHED_POLICY_SOF ? O : policy == SCHED_POLICY_TOTAL_SIZE ? T : (T << 32) | O;
    }
};

// Every batch by ascending (o, index): (batch, o) of the request at list position q.
struct K1BatchKey {
    const int *o, *list, *batch_off, *num_batches;
    __device__ __forceinline__ u64 key(int, int q, int n, int& val) const {
        const int id = (int)KV_IDX(list[q], n, 702);
        val = id;
        int lo = 0, hi = *num_batches - 1;               // the batch with batch_off[b] <= q < batch_off[b+1]
        while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (batch_off[mid] <= q) lo = mid; else hi = mid - 1; }
        return ((u64)(unsigned)lo << 32) | (u64)(unsigned)o[id];
    }
};

// Explicit schedules: (start, id) of request i of schedule `row`.
struct K1StartKey {
    const int* starts;
    __device__ __forceinline__ u64 key(int row, int i, int n, int& val) const {
        val = i;
        return (u64)(unsigned)starts[(size_t)row * n + i];
    }
};
