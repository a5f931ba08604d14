// K2d -- Algorithm 4 (Quantile Greedy Selection, Section 5.3) as the Phase-1 solver, all batches in one
// launch of one CTA (every batch is built from what the previous ones left).
//
// Per batch, over the nr remaining requests, which the algorithm lists in ascending (o, index):
//   sample    the m = max(1, floor(nr/2)) requests with the smallest keys
//             mix(seed ^ mix(batch * 2^32 + id)); Q_p and Q_o are the sample's (s+o) and o at position
//             floor(3 (m-1) / 10) of their ascending orders;
//   pass 1    first fit down the list over the requests with s+o <= Q_p and o <= Q_o;
//   pass 2    first fit over the others in ascending o/(s+o), equal ratios in list order;
//   batch     the requests taken, in list order.
//
// Nothing is sorted per batch.  The three orders (list, size, ratio) do not change, so they are sorted
// once and what has been taken is skipped (and dropped from the lists when it makes up half of them).
// The m-th smallest key is found with one histogram of the keys' leading 12 bits and a ranking of the
// few keys of the bin it falls in (further bits where a bin holds more than K2Q_CAND); the elements at
// a position of the sample's orders by counting sample members along the lists.
//
// The ratio key floor(o * 2^F / (s+o)) orders the requests exactly as the rationals do when
// 2^F exceeds the product of any two denominators: two different ratios differ by at least
// 1 / ((s_a+o_a)(s_b+o_b)) > 2^-F, so their keys differ; equal ratios give equal keys.
//
// First fit is sequential by definition (whether a request is admitted depends on the memory the
// earlier ones took).  Here a CTA takes 1,024 list positions at a time: requests that cannot fit
// even alone in what is left are dropped (the free memory only shrinks, so they would be refused
// at their turn anyway), an inclusive scan over the sizes of the others finds the first one that
// no longer fits after its predecessors; everything before it is admitted, it is refused, and the
// walk goes on right after it.  Every turn either finishes a tile or admits at least one request; the
// walk ends when not even the smallest request would fit.
//
// What bounds it: 23,000 cycles per batch of the 10,000-request backlog (100 batches, 13 turns of first fit each): a quarter the
// histogram's shared-memory atomics, a third the turns of first fit (two barriers where somebody is refused, one
// otherwise), the rest passes over the lists in shared memory.  The keys do not depend on what has been taken, so the whole
// chip makes their leading halves beforehand; entries are counted by votes of 32 consecutive ones (a thread for ten
// consecutive ones met five others on its bank); sums of a tile are 32-bit reductions where they fit.  sorted_f_quantile of
// 10,000 / 4,000 requests 2.59 / 1.45 -> 2.51 / 1.37 with the keys, 2.26 / 1.17 ms with all of it; 1,500 / 500 requests
// 0.85 / 0.28 -> 0.71 / 0.24.  The arrays are in shared memory (19 bytes per request, 10,000 requests) where they fit.
#pragma once

#include "common.cuh"

#define K2Q_THREADS 1024
#define K2Q_BINS 4096
#define K2Q_CAND 512
enum { K2Q_SAMPLE = 1, K2Q_NEW = 2, K2Q_GONE = 4 };

// Entry i of the list in ascending (o, index): its size, or its ratio key; the value is the place i.
struct K2qSlotKey {
    const int *s, *o, *list;
    int F;                       // 0: size
    __device__ __forceinline__ u64 key(int, int i, int n, int& val) const {
        val = i;
        const int id = (int)KV_IDX(list[i], n, 821);
        const u64 T = (u64)(s[id] + o[id]);
        return F ? ((u64)o[id] << F) / T : T;
    }
};

// The sample's key of request `id` in batch b.
__device__ __forceinline__ u64 k2q_key(u64 seed, int b, int id) { return kv_mix64(seed ^ kv_mix64(((u64)(unsigned)b << 32) + (u64)id)); }

// Leading halves of the keys of the first `batches` batches: out[b * n + place in the list].  A key does not depend on
// what has been taken, so the chip makes them before the one CTA that needs them begins.
__global__ void __launch_bounds__(256) k2q_leading(const int* __restrict__ list, int n, int batches, u64 seed, unsigned* __restrict__ out) {
    const i64 total = (i64)batches * n;
    for (i64 k = (i64)blockIdx.x * 256 + threadIdx.x; k < total; k += (i64)gridDim.x * 256) {
        const int b = (int)(k / n);
        out[k] = (unsigned)(k2q_key(seed, b, list[k - (i64)b * n]) >> 32);
    }
}

template <typename IX>
struct K2qArrays {               // by place in the list of all requests
    int *T, *O, *id;
    IX *L, *TL, *RL;             // places in list / size / ratio order
    unsigned char* flag;
};
template <typename IX>
__host__ __device__ inline size_t k2q_bytes(int n) { return (size_t)n * (3 * sizeof(int) + 3 * sizeof(IX) + 1) + 16; }

struct K2qShared {
    int hist[K2Q_BINS];
    u64 cand_key[K2Q_CAND];
    int cand[K2Q_CAND];
    u64 tot[2][32];
    int pick[2];
    u64 taken[2];
    int cnt[2][32];
    int bin, bin_count, bin_before, ncand, Qp, Qo, min_T;
};

// exclusive scan of one value per thread over the CTA; `total` in every thread.  Ends with a barrier
// between its reads of sh.tot and the caller.
__device__ __forceinline__ u64 k2q_scan(u64 v, u64& total, K2qShared& sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    u64 incl = v;
    for (int d = 1; d < 32; d <<= 1) { const u64 y = __shfl_up_sync(KV_FULL, incl, d); if (lane >= d) incl += y; }
    if (lane == 31) sh.tot[0][w] = incl;
    __syncthreads();
    u64 t = sh.tot[0][lane];
    for (int d = 1; d < 32; d <<= 1) { const u64 y = __shfl_up_sync(KV_FULL, t, d); if (lane >= d) t += y; }
    total = __shfl_sync(KV_FULL, t, 31);
    const u64 before = __shfl_sync(KV_FULL, t, w > 0 ? w - 1 : 0);
    __syncthreads();
    return incl - v + (w > 0 ? before : 0);
}

// Sums of a tile's sizes: in 32 bits where 1,024 of them cannot pass 2^31 (their reductions are one instruction).
__device__ __forceinline__ unsigned k2q_sum(unsigned v) { return __reduce_add_sync(KV_FULL, v); }
__device__ __forceinline__ u64 k2q_sum(u64 v) { for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(KV_FULL, v, d); return v; }

// First fit over list[0 .. len); kRatio: everything not taken yet, otherwise sizes up to Qp and decodes
// up to Qo of a list in ascending o.  Flags what it takes; returns the memory in use afterwards.
template <bool kRatio, typename SUM, typename IX>
__device__ i64 k2q_first_fit(const K2qArrays<IX>& a, const IX* list, int len, i64 M, i64 mem, K2qShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int Qp = sh.Qp, Qo = sh.Qo, min_T = sh.min_T;
    int pos = 0, par = 0;
    while (pos < len) {                                   // pos grows by at least one per turn
        const i64 slack = M - mem;
        if (slack < min_T) break;
        if (!kRatio && a.O[list[pos]] > Qo) break;
        const int idx = pos + tid;
        int slot = 0;
        SUM T = 0;
        if (idx < len) {
            slot = list[idx];
            const int t = a.T[slot];
            if (!(a.flag[slot] & (K2Q_NEW | K2Q_GONE)) && t <= slack && (kRatio || (t <= Qp && a.O[slot] <= Qo))) T = (SUM)t;
        }
        SUM incl = T;
        for (int d = 1; d < 32; d <<= 1) { const SUM y = __shfl_up_sync(KV_FULL, incl, d); if (lane >= d) incl += y; }
        SUM* const tot = reinterpret_cast<SUM*>(sh.tot[par]);
        if (lane == 31) tot[w] = incl;
        __syncthreads();
        const SUM t = tot[lane], total = k2q_sum(t), before = k2q_sum(lane < w ? t : (SUM)0);
        const bool cut = total > (SUM)slack;              // somebody is refused
        int first = K2Q_THREADS;
        if (cut) {
            // in the one warp in which the sum passes the slack
            if (before <= (SUM)slack) {
                const unsigned v = __ballot_sync(KV_FULL, T > 0 && before + incl > (SUM)slack);
                if (v && lane == __ffs(v) - 1) { sh.pick[par] = tid; sh.taken[par] = (u64)(before + incl - T); }
            }
            __syncthreads();
            first = sh.pick[par];
        }
        if (T > 0 && tid < first) a.flag[slot] |= K2Q_NEW;
        mem += (i64)(cut ? sh.taken[par] : (u64)total);
        pos += cut ? first + 1 : K2Q_THREADS;
        par ^= 1;                                         // what is written now was last read one turn, and a barrier, ago
    }
    __syncthreads();
    return mem;
}

// list[0 .. len) without what is gone, in the same order; returns the new length
template <typename IX>
__device__ int k2q_compact(const K2qArrays<IX>& a, IX* list, int len, K2qShared& sh) {
    int left = 0;
    for (int base = 0; base < len; base += K2Q_THREADS) {
        const int idx = base + threadIdx.x;
        const IX slot = idx < len ? list[idx] : (IX)0;
        const bool keep = idx < len && !(a.flag[slot] & K2Q_GONE);
        u64 total;
        const int rank = (int)k2q_scan(keep ? 1 : 0, total, sh);
        if (keep) list[left + rank] = slot;
        left += (int)total;
    }
    __syncthreads();
    return left;
}

// list: request ids by ascending (o, index); by_size, by_ratio: places in it.  scratch: k2q_bytes<int>(n)
// bytes of global memory, or nullptr: the arrays are in dynamic shared memory.  Leaves the batches one
// behind the other in order_out, their members in list order, and the boundaries in batch_off.
template <typename IX>
__global__ void __launch_bounds__(K2Q_THREADS)
k2_quantile(const int* __restrict__ s, const int* __restrict__ o, const int* __restrict__ list,
            const int* __restrict__ by_size, const int* __restrict__ by_ratio, int n, i64 M, u64 seed, void* scratch,
            const unsigned* __restrict__ leading, int leading_batches,
            int* __restrict__ order_out, int* __restrict__ batch_off, int* __restrict__ num_batches, int* status) {
    extern __shared__ __align__(16) unsigned char k2q_smem[];
    __shared__ K2qShared sh;
    const int tid = threadIdx.x, lane = tid & 31;
    K2qArrays<IX> a;
    {
        int* p = scratch ? (int*)scratch : (int*)k2q_smem;
        a.T = p; a.O = p + n; a.id = p + 2 * (size_t)n;
        a.L = (IX*)(p + 3 * (size_t)n); a.TL = a.L + n; a.RL = a.TL + n;
        a.flag = (unsigned char*)(a.RL + n);
    }
    for (int p = tid; p < n; p += K2Q_THREADS) {
        const int id = list[p];
        a.T[p] = s[id] + o[id]; a.O[p] = o[id]; a.id[p] = id;
        a.L[p] = (IX)p; a.TL[p] = (IX)by_size[p]; a.RL[p] = (IX)by_ratio[p];
        a.flag[p] = 0;
    }
    if (tid == 0) batch_off[0] = 0;
    __syncthreads();
    int len = n, nr = n, done = 0, nb = 0;
    while (nr > 0) {
        const int m = nr / 2 > 1 ? nr / 2 : 1;
        auto key_of = [&](int slot) { return k2q_key(seed, nb, a.id[slot]); };
        const unsigned* const lead_of = nb < leading_batches ? leading + (size_t)nb * n : nullptr;
        // the key's first 12 bits
        auto first_bits = [&](int slot) { return (lead_of ? lead_of[slot] : (unsigned)(key_of(slot) >> 32)) >> (32 - 12); };
        // ---- the sample: keys whose leading bits are below `top`, and the first of those that have them equal
        int shift = 64 - 12, before = 0;
        u64 top = 0;
        for (;;) {
            for (int k = tid; k < K2Q_BINS; k += K2Q_THREADS) sh.hist[k] = 0;
            if (tid == 0) { sh.ncand = 0; sh.min_T = INT_MAX; }
            __syncthreads();
            for (int i = tid; i < len; i += K2Q_THREADS) {
                const int slot = a.L[i];
                if (a.flag[slot] & K2Q_GONE) continue;
                if (shift == 64 - 12) { atomicAdd(&sh.hist[first_bits(slot)], 1); continue; }
                const u64 h = key_of(slot);
                if ((h >> (shift + 12)) == top) atomicAdd(&sh.hist[(int)(h >> shift) & (K2Q_BINS - 1)], 1);
            }
            __syncthreads();
            int c[K2Q_BINS / K2Q_THREADS], sum = 0;
            u64 total;
#pragma unroll
            for (int k = 0; k < K2Q_BINS / K2Q_THREADS; ++k) { c[k] = sh.hist[tid * (K2Q_BINS / K2Q_THREADS) + k]; sum += c[k]; }
            int ex = (int)k2q_scan((u64)sum, total, sh);
            const int want = m - before;
            if (ex < want && want <= ex + sum) {
#pragma unroll
                for (int k = 0; k < K2Q_BINS / K2Q_THREADS; ++k) {
                    if (ex < want && want <= ex + c[k]) { sh.bin = tid * (K2Q_BINS / K2Q_THREADS) + k; sh.bin_count = c[k]; sh.bin_before = ex; }
                    ex += c[k];
                }
            }
            __syncthreads();
            top = (top << 12) | (u64)sh.bin;
            before += sh.bin_before;
            if (sh.bin_count <= K2Q_CAND || shift < 12) break;             // 4 bits: at most 16 distinct keys
            shift -= 12;
            __syncthreads();
        }
        for (int i = tid; i < len; i += K2Q_THREADS) {
            const int slot = a.L[i];
            if (a.flag[slot] & K2Q_GONE) continue;
            const u64 lead = shift == 64 - 12 ? (u64)first_bits(slot) : key_of(slot) >> shift;
            a.flag[slot] = lead < top ? K2Q_SAMPLE : 0;
            if (lead == top) {
                const u64 h = key_of(slot);
                const int k = (int)KV_IDX(atomicAdd(&sh.ncand, 1), K2Q_CAND, 822);
                sh.cand_key[k] = h; sh.cand[k] = slot;
            }
        }
        __syncthreads();
        if (tid < sh.ncand) {
            const u64 h = sh.cand_key[tid];
            int rank = 0;
            for (int k = 0; k < sh.ncand; ++k) rank += sh.cand_key[k] < h ? 1 : 0;
            if (rank < m - before) a.flag[sh.cand[tid]] = K2Q_SAMPLE;
        }
        __syncthreads();
        // ---- quantiles: the q-th sample member along the list (o) and along the sizes (s+o).  A warp takes 32
        // consecutive entries at a time, `rows` of them: the count of a row is a vote, and its loads are one line each
        const int rows = (len + K2Q_THREADS - 1) / K2Q_THREADS, i0 = (tid >> 5) * rows * 32 + lane;
        auto in_sample = [&](int slot) { return (a.flag[slot] & (K2Q_SAMPLE | K2Q_GONE)) == K2Q_SAMPLE; };
        {
            const int q = (int)((3ll * (m - 1)) / 10);
            int cl = 0, ct = 0, least = INT_MAX;
            for (int r = 0; r < rows; ++r) {
                const int i = i0 + 32 * r, sl = i < len ? a.L[i] : 0, st = i < len ? a.TL[i] : 0, ft = a.flag[st];
                cl += __popc(__ballot_sync(KV_FULL, i < len && in_sample(sl)));
                ct += __popc(__ballot_sync(KV_FULL, i < len && (ft & (K2Q_SAMPLE | K2Q_GONE)) == K2Q_SAMPLE));
                if (i < len && !(ft & K2Q_GONE) && least == INT_MAX) least = a.T[st];
            }
            least = kv_warp_min(least);
            if (lane == 0) {
                sh.cnt[0][tid >> 5] = cl; sh.cnt[1][tid >> 5] = ct;
                if (least != INT_MAX) atomicMin(&sh.min_T, least);
            }
            __syncthreads();
            int el = __reduce_add_sync(KV_FULL, lane < (tid >> 5) ? sh.cnt[0][lane] : 0);
            int et = __reduce_add_sync(KV_FULL, lane < (tid >> 5) ? sh.cnt[1][lane] : 0);
            if (el <= q && q < el + cl) {
                for (int r = 0; r < rows; ++r) {
                    const int i = i0 + 32 * r, slot = i < len ? a.L[i] : 0;
                    const unsigned v = __ballot_sync(KV_FULL, i < len && in_sample(slot));
                    if (((v >> lane) & 1u) && el + __popc(v & ((1u << lane) - 1u)) == q) sh.Qo = a.O[slot];
                    el += __popc(v);
                }
            }
            if (et <= q && q < et + ct) {
                for (int r = 0; r < rows; ++r) {
                    const int i = i0 + 32 * r, slot = i < len ? a.TL[i] : 0;
                    const unsigned v = __ballot_sync(KV_FULL, i < len && in_sample(slot));
                    if (((v >> lane) & 1u) && et + __popc(v & ((1u << lane) - 1u)) == q) sh.Qp = a.T[slot];
                    et += __popc(v);
                }
            }
            __syncthreads();
        }
        // ---- the two passes
        i64 mem;
        if (M < (1ll << 21)) {
            mem = k2q_first_fit<false, unsigned>(a, a.L, len, M, 0, sh);
            mem = k2q_first_fit<true, unsigned>(a, a.RL, len, M, mem, sh);
        } else {
            mem = k2q_first_fit<false, u64>(a, a.L, len, M, 0, sh);
            mem = k2q_first_fit<true, u64>(a, a.RL, len, M, mem, sh);
        }
        // ---- hand the batch out
        int mine = 0;
        for (int r = 0; r < rows; ++r) {
            const int i = i0 + 32 * r;
            mine += __popc(__ballot_sync(KV_FULL, i < len && (a.flag[a.L[i]] & K2Q_NEW)));
        }
        if (lane == 0) sh.cnt[0][tid >> 5] = mine;
        __syncthreads();
        const int taken = __reduce_add_sync(KV_FULL, sh.cnt[0][lane]);
        int at = done + __reduce_add_sync(KV_FULL, lane < (tid >> 5) ? sh.cnt[0][lane] : 0);
        for (int r = 0; r < rows && mine > 0; ++r) {
            const int i = i0 + 32 * r, slot = i < len ? a.L[i] : 0;
            const bool is_new = i < len && (a.flag[slot] & K2Q_NEW);
            const unsigned v = __ballot_sync(KV_FULL, is_new);
            if (is_new) { order_out[KV_IDX(at + __popc(v & ((1u << lane) - 1u)), n, 823)] = a.id[slot]; a.flag[slot] = K2Q_GONE; }
            at += __popc(v);
        }
        if (taken < 1) { if (tid == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }      // every batch places a request
        done += taken; nr -= taken; ++nb;
        if (tid == 0) batch_off[KV_IDX(nb, n + 1, 824)] = done;
        __syncthreads();
        if (2 * nr <= len && len > K2Q_THREADS / 4) {
            const int kept = k2q_compact(a, a.L, len, sh);
            k2q_compact(a, a.TL, len, sh);
            k2q_compact(a, a.RL, len, sh);
            len = kept;
        }
    }
    if (tid == 0) *num_batches = nb;
}
