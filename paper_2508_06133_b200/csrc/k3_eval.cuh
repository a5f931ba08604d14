// K3 (+K4) -- batched schedule evaluation kernels.
//
//   k3_base_run       accepts the best move of a sweep if asked to, gathers (s, o) of the request at every
//                     position of the base order, list-schedules it and stores the simulator state in
//                     front of every `stride`-th position (snapshots) plus the start of every position.
//   k3_eval_moves     one warp per candidate; the candidate is a move applied to the base order
//                     (K4: index -> (type, i, j) -> position map, never materialised; launch order
//                     bucketed by first moved position); simulation resumes from the last snapshot
//                     at or before the first moved position.
//   k3_eval_orders    explicit permutations, simulated from t = 0.
//   (k3_policy.cuh)   k3_eval_policy: one warp per (instance, policy) pair: order construction,
//                     optional prefix-F batching, simulation -- all in shared memory.
//   k3_check_starts   explicit start times: occupancy by the integer program's memory row
//                     (Section 6.1), flag raised where a request takes a round above M.
//
// The request table is read through L1/L2, 32 positions (256 consecutive bytes) at a time: one such
// load per 32 admissions, whereas a copy of it in shared memory takes the room of 20 simulators.
#pragma once

#include "common.cuh"
#include "k2_fmetric.cuh"
#include "k4_moves.cuh"
#include "k5_argmin.cuh"
#include "sim_chunk.cuh"
#include "sim_hyb.cuh"

__device__ __forceinline__ int kv_wrap(int idx, int L) {   // idx < 3L
    if (idx >= L) idx -= L;
    if (idx >= L) idx -= L;
    return (int)KV_IDX(idx, L, 301);
}

#define K3S_WARPS 16                       // warps per CTA of the start-time checker

__global__ void k3_make_table(const int* __restrict__ s, const int* __restrict__ o, int total, int2* __restrict__ tbl) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < total) tbl[i] = make_int2(s[i], o[i]);
}

__global__ void k3_iota(int* a, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = i;
}

// ------------------------------------------------------------------------------------------------
// Base run: positions 0 .. n-1 of the base order; snapshot idx holds the state in front of
// position idx * stride.  One CTA; all of it gathers the table, one warp runs: the run is a chain of n
// admissions, each of which needs the one before it, so what counts is the latency of one admission.
// The next 32 requests are loaded while the 32 in hand are admitted, and their starts are stored
// together.  Dynamic shared memory: the simulator's ring.
//
// With `accept`, the best move of a sweep comes first, so that an iteration of a small local search is
// two launches: the smallest (TEL, index) of tel[0 .. count) (or what `best` already holds, count = 0)
// is applied to the order if it strictly improves the base TEL (Section 5.2's rule); if it does not,
// nothing else happens.
// ------------------------------------------------------------------------------------------------
#define K3B_THREADS 256

struct BaseRunParams {
    const int2* tbl_id;
    int2* tbl_base;
    int* order;
    int n, L, M, stride, snap_count;
    int* snap_ring;
    SnapHeader* snap_hdr;
    int* starts_pos;
    i64* base_tel;
    int* status;
    int accept;
    const i64* tel;
    const int* index_map;
    i64 count;
    i64* best;                         // (TEL, index)
    int* accepted;
    int* scratch;                      // [n]
    int sampled, iteration;
    u64 seed;
};

// Applies the best move to the order if it improves; the same answer in every thread.
__device__ bool k3_accept(const BaseRunParams& p) {
    __shared__ i64 sh_v[K3B_THREADS / 32], sh_i[K3B_THREADS / 32];
    __shared__ Move mv;
    __shared__ int sh_do;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, n = p.n;
    if (p.count > 0) {
        i64 bv = INT64_MAX, bi = INT64_MAX;
        for (i64 k = tid; k < p.count; k += K3B_THREADS) k5_take(bv, bi, p.tel[k], p.index_map ? (i64)p.index_map[k] : k);
        for (int d = 16; d >= 1; d >>= 1) {
            const i64 ov = __shfl_xor_sync(KV_FULL, bv, d), oi = __shfl_xor_sync(KV_FULL, bi, d);
            k5_take(bv, bi, ov, oi);
        }
        if (lane == 0) { sh_v[w] = bv; sh_i[w] = bi; }
        __syncthreads();
        if (tid == 0) {
            for (int k = 1; k < K3B_THREADS / 32; ++k) k5_take(bv, bi, sh_v[k], sh_i[k]);
            p.best[0] = bv; p.best[1] = bi;
        }
    }
    if (tid == 0) {
        const i64 bv = p.best[0], bi = p.best[1];
        bool improve = bi != INT64_MAX && bv < *p.base_tel;
        if (improve) {
            mv = p.sampled ? kv_sample_move(n, p.seed, p.iteration, bi) : kv_decode_move(n, bi);
            if ((unsigned)mv.i >= (unsigned)n || (unsigned)mv.j >= (unsigned)n) improve = false;   // not a move of this list
        }
        sh_do = improve ? 1 : 0;
        *p.accepted = sh_do;
    }
    __syncthreads();
    if (!sh_do) return false;
    const Move m = mv;
    if (m.type == 0) {
        if (tid == 0) { const int x = p.order[m.i]; p.order[m.i] = p.order[m.j]; p.order[m.j] = x; }
    } else {
        // insert: build the moved range in scratch, then copy it back
        const int lo = min(m.i, m.j), hi = max(m.i, m.j);
        for (int q = lo + tid; q <= hi; q += K3B_THREADS) p.scratch[q] = p.order[kv_map_pos(m, q)];
        __syncthreads();
        for (int q = lo + tid; q <= hi; q += K3B_THREADS) p.order[q] = p.scratch[q];
    }
    __syncthreads();
    return true;
}

template <class SIM, int kForm, bool kTogether>
__global__ void __launch_bounds__(K3B_THREADS)
k3_base_run(const BaseRunParams p) {
    if (p.accept && !k3_accept(p)) return;
    for (int q = threadIdx.x; q < p.n; q += K3B_THREADS) p.tbl_base[q] = p.tbl_id[KV_IDX(p.order[q], p.n, 409)];
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int2* tbl_base = p.tbl_base;
    const int n = p.n, L = p.L, M = p.M, stride = p.stride;
    int* const snap_ring = p.snap_ring;
    SnapHeader* const snap_hdr = p.snap_hdr;
    int* const base_starts_pos = p.starts_pos;
    int* const status = p.status;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x;
    SIM sim;
    sim.attach((int*)smem_raw, L);
    sim.reset(M);
    i64 tel = 0;                                         // this lane's share of the completion times so far
    int2 next = lane < n ? tbl_base[lane] : make_int2(1, 1);
    int to_snap = 0, idx = 0;                            // positions until the next snapshot, its number
    bool calm = kTogether;                                    // nothing has waited, or not since the last snapshot
    int t_snap = 0;
    for (int q0 = 0; q0 < n;) {
        const int2 so = next;
        // a block ends where a snapshot is due
        if (to_snap == 0) {
            const int i = (int)KV_IDX(idx, p.snap_count, 401);
            i64 before = tel;
            for (int d = 16; d >= 1; d >>= 1) before += __shfl_xor_sync(KV_FULL, before, d);
            sim.store(snap_ring + (size_t)i * L, snap_hdr + i, before);
            ++idx;
            to_snap = stride;
            calm = kTogether && (calm || (sim.start() == t_snap && (idx & 7) == 0));       // a mistake costs a block of four
            t_snap = sim.start();
        }
        const int cnt = min(min(32, n - q0), to_snap);
        if (q0 + cnt + lane < n) next = tbl_base[q0 + cnt + lane];
        int mine;
        if constexpr (kForm < 0) mine = sim.run(so, cnt, status);
        else if constexpr (!kTogether) mine = sim.template run_alone<kForm>(so, cnt, status);
        else mine = calm ? sim.run_together(so, cnt, calm, status) : sim.template run_alone<kForm>(so, cnt, status);
        if (lane < cnt) base_starts_pos[q0 + lane] = mine;
        if (lane < cnt) tel += (i64)mine + so.y;
        q0 += cnt;
        to_snap -= cnt;
    }
    for (int d = 16; d >= 1; d >>= 1) tel += __shfl_xor_sync(KV_FULL, tel, d);
    if (lane == 0) *p.base_tel = tel;
}

// ------------------------------------------------------------------------------------------------
// Moves.  mode 0: codes[c]; mode 1: code = first + c; mode 2: sampled move m = first + c.
// ------------------------------------------------------------------------------------------------
struct MoveEvalParams {
    int n, L, M, stride, snap_count;
    const int2* tbl_base;
    const int* snap_ring;
    const SnapHeader* snap_hdr;
    MoveSource src;
    i64 count;
    const int* launch_order;           // candidate index of every launch slot (K4), nullptr: the slot itself
    i64* tel_out;
    int tel_by_slot;                   // 1: tel_out is indexed by launch slot (full-sector writes; the arg-min maps
                                       // slots back through launch_order), 0: by candidate index
    int* starts_out;                   // nullable [count][n], by request id
    const int* base_order;
    const int* base_starts_pos;
    i64 first_slot, end_slot;          // launch slots of this launch
    int* rings;                        // simulators with rings in device memory: one per slot of this launch
    int* status;
};

// One warp per candidate, no loop over candidates (a persistent loop around the simulator costs
// ~15 % more instructions per admission with this compiler): warp w of CTA b takes launch slot
// kWarps b + w, whose candidate K4 chose so that the warps of a CTA have nearly equal work.
template <class SIM, bool kStarts>
__global__ void __launch_bounds__(SIM::kWarps * 32, SIM::kMinCtas)
k3_eval_moves(const MoveEvalParams p) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int2* __restrict__ tbl = p.tbl_base;
    const int n = p.n, L = p.L, M = p.M;
    const i64 at = (i64)blockIdx.x * (blockDim.x >> 5) + warp, slot = p.first_slot + at;
    if (slot >= p.end_slot) return;
    const i64 c = p.launch_order ? KV_IDX(p.launch_order[slot], p.count, 402) : slot;
    i64* tel_dst = p.tel_out + (p.tel_by_slot ? slot : c);
    SIM sim;
    sim.attach((SIM::kGlobal ? p.rings + at * SIM::ring_cells(L) : (int*)smem_raw + (size_t)warp * SIM::ring_cells(L)), L);
    const Move mv = k4_move_of(p.src, n, c);
    if ((unsigned)mv.i >= (unsigned)n || (unsigned)mv.j >= (unsigned)n) {      // code outside the neighbourhood
        if (lane == 0) *tel_dst = INT64_MAX;
        return;
    }
    const int first_pos = min(mv.i, mv.j);
    const int idx = (int)KV_IDX(first_pos / p.stride, p.snap_count, 403);
    const int q_start = idx * p.stride;
    // restore the base run's state in front of q_start
    sim.load(p.snap_ring + (size_t)idx * L, p.snap_hdr[idx], M);
    i64 sum_o = 0;
    int* starts = kStarts ? p.starts_out + (size_t)c * n : nullptr;
    if (kStarts)
        for (int q = lane; q < q_start; q += 32) starts[KV_IDX(p.base_order[q], n, 406)] = p.base_starts_pos[q];
    for (int q0 = q_start; q0 < n; q0 += 32) {
        const int qq = q0 + lane;
        int2 so = make_int2(1, 1);
        int id = 0;
        if (qq < n) {
            const int bp = (int)KV_IDX(kv_map_pos(mv, qq), n, 404);
            so = tbl[bp];
            if (kStarts) id = p.base_order[bp];
        }
        const int cnt = min(32, n - q0);
        if (lane < cnt) sum_o += so.y;
        const int mine = sim.run(so, cnt, p.status);
        if (kStarts && lane < cnt) starts[KV_IDX(id, n, 405)] = mine;
    }
    for (int d = 16; d >= 1; d >>= 1) sum_o += __shfl_xor_sync(KV_FULL, sum_o, d);
    if (lane == 0) *tel_dst = sim.total(sum_o);
}

// ------------------------------------------------------------------------------------------------
// Checks of the host entry point's candidates: every order a permutation of 0 .. n-1 (one bit per id in
// dynamic shared memory), every start time in 0 .. 2^30 - 1.
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k3_check_orders(const int* __restrict__ orders, int n, i64 count, int* bad) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned* seen = (unsigned*)smem_raw;
    const int words = (n + 31) >> 5;
    for (i64 c = blockIdx.x; c < count; c += gridDim.x) {
        for (int k = threadIdx.x; k < words; k += 256) seen[k] = 0u;
        __syncthreads();
        bool wrong = false;
        for (int q = threadIdx.x; q < n; q += 256) {
            const int id = orders[(size_t)c * n + q];
            if ((unsigned)id >= (unsigned)n) { wrong = true; continue; }
            const unsigned bit = 1u << (id & 31);
            if (atomicOr(&seen[id >> 5], bit) & bit) wrong = true;
        }
        if (wrong) *bad = 1;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) k3_check_start_range(const int* __restrict__ starts, i64 total, int* bad) {
    bool wrong = false;
    for (i64 k = (i64)blockIdx.x * 256 + threadIdx.x; k < total; k += (i64)gridDim.x * 256) wrong = wrong || (unsigned)starts[k] >= (1u << 30);
    if (wrong) *bad = 1;
}

// ------------------------------------------------------------------------------------------------
// Explicit orders: orders[c][q] = request id at position q.
// ------------------------------------------------------------------------------------------------
struct OrderEvalParams {
    int n, L, M;
    const int2* tbl_id;
    const int* orders;
    i64 count;
    i64* tel_out;
    int* starts_out;
    const int* bad;                    // nullable: not 0, what k3_check_orders has found
    int* status;
};

template <class SIM, bool kStarts>
__global__ void __launch_bounds__(SIM::kWarps * 32, SIM::kMinCtas)
k3_eval_orders(const OrderEvalParams p) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int2* __restrict__ tbl = p.tbl_id;
    const int n = p.n, L = p.L, M = p.M;
    const i64 c = (i64)blockIdx.x * (blockDim.x >> 5) + warp;      // every order has the same length
    if (c >= p.count || (p.bad && *p.bad)) return;
    SIM sim;
    sim.attach((int*)smem_raw + (size_t)warp * SIM::ring_cells(L), L);
    const int* ord = p.orders + (size_t)c * n;
    int* starts = kStarts ? p.starts_out + (size_t)c * n : nullptr;
    sim.reset(M);
    int bad = 0, base = 0;                                // rounds are counted from `base` on (0 in permutations)
    i64 sum_o = 0;
    for (int q0 = 0; q0 < n; q0 += 32) {
        const int qq = q0 + lane;
        int2 so = make_int2(1, 1);
        int id = 0;
        if (qq < n) { id = ord[qq]; if ((unsigned)id >= (unsigned)n) { id = 0; bad = 1; } so = tbl[id]; }
        if (__any_sync(KV_FULL, bad)) {                                       // an id outside 0..n-1
            if (lane == 0) p.tel_out[c] = INT64_MAX;
            return;
        }
        const int cnt = min(32, n - q0);
        base += sim.rebase();
        if (lane < cnt) sum_o += (i64)so.y + (unsigned)base;
        const int mine = sim.run(so, cnt, p.status);
        if (kStarts && lane < cnt) starts[id] = mine + base;
    }
    for (int d = 16; d >= 1; d >>= 1) sum_o += __shfl_xor_sync(KV_FULL, sum_o, d);
    if (lane == 0) p.tel_out[c] = sim.total(sum_o);
}

// ------------------------------------------------------------------------------------------------
// Explicit start times p[c][i].  One warp per candidate.  Requests are visited in ascending start
// order (ids sorted by K1 beforehand: sorted_ids[c][k]), so a window never begins before the ones in
// front of it and the simulator's test answers the question: the schedule stays within M in every
// round  <=>  every request fits at its start beside those with an earlier start (or a lower id).
// feasible[c] = 0 from the first that does not (the remaining requests are still summed into the TEL
// but no longer placed).
// ------------------------------------------------------------------------------------------------
struct StartsEvalParams {
    int n, L, M;
    const int2* tbl_id;
    const int* starts;        // [count][n]
    const int* sorted_ids;    // [count][n] ids by ascending (start, id)
    i64 count;
    i64* tel_out;
    unsigned char* feasible_out;
    const int* bad;           // nullable: not 0, what k3_check_start_range has found
    unsigned int* counter;
};

template <class SIM>
__global__ void __launch_bounds__(SIM::kWarps * 32)
k3_check_starts(const StartsEvalParams p) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const i64 c = (i64)blockIdx.x * SIM::kWarps + warp;
    if (c >= p.count || (p.bad && *p.bad)) return;
    const int n = p.n, M = p.M;
    const int* st_c = p.starts + (size_t)c * n;
    const int* ids = p.sorted_ids + (size_t)c * n;
    SIM sim;
    sim.attach((int*)smem_raw + (size_t)warp * SIM::ring_cells(p.L), p.L);
    sim.reset(M);
    i64 tel = 0;
    bool ok = true;
    int base = 0;                                                              // rounds are counted from here on
    int id_next = lane < n ? ids[lane] : 0;
    for (int q0 = 0; q0 < n; q0 += 32) {
        const int cnt = min(32, n - q0), id = id_next;
        if (q0 + 32 + lane < n) id_next = ids[q0 + 32 + lane];
        int2 so = make_int2(1, 1);
        int pi = 0;
        if (lane < cnt) { so = p.tbl_id[KV_IDX(id, n, 407)]; pi = st_c[id]; tel += (i64)pi + so.y; }
        if (__any_sync(KV_FULL, pi < 0)) ok = false;                           // the simulator cannot go back
        base += sim.rebase();
        for (int k = 0; k < cnt && ok; ++k) {
            const int sp = __shfl_sync(KV_FULL, so.x, k) + 1, om = __shfl_sync(KV_FULL, so.y, k) - 1;
            const int wait = __shfl_sync(KV_FULL, pi, k) - base - sim.start();
            if (wait < 0) { ok = false; break; }
            if (wait > sim.mask + 128) { base += sim.start() + wait; sim.reset(M); }          // nothing is resident any more
            else if (wait > 0) sim.advance(wait);
            ok = sim.put_if_fits(sp, om);
        }
    }
    for (int d = 16; d >= 1; d >>= 1) tel += __shfl_xor_sync(KV_FULL, tel, d);
    if (lane == 0) {
        p.tel_out[c] = tel;
        if (p.feasible_out) p.feasible_out[c] = ok ? 1 : 0;
    }
}

// The same on a ring of single rounds, for decodes beyond what the chunked simulator covers.
__global__ void __launch_bounds__(K3S_WARPS * 32, 1)
k3_check_starts_cells(const StartsEvalParams p) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* ring = (int*)smem_raw + (size_t)warp * p.L;
    const int n = p.n, L = p.L, M = p.M;
    if (p.bad && *p.bad) return;
    for (;;) {
        unsigned c32 = 0;
        if (lane == 0) c32 = atomicAdd(p.counter, 1u);
        const i64 c = (i64)__shfl_sync(KV_FULL, c32, 0);
        if (c >= p.count) break;
        const int* st_c = p.starts + (size_t)c * n;
        const int* ids = p.sorted_ids + (size_t)c * n;
        for (int r = lane; r < L; r += 32) ring[r] = 0;
        __syncwarp();
        int t = 0, tr = 0;
        i64 tel = 0;
        bool ok = true;
        for (int q0 = 0; q0 < n; q0 += 32) {
            const int qq = q0 + lane;
            int2 so = make_int2(1, 1);
            int pi = 0;
            if (qq < n) { const int id = ids[qq]; so = p.tbl_id[id]; pi = st_c[id]; }
            const int cnt = min(32, n - q0);
            for (int k = 0; k < cnt; ++k) {
                const int s = __shfl_sync(KV_FULL, so.x, k), o = __shfl_sync(KV_FULL, so.y, k);
                const int pk = __shfl_sync(KV_FULL, pi, k);
                tel += (i64)pk + o;
                if (!ok) continue;
                // advance the ring to round pk: cells of rounds t .. pk-1 are finished
                const int adv = pk - t;
                if (adv < 0) { ok = false; continue; }                       // starts not ascending: unsorted or negative input
                if (adv >= L) { for (int r = lane; r < L; r += 32) ring[r] = 0; }
                else for (int r = lane; r < adv; r += 32) ring[kv_wrap(tr + r, L)] = 0;
                __syncwarp();
                tr = adv >= L ? 0 : kv_wrap(tr + adv, L);
                t = pk;
                int over = 0;
                for (int r = lane; r < o; r += 32) {
                    const int idx = kv_wrap(tr + r, L);
                    const int v = ring[idx] + s + 1 + r;
                    ring[idx] = v;
                    over |= v > M;
                }
                __syncwarp();
                if (__any_sync(KV_FULL, over)) ok = false;
            }
        }
        if (lane == 0) {
            p.tel_out[c] = tel;
            if (p.feasible_out) p.feasible_out[c] = ok ? 1 : 0;
        }
    }
}
