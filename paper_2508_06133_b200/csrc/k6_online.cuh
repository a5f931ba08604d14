// K6 -- online arrivals (Section 6.2 "Heuristics under Online Arrival"; Section 7, "Experiment under
// Online Poisson Arrivals"): many independent arrival streams, one warp each, one policy per launch.
//
// Model.  Request i arrives at the integer time a_i >= 0 (non-decreasing in i) and may start at any
// p_i >= a_i: it is first seen by iteration a_i + 1.  In iteration t the policy orders the pending
// requests and the executor admits the longest prefix of that order that fits the live memory
// profile (Algorithm 1, Phase 2: stop at the first request that does not fit).
//   FCFS            arrival order;
//   SOF             ascending (o, index), recomputed every iteration;
//   Sorted-F-Online a cached priority list: arrivals go to its tail; it is planned again when it has
//                   never been planned, `period` iterations after the last plan, when it had run
//                   empty, or when the arrivals since the last plan reach half of the backlog at
//                   that plan.  A plan sorts the pending requests by ascending (s+o, index), orders
//                   the first `lookahead` of them by Sorted-F with Algorithm 3 (batch after batch,
//                   every batch by ascending (o, index)) and lets the others follow in sorted order.
//
// The iterations are not walked one by one.  Nothing changes between two iterations unless a
// request arrives, a plan is due, or the head of the list starts; while the head is refused, the
// window test yields the same lower bound on the wait as in the offline simulator (a cell over
// budget by e at offset r needs min(e, r+1) more rounds), so the loop jumps to the earliest of:
// that bound, the next arrival, the next due plan.
//
// What bounds it: one stream is a chain of admissions, plans and waits (about 1,240, 540 and 1,200 for
// the busiest stream of the paper's experiment), so the latency of each of them:
//   - a plan's batches are built when the head of the list reaches them.  A plan lives a few
//     iterations, in which the first of its batches (of up to 18) is hardly ever used up: one batch
//     per plan is built instead of 16, and 1/25 of the swaps is made.  What the list would have held
//     behind that point is a function of the window alone, so nothing else changes;
//   - the pending requests stay sorted from plan to plan, new ones are merged in;
//   - the memory profile is the chunked simulator (sim_chunk.cuh), so a test costs the same for every
//     decode length; one warp does everything, without block barriers.
#pragma once

#include "common.cuh"
#include "k2_local_swap.cuh"
#include "sim_chunk.cuh"

#define K6_THREADS 32
#define K6_MAX_N 2048            // requests per stream
#define K6_MAX_LOOKAHEAD 1024
#define K6_MAX_O 8192
#define K6_IDX_BITS 12           // (o << 12) | index fits 32 bits for o <= 2^14, index < 2^12

struct OnlineParams {
    int n_max;
    const int* n_each;           // [B]
    const int* a;                // [B, n_max]
    const int* s;
    const int* o;
    int M;
    int policy, period, lookahead;
    int L;                       // ints per simulator state
    int* start_out;              // [B, n_max]
    i64* latency_out;            // [B]  sum of (p + o - a)
    int* status;
};

typedef unsigned short k6_ix;

// Algorithm 3 on a window of up to 128 requests by one warp, in registers: lane l holds the positions
// l, l + 32, ..., and the members l, l + 32, ... of X.  The members are asked one after the other in walking
// order (a comparison with every position outside X at once), so the first that has a partner ends the
// turn.  A swap of the windows of the paper's experiment (67 requests, 12 members) takes a quarter of
// what it takes through the prefix minima of k2l_batch.  Same contract as k2l_batch.
#define K6_SMALL 128
__device__ int k6_batch_small(const K2lArrays<k6_ix>& a, int m, int M, int* status) {
    constexpr int R = K6_SMALL / 32;
    const int lane = threadIdx.x & 31;
    int T[R], O[R], MT[R], MO[R], MP[R];                 // positions; members: size, weight, position
    unsigned out = 0;                                    // bit i: position lane + 32 i exists and is outside X
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int p = lane + 32 * i;
        T[i] = p < m ? a.T[p] : INT_MAX; O[i] = p < m ? a.O[p] : INT_MAX;
        if (p < m) out |= 1u << i;
    }
    // first fit = longest prefix with sum(s+o) <= M; sums are held at M + 1
    int k0 = 0, mem = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        if (k0 < 32 * i) break;
        const unsigned most = (unsigned)M + 1u;
        unsigned incl = min((unsigned)T[i], most);
        for (int d = 1; d < 32; d <<= 1) { const unsigned y = __shfl_up_sync(KV_FULL, incl, d); if (lane >= d) incl = min(incl + y, most); }
        incl = min(incl + (unsigned)mem, most);
        const unsigned v = __ballot_sync(KV_FULL, lane + 32 * i < m && incl <= (unsigned)M);
        const int c = __popc(v);
        if (c > 0) mem = (int)__shfl_sync(KV_FULL, incl, c - 1);
        if (lane < c) out &= ~(1u << i);
        k0 += c;
    }
#pragma unroll
    for (int i = 0; i < R; ++i) { MT[i] = T[i]; MO[i] = O[i]; MP[i] = lane + 32 * i; }      // valid below k0
    const i64 step_cap = kv_loop_cap(((i64)k0 << 30) + 16);
    for (i64 step = 0;; ++step) {
        bool swapped = false;
#pragma unroll
        for (int g = 0; g < R; ++g) {
            if (swapped || k0 <= 32 * g) break;
            const int cnt = min(32, k0 - 32 * g);
            for (int k = 0; k < cnt; ++k) {
                const int tk = __shfl_sync(KV_FULL, MT[g], k), ok = __shfl_sync(KV_FULL, MO[g], k);
                const int cap = M - mem + tk;
                bool hit[R], any = false;
#pragma unroll
                for (int i = 0; i < R; ++i) { hit[i] = ((out >> i) & 1u) && T[i] <= cap && O[i] < ok; any = any || hit[i]; }
                if (!__any_sync(KV_FULL, any)) continue;
                // the first such position
                int j = 0, tj = 0, oj = 0;
                bool found = false;
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const unsigned v = __ballot_sync(KV_FULL, hit[i]);
                    if (!found && v) {
                        const int l = __ffs(v) - 1;
                        j = l + 32 * i; tj = __shfl_sync(KV_FULL, T[i], l); oj = __shfl_sync(KV_FULL, O[i], l);
                        found = true;
                    }
                }
                const int pos = __shfl_sync(KV_FULL, MP[g], k);
                if (lane == (pos & 31)) out |= 1u << (pos >> 5);
                if (lane == (j & 31)) out &= ~(1u << (j >> 5));
                mem += tj - tk;
                if (lane == k) { MT[g] = tj; MO[g] = oj; MP[g] = j; }
                swapped = true;
                break;
            }
        }
        if (!swapped) break;
        if (step > step_cap) { if (lane == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int p = lane + 32 * i;
        if (p < m && !((out >> i) & 1u)) a.id[p] |= K2L_IN;
        if (p < k0) a.xpos[p] = (k6_ix)MP[i];
    }
    __syncwarp();
    return k0;
}

// dynamic shared memory: the simulator's ring; a, s, o, started flags and two id lists of n_max; the
// local swap scratch and one batch for `lookahead` requests
__host__ __device__ inline size_t k6_smem_bytes(int ring_cells, int n_max, int lookahead) {
    return ((size_t)ring_cells + 6 * (size_t)n_max + lookahead) * sizeof(int) + k2l_bytes<k6_ix>(lookahead) + 64;
}

struct K6Stream {
    int *sa, *ss, *so, *started;
    int *S, *S2;                 // pending requests of the last plan by ascending (s+o, index); scratch
    int* B;                      // the batch in hand by ascending (o, index)
    K2lArrays<k6_ix> win;        // what is left of the plan's window
    int n, nvis;
    int slen, sused;             // S[0 .. slen): the window first; sused: how far the list has come in it
    int wlen;                    // requests left in the window
    int blen, bused;
    int tail;                    // next arrival behind the plan

    __device__ __forceinline__ int size_of(int id) const { return ss[id] + so[id]; }

    // S <- the requests of S that have not started, with the arrivals tail .. nvis-1 that have not
    // started merged in by (s+o, index); arrivals have higher indices than everything in S
    __device__ void merge(int lane) {
        int m = 0;
        for (int base = 0; base < slen; base += 32) {
            const int k = base + lane;
            const int id = k < slen ? S[k] : 0;
            const bool keep = k < slen && !started[id];
            const unsigned v = __ballot_sync(KV_FULL, keep);
            if (keep) S[m + __popc(v & ((1u << lane) - 1u))] = id;
            m += __popc(v);
            __syncwarp();
        }
        int c = 0;                                       // new ones, in arrival order, at the end of S2
        int* fresh = S2 + n - (nvis - tail);
        for (int base = tail; base < nvis; base += 32) {
            const int id = base + lane;
            const bool keep = id < nvis && !started[id];
            const unsigned v = __ballot_sync(KV_FULL, keep);
            if (keep) fresh[c + __popc(v & ((1u << lane) - 1u))] = id;
            c += __popc(v);
        }
        __syncwarp();
        if (c > 0) {
            // new position of a new one: the old ones not above its size + its rank among the new;
            // of an old one: its old position + the new ones below its size
            for (int k = lane; k < c; k += 32) {
                const int id = fresh[k], T = size_of(id);
                int lo = 0, hi = m;
                while (lo < hi) { const int mid = (lo + hi) >> 1; if (size_of(S[mid]) <= T) lo = mid + 1; else hi = mid; }
                int r = lo;
                for (int j = 0; j < c; ++j) { const int Tj = size_of(fresh[j]); r += (Tj < T || (Tj == T && j < k)) ? 1 : 0; }
                started[id] = -1 - r;                    // its position, until everything has moved
            }
            __syncwarp();
            // old ones move up, from the end so that nothing is overwritten before it is read
            for (int base = (m - 1) & ~31; base >= 0 && m > 0; base -= 32) {
                const int k = base + lane;
                int id = 0, r = 0;
                if (k < m) {
                    id = S[k];
                    const int T = size_of(id);
                    for (int j = 0; j < c; ++j) r += size_of(fresh[j]) < T ? 1 : 0;
                }
                __syncwarp();
                if (k < m) S[KV_IDX(k + r, n, 1002)] = id;
                __syncwarp();
            }
            for (int k = lane; k < c; k += 32) {
                const int id = fresh[k];
                S[KV_IDX(-1 - started[id], n, 1003)] = id;
                started[id] = 0;
            }
            __syncwarp();
        }
        slen = m + c;
    }

    // a new plan over everything pending
    __device__ void plan(int lookahead, int lane) {
        merge(lane);
        tail = nvis;
        wlen = min(slen, lookahead);
        for (int k = lane; k < wlen; k += 32) {
            const int id = S[k];
            win.id[k] = id; win.T[k] = size_of(id); win.O[k] = so[id];
        }
        sused = wlen; blen = 0; bused = 0;
        __syncwarp();
    }

    // head of the priority list, -1: nothing pending
    __device__ int head(int M, int lane, int* status, K2lShared<32>& sh) {
        if (bused == blen && wlen > 0) {
            const int k0 = wlen <= K6_SMALL ? k6_batch_small(win, wlen, M, status)
                                            : k2l_batch<32, k6_ix>(win, wlen, (i64)M, status, sh);
            if (k0 < 1) { if (lane == 0) atomicExch(status, KV_DEV_LOOP_CAP); wlen = 0; return -1; }
            // the batch by ascending (o, index): rank of every member among the members
            for (int k = lane; k < k0; k += 32) {
                const int id = win.id[win.xpos[k]] & ~K2L_IN;
                S2[k] = (so[id] << K6_IDX_BITS) | id;
            }
            __syncwarp();
            for (int k = lane; k < k0; k += 32) {
                const int key = S2[k];
                int rank = 0;
                for (int j = 0; j < k0; ++j) rank += S2[j] < key ? 1 : 0;
                B[rank] = key & ((1 << K6_IDX_BITS) - 1);
            }
            __syncwarp();
            wlen = k2l_compact<32, k6_ix>(win, wlen, sh);
            blen = k0; bused = 0;
        }
        if (bused < blen) return B[bused];
        if (sused < slen) return S[sused];
        return tail < nvis ? tail : -1;
    }
    __device__ __forceinline__ void pop() {
        if (bused < blen) ++bused;
        else if (sused < slen) ++sused;
        else ++tail;
    }
};

template <class SIM>
__global__ void __launch_bounds__(K6_THREADS) k6_online(const OnlineParams P) {
    extern __shared__ __align__(16) unsigned char k6_smem[];
    __shared__ K2lShared<32> sh;
    const int lane = threadIdx.x;
    const int b = blockIdx.x;
    const int n = P.n_each[b];
    const int nm = P.n_max;
    K6Stream q;
    int* ring = reinterpret_cast<int*>(k6_smem);
    q.sa = ring + SIM::ring_cells(P.L);
    q.ss = q.sa + nm; q.so = q.ss + nm; q.started = q.so + nm; q.S = q.started + nm; q.S2 = q.S + nm;
    q.B = q.S2 + nm;
    {
        const size_t at = (size_t)((unsigned char*)(q.B + P.lookahead) - k6_smem);
        q.win = k2l_arrays<k6_ix>(k6_smem + ((at + 15) & ~(size_t)15), P.lookahead);
    }
    q.n = n; q.nvis = 0; q.slen = 0; q.sused = 0; q.wlen = 0; q.blen = 0; q.bused = 0; q.tail = 0;

    const size_t base = (size_t)b * nm;
    i64 sum_o = 0;
    for (int i = lane; i < n; i += 32) {
        q.sa[i] = P.a[base + i]; q.ss[i] = P.s[base + i]; q.so[i] = P.o[base + i];
        q.started[i] = 0;
        sum_o += q.so[i];
    }
    for (int d = 16; d >= 1; d >>= 1) sum_o += __shfl_xor_sync(KV_FULL, sum_o, d);
    __syncwarp();
    const i64 horizon = 2 + sum_o + q.sa[n - 1];
    const i64 turn_cap = kv_loop_cap(4 * (horizon + n) + 64);   // every turn is an arrival, a plan or a wait that ends

    SIM sim;
    sim.attach(ring, P.L);
    sim.reset(P.M);

    int t = 1, remaining = n;                           // iteration t: the simulator stands at round t - 1
    bool computed = false;
    int t_last = 0, backlog_last = 0, new_since = 0;
    bool changed = true;                                // pending set differs from the one last planned
    i64 latency = 0;

    for (i64 turn = 0; remaining > 0; ++turn) {
        if (turn > turn_cap) { if (lane == 0) atomicExch(P.status, KV_DEV_LOOP_CAP); break; }
        // arrivals seen by iteration t
        const bool was_empty = q.nvis == n - remaining;
        const int old = q.nvis;
        for (;;) {                                      // 32 at a time: arrivals are in order
            const int i = q.nvis + lane;
            const int c = __popc(__ballot_sync(KV_FULL, i < n && q.sa[i] <= t - 1));
            q.nvis += c;
            if (c < 32) break;
        }
        const int newly = q.nvis - old, pending = q.nvis - (n - remaining);
        if (P.policy == SCHED_POLICY_SORTED_F) {
            new_since += newly;
            if (newly > 0) changed = true;
            const bool due = pending > 0 && (!computed || t - t_last >= P.period || was_empty || 2 * new_since >= backlog_last);
            if (due && !changed) {
                // same pending set as at the last plan (no arrival, no start since): the plan is a
                // function of that set alone, so it would come out as the list already is
                t_last = t;
            } else if (due) {
                q.plan(P.lookahead, lane);
                computed = true; t_last = t; backlog_last = pending; new_since = 0;
                changed = false;
            }
        }
        // ---- admission: the longest prefix of the list that fits
        int r = -1, need = 0;
        for (;;) {
            if (P.policy == SCHED_POLICY_FCFS) {
                r = q.tail < q.nvis ? q.tail : -1;
            } else if (P.policy == SCHED_POLICY_SOF) {
                int best = INT_MAX;
                for (int i = lane; i < q.nvis; i += 32)
                    if (!q.started[i]) best = min(best, (q.so[i] << K6_IDX_BITS) | i);
                best = kv_warp_min(best);
                r = best == INT_MAX ? -1 : (best & ((1 << K6_IDX_BITS) - 1));
            } else {
                r = q.head(P.M, lane, P.status, sh);
            }
            if (r < 0) break;
            const int s = q.ss[r], o = q.so[r];
            need = sim.need(s + 1, o - 1);
            if (need > 0) break;
            sim.add(s + 1, o - 1);
            if (lane == 0) { P.start_out[base + KV_IDX(r, n, 1001)] = t - 1; q.started[r] = 1; }
            latency += (i64)(t - 1) + o - q.sa[r];
            --remaining;
            if (P.policy == SCHED_POLICY_FCFS) ++q.tail;
            else if (P.policy == SCHED_POLICY_SORTED_F) { q.pop(); changed = true; }
            __syncwarp();
        }
        if (remaining == 0) break;
        // ---- the next iteration at which anything can change
        i64 t_next;
        if (r < 0) {
            if (q.nvis == n) { if (lane == 0) atomicExch(P.status, KV_DEV_LOOP_CAP); break; }   // a batch gave up
            t_next = (i64)q.sa[q.nvis] + 1;             // nothing pending: wait for the next arrival
        } else {
            t_next = (i64)t + need;
            if (q.nvis < n) t_next = min(t_next, (i64)q.sa[q.nvis] + 1);
            if (P.policy == SCHED_POLICY_SORTED_F) t_next = min(t_next, (i64)t_last + P.period);
        }
        sim.skip((int)(t_next - t), P.M);
        t = (int)t_next;
    }
    if (lane == 0) P.latency_out[b] = latency;
}
