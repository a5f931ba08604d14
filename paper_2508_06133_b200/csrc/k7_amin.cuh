// K7 -- Sorted-F + A_min, Phase 2 (Section 5.5 "Handling Prediction Uncertainty via Adaptive Output
// Length Refinement"; Algorithm 5, the supplement to Section 5): the executor when only a lower bound l_i <= o_i of
// every decode length is known.  Many independent scenarios (a backlog, its list and one vector of
// lower bounds each), one CTA per scenario.
//
// Every request carries a running estimate e_i (initially l_i).  Iteration t = 1, 2, ...:
//   1. requests that have run their o_i rounds leave; every other running request is about to run
//      round number t - p_i, so e_i <- max(e_i, t - p_i);
//   2. the head of the pending queue (list order) starts, p = t - 1, iff the memory PROJECTED from
//      the estimates stays within M in every round >= t with it; the first refusal ends the round's
//      admissions (Algorithm 1, Phase 2, on the estimates);
//   3. while the projection exceeds M, the running request with the smallest estimate (ties: lower
//      request index) is evicted: it loses its progress, keeps its estimate and goes back to its
//      place in the list;
//   4. the round runs.
//
// How the kernel avoids touching every running request in every round.
//   The projected memory of the rounds from t on is a chunked timeline (sim_chunk.cuh; a start p is the
//   simulator's round p + 1): request j contributes s_j + (tau - p_j) for
//   tau in [p_j + 1, p_j + e_j].  A request whose estimate e (fixed at its admission) is below its
//   true length o is OVERDUE in rounds p+e+1 .. p+o: there its estimate is t - p, i.e. step 1 extends
//   its projection by exactly the current round.  The overdue requests are kept as two aggregates,
//   cnt = how many and A = sum of (s_j - p_j), so step 1 adds A + cnt * t to round t; a request joins the
//   aggregates at p+e+1 and leaves them at p+o+1 through per-round event cells (ev, dA) written when
//   it is admitted (and taken back if it is evicted).  A is kept modulo 2^32: the sum A + cnt * t is
//   a memory amount and fits, its two terms need not.  The estimate of a running request is never
//   stored: it is max(e at admission, t - p).
//   The projection is within M in every round >= t at the end of an iteration, so only step 1 can
//   break it, and only in round t.
//   While the head of the queue is refused nothing is admitted and the projection only grows, so the
//   bound on its wait that the window test gives (a cell over budget by x at offset r needs min(x, r+1)
//   more rounds) stays valid until the next eviction.  Rounds in which nothing can happen (no overflow;
//   head still bound to wait, or not even its first round fits) are walked up to 32 at a time, one lane
//   each (the running aggregates of a round are prefix sums of the event cells).
//   The running requests are a compact list, so an eviction looks at them and not at everything that
//   has ever started; all warps of the CTA do.
// What bounds it: a scenario is a chain (2,000 requests of the paper's lengths: 2,400 admissions, 440
// evictions among 620 running, 1,450 walks), so the latency of each of these: about 350 cycles an admission, 750 a walk of up
// to 32 rounds, and an eviction 4,050 with one warp looking through the list, 1,100 with four.  The events of a round's
// admissions are put together, a lane each (they were 300 of 890 cycles per admission).  Kernel with 1 / 64 / 592
// scenarios (l uniform in [o / 2, o]) 2.71 / 2.80 / 5.37 -> 1.99 / 2.05 / 3.97 ms, the call around it 2.83 / 3.30 / 9.72 -> 2.12 /
// 2.57 / 8.2.
#pragma once

#include "common.cuh"
#include "sim_chunk.cuh"

#define K7_WARPS 4               // one runs the scenario, all of them look for the request to evict
#define K7_MAX_N 4096
#define K7_MAX_O 8192
#define K7_ID_BITS 12            // (estimate << 12) | id fits 32 bits

struct AminParams {
    int n_max;
    const int* n_each;           // [B]
    const int* s;                // [B, n_max] by request id
    const int* lower;
    const int* o;
    const int* order;            // [B, n_max] the list: request ids; or one row shared by all (order_stride 0)
    size_t order_stride;
    int M;
    int L;                       // event ring length, a power of two >= the longest decode + 2
    int sim_L;                   // ints per simulator state
    int* start_out;              // [B, n_max] by request id
    i64* tel_out;                // [B] sum of (p + o)
    i64* evict_out;              // [B] evictions
    i64* peak_out;               // [B] largest memory actually in use in a round
    int* status;
};

__host__ __device__ inline size_t k7_smem_bytes(int ring_cells, int n_max, int L) {
    return ((size_t)ring_cells + 4 * (size_t)n_max + 2 * (size_t)L) * sizeof(int) + 2 * (size_t)n_max * sizeof(unsigned short) + 16;
}

// Smallest (estimate, request id) of the running ones that this warp looks at, and its place in the list: to sh.
struct K7Scan {
    int t, nrun;                                                  // nrun < 0: the scenario is over
    unsigned key[K7_WARPS];
    int at[K7_WARPS];
};
__device__ __forceinline__ void k7_scan(K7Scan& sh, const unsigned short* run, const int* pp, const int* po, const int* pe,
                                        const unsigned short* pid) {
    const int warp = threadIdx.x >> 5, nrun = sh.nrun, t = sh.t;
    unsigned best = ~0u;
    int at = 0;
#pragma unroll 2
    for (int k = threadIdx.x; k < nrun; k += 32 * K7_WARPS) {
        const int r = run[k], p = pp[r];
        const unsigned key = t <= p + po[r] ? ((unsigned)max(pe[r], t - p) << K7_ID_BITS) | pid[r] : ~0u;
        if (key < best) { best = key; at = k; }
    }
    const unsigned least = __reduce_min_sync(KV_FULL, best);
    if (best == least && least != ~0u) { sh.key[warp] = least; sh.at[warp] = at; }      // one lane: ids differ
    else if (least == ~0u) sh.key[warp] = ~0u;
}

template <class SIM>
__global__ void __launch_bounds__(32 * K7_WARPS) k7_amin(const AminParams P) {
    extern __shared__ __align__(16) unsigned char k7_smem[];
    __shared__ K7Scan scan;
    const int lane = threadIdx.x & 31;
    const int b = blockIdx.x;
    const int n = P.n_each[b];
    const int nm = P.n_max;
    // per list position: prefill, true length, estimate while pending, start (-1: pending), request id
    int* ring = reinterpret_cast<int*>(k7_smem);
    int* ps = ring + SIM::ring_cells(P.sim_L);
    int* po = ps + nm;
    int* pe = po + nm;
    int* pp = pe + nm;
    int* ev = pp + nm;                                            // at the start of a round: 2^16 times the change of cnt, plus the requests that leave
    unsigned* dA = reinterpret_cast<unsigned*>(ev + P.L);         // change of A
    unsigned short* pid = reinterpret_cast<unsigned short*>(dA + P.L);
    unsigned short* run = pid + nm;                               // positions that run (and some that have finished)

    const size_t base = (size_t)b * nm;
    const int* ord = P.order + (size_t)b * P.order_stride;
    {
        bool bad = false;
        for (int q = threadIdx.x; q < n; q += 32 * K7_WARPS) {
            const int id = ord[q];
            if (id < 0 || id >= n) { bad = true; continue; }      // never read outside the row
            ps[q] = P.s[base + id]; po[q] = P.o[base + id]; pe[q] = P.lower[base + id];
            pp[q] = -1; pid[q] = (unsigned short)id;
        }
        for (int k = threadIdx.x; k < P.L; k += 32 * K7_WARPS) { ev[k] = 0; dA[k] = 0u; }
        if (__syncthreads_or(bad)) {
            if (threadIdx.x == 0) atomicExch(P.status, KV_DEV_LOOP_CAP);
            return;
        }
    }
    if (threadIdx.x >= 32) {                                      // called at every eviction, and at the end
        for (;;) {
            __syncthreads();
            if (scan.nrun < 0) return;
            k7_scan(scan, run, pp, po, pe, pid);
            __syncthreads();
        }
    }
    i64 sum_o = 0;
    for (int q = lane; q < n; q += 32) sum_o += po[q];
    for (int d = 16; d >= 1; d >>= 1) sum_o += __shfl_xor_sync(KV_FULL, sum_o, d);
    i64 round_cap = 16 + sum_o * (i64)(n + 1);
    if (round_cap > (1ll << 30)) round_cap = 1ll << 30;           // t stays a 32-bit round index

    const int mask = P.L - 1;
    const int M = P.M;
    SIM sim;
    sim.attach(ring, P.sim_L);
    sim.reset(M, 1);                                              // the simulator's round is the iteration t
    int remaining = n, peak = 0, nrun = 0;
    unsigned cnt = 0, A = 0;
    int head = 0, frontier = 0, npe = 0;     // first pending position; first never-started one; pending ones below it
    int t_ok = 1;                            // the head cannot start in an iteration before this one
    i64 evictions = 0;
    bool failed = false, done = false;

    for (i64 turn = 0;; ++turn) {
        if (turn > round_cap) { failed = true; break; }
        // rounds in which nothing can be decided (step 1 only): the lanes whose round of the chunk is still
        // to come take one each.  A round reads only its own cell and the running (cnt, A, remaining),
        // which are prefix sums of the event cells; the walk stops at the first round that needs a
        // decision (or ends the run).
        const int head_s = head < n ? ps[head] : 0;
        for (;;) {
            const int tau = sim.t & 31;
            const bool live = lane >= tau;
            const int round = sim.x0, k = round & mask;
            int es = live ? ev[k] : 0;
            unsigned as = live ? dA[k] : 0u;
            if (__any_sync(KV_FULL, es != 0 || as != 0u)) {
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int e2 = __shfl_up_sync(KV_FULL, es, d);
                    const unsigned a2 = __shfl_up_sync(KV_FULL, as, d);
                    if (lane >= d) { es += e2; as += a2; }
                }
            }
            const unsigned cnt_l = cnt + (unsigned)(es >> 16), A_l = A + as;
            const int rem_l = remaining - (es & 0xffff);
            const int u = sim.cur + M - round + (int)(A_l + cnt_l * (unsigned)round);
            const bool end = live && rem_l == 0;
            // the head's first round is the current one: if it does not fit there, the window test cannot
            // succeed in this iteration
            const bool work = live && (u > M || (head < n && round >= t_ok && u + head_s + 1 <= M));
            const bool cap = (i64)round >= round_cap;
            const unsigned ends = __ballot_sync(KV_FULL, end), works = __ballot_sync(KV_FULL, work);
            const unsigned stops = ends | works | __ballot_sync(KV_FULL, live && cap);
            const int first = stops ? __ffs(stops) - 1 : 32;
            if (live && lane <= first) { ev[k] = 0; dA[k] = 0u; }                        // events consumed
            const int run_max = kv_warp_max(live && lane < first ? u : 0);
            peak = max(peak, run_max);
            const int src = first < 32 ? first : 31;
            cnt = __shfl_sync(KV_FULL, cnt_l, src);
            A = __shfl_sync(KV_FULL, A_l, src);
            remaining = __shfl_sync(KV_FULL, rem_l, src);
            if (first < 32) {
                if (lane == first) sim.cur = u + round - M;                             // step 1 of the round that is decided
                sim.t += first - tau;
                if ((ends >> first) & 1u) done = true;
                else if (!((works >> first) & 1u)) failed = true;
                break;
            }
            sim.t = sim.tn; sim.rotate();
        }
        if (done || failed) break;
        const int t = sim.t;

        // ---- step 2: admissions of iteration t
        if (head < n && t >= t_ok) {
            const int had = nrun;
            int s = ps[head], e = pe[head];
            for (;;) {
                const int q = head, q1 = q + 1 < n ? q + 1 : q, s1 = ps[q1], e1 = pe[q1];      // the next one, mostly
                const int need = sim.need(s + 1, e - 1);
                if (need > 0) { t_ok = t + need; break; }
                sim.add(s + 1, e - 1);
                run[KV_IDX(nrun, nm, 1102)] = (unsigned short)q;
                ++nrun;
                if (q == frontier) ++frontier; else --npe;
                if (npe == 0) {
                    head = frontier;
                } else {                                           // an evicted request further down the list
                    int found = INT_MAX;
                    for (int k0 = q + 1; k0 < frontier && found == INT_MAX; k0 += 32) {
                        const unsigned v = __ballot_sync(KV_FULL, k0 + lane < frontier && pp[k0 + lane] < 0);
                        if (v) found = k0 + __ffs(v) - 1;
                    }
                    head = found;
                    if (head == INT_MAX) { failed = true; break; }
                }
                if (head >= n) break;
                s = s1; e = e1;
                if (head != q1) { s = ps[head]; e = pe[head]; }
            }
            __syncwarp();
            // their events: overdue in rounds t+e .. t+o-1 if the estimate is short, then over
            for (int k = had + lane; k < nrun; k += 32) {
                const int q = run[k], o = po[q], est = pe[q];
                const unsigned v = (unsigned)(ps[q] - (t - 1));
                pp[q] = t - 1;
                if (est < o) {
                    atomicAdd(&ev[(t + est) & mask], 1 << 16); atomicAdd(&dA[(t + est) & mask], v);
                    atomicAdd(&dA[(t + o) & mask], 0u - v);
                }
                atomicAdd(&ev[(t + o) & mask], est < o ? 1 - (1 << 16) : 1);
            }
            __syncwarp();
            if (failed) break;
        }

        // ---- step 3: ordered eviction while round t is over budget
        for (;;) {
            const int used = __shfl_sync(KV_FULL, sim.cur + M - sim.x0, sim.t & 31);
            if (used <= M) { peak = max(peak, used); break; }
            // smallest (estimate, request id) among the running
            if (lane == 0) { scan.t = t; scan.nrun = nrun; }
            __syncthreads();
            k7_scan(scan, run, pp, po, pe, pid);
            __syncthreads();
            const unsigned key = lane < K7_WARPS ? scan.key[lane] : ~0u, least = __reduce_min_sync(KV_FULL, key);
            if (least == ~0u) { failed = true; break; }
            const int est = (int)(least >> K7_ID_BITS);
            const int at = scan.at[__ffs(__ballot_sync(KV_FULL, key == least)) - 1];
            const int q = run[KV_IDX(at, nm, 1103)];
            const int p = pp[q], s = ps[q], o = po[q], e0 = pe[q];
            sim.remove(s - p, p + est);        // what is left of its projection
            const unsigned v = (unsigned)(s - p);
            const bool overdue = e0 < o && t >= p + e0 + 1;
            if (overdue) { cnt -= 1u; A -= v; }
            __syncwarp();
            --nrun;
            if (lane == 0) {
                run[at] = run[nrun];
                if (e0 < o) {
                    if (!overdue) { ev[(p + e0 + 1) & mask] -= 1 << 16; dA[(p + e0 + 1) & mask] -= v; }
                    ev[(p + o + 1) & mask] += 1 << 16; dA[(p + o + 1) & mask] += v;
                }
                ev[(p + o + 1) & mask] -= 1;
                pe[q] = est;
                pp[q] = -1;
            }
            __syncwarp();
            ++evictions; ++npe;
            head = min(head, q);
            t_ok = t + 1;
            // as many as have started and neither left nor been evicted; drop what has finished
            if (2 * (remaining - (n - frontier) - npe) < nrun) {
                int kept = 0;
                for (int k0 = 0; k0 < nrun; k0 += 32) {
                    const int k = k0 + lane, r = k < nrun ? run[k] : 0;
                    const bool keep = k < nrun && t <= pp[r] + po[r];
                    const unsigned w = __ballot_sync(KV_FULL, keep);
                    if (keep) run[kept + __popc(w & ((1u << lane) - 1u))] = (unsigned short)r;
                    kept += __popc(w);
                    __syncwarp();
                }
                nrun = kept;
            }
            __syncwarp();
        }
        if (failed) break;
        // ---- step 4: the round runs
        if (++sim.t == sim.tn) sim.rotate();
    }
    if (lane == 0) scan.nrun = -1;
    __syncthreads();
    if (failed) {
        if (lane == 0) atomicExch(P.status, KV_DEV_LOOP_CAP);
        return;
    }
    i64 part = 0;
    for (int q = lane; q < n; q += 32) {
        P.start_out[base + KV_IDX(pid[q], n, 1101)] = pp[q];
        part += (i64)pp[q] + po[q];
    }
    for (int d = 16; d >= 1; d >>= 1) part += __shfl_xor_sync(KV_FULL, part, d);
    if (lane == 0) { P.tel_out[b] = part; P.evict_out[b] = evictions; P.peak_out[b] = peak; }
}
