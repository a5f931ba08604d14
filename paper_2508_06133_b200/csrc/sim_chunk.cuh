// Chunked schedule simulator: Phase 2 of Algorithm 1 (the supplement to Section 3) for one ordered
// list, one warp per candidate, at a cost per admission that does not depend on the window's length.
//
// Rounds are 0-based (x = tau - 1 for the paper's round tau); a request that starts at p is resident
// in rounds p .. p+o-1 and uses s + 1 + (x - p) tokens in round x (Section 2.1: token j needs s + j).
// t is the round the next request may start at.  Starts never go backwards along the list (a request
// that does not fit blocks everything behind it), so every window that is ever tested or filled
// begins at the current t: an admission touches a PREFIX of the rounds still ahead.
//
// The timeline is cut into chunks of 32 rounds.  With V[x] = (tokens in use in round x) + x, a request
// (s, o) fits at t  <=>  V[x] <= M - s - 1 + t for every x in [t, t+o), and its admission is
// V[x] += (s+1-t) + x on the same rounds.
//   chunk 0 (the one t lies in)   the exact V[x], one round per lane, in a register.
//   far chunks                    an admission that covers a far chunk whole adds a constant and a
//       slope to it, so only their sums are kept: A = sum of (s+1-p), C = how many; the chunk in which
//       a window ends is the one chunk per admission whose 32 cells are written (a ring in shared
//       memory, one column per lane: own[x] = sum of (s+1-p) + x over the windows that end in the
//       chunk and reach x).  V[x] = own[x] + A + C x + x.  Lane l holds A, C of the (l+1)-th chunk
//       ahead (and of every 32nd behind it for decodes beyond 1,025 rounds: NM registers of each).
//   U (per far chunk)             an upper bound of V over the chunk: every admission that reaches the
//       chunk raises it by its ramp's value in the chunk's last round.  One compare per lane tests 32
//       chunks.  Where U says "perhaps", the chunk's cells are put together, U becomes their exact
//       maximum and the cells decide.  Occupancy falls behind the chunk t lies in, so this is rare:
//       0.01 to 0.1 chunks per admission on the synthetic backlogs (and 0.3 to 1.1 waits).
// Measured against a register-resident timeline that tested and filled every cell of the window (one and
// a half instructions per 32 cells and admission), k3_eval_moves: 10,000 requests (decodes to 1,024),
// 65,536 moves 43.3 -> 33.0 ms; 100,000 requests (decodes to 4,096), 7,000 moves 108.8 -> 50.7 ms (40.7 with kGlobal), where
// the far part of the timeline was read and written in shared memory; one run of the 100,000 from the
// empty state (sorted_f) 71.6 -> 15.6 ms.  Bound by the issue rate: 80 instructions per admission, 0.87 of the slots.
// When t enters the next chunk its cells are put together from own, A and C, and the lanes' far
// values move down by one.
//
// Wait of a request that does not fit: a round over budget by e > 0 at offset r from t rules out every
// start before t + min(e, r+1) (either the ramp has dropped by e or the window has moved past the
// round); t moves by the largest such bound and the test is repeated.  Chunk 0 is asked first.
//
// What is kept is counted from T0 = t rounded down to a multiple of 32 (rounds, starts and with them V,
// A and U), so that one admission is a handful of three-input additions of per-lane constants that
// only change when t does; entering the next chunk takes 32 off every V and U and gives 32 C to A.
// The sum of starts is kept as the sum of t - T0 plus, per chunk entered, 32 for every request still
// to come.  A request is passed as sp = s + 1 and om = o - 1.
//
// Sums may wrap; V itself fits 31 bits (the host checks M, sum of o and n), so arithmetic modulo 2^32
// gives it exactly.
#pragma once

#include "common.cuh"

// kGlobal: the rings are in device memory.  A simulator for decodes up to 4,097 rounds has 16 KB of ring,
// so shared memory holds 13 of them per SM and registers 32; the ring is written without waiting and read once per
// 32 rounds.  100,000 requests, 7,000 moves, 1.0 rounds per request: 50.7 -> 40.7 ms; device_rings_fit has the rule.
//
// kShort: a window that ends in chunk 0 leaves everything else alone.  Where nearly every decode is a few rounds,
// a sweep takes 0.75 to 0.99 of the time (mean 2 to 10; without it 1.1 times that of the timeline of single
// cells that was here before); with longer ones the branches cost more than they save (mean 20: 0.92 to 1.07,
// mean 200: 1.04 to 1.11).  short_windows (api.cu) has the rule.
template <int NM, bool kGlobal_ = false, bool kShort = false>
struct ChunkSim {
    static constexpr bool kGlobal = kGlobal_;
    static constexpr int kWarps = NM == 1 || kGlobal ? 4 : NM == 2 ? 2 : 1;    // per CTA: 16 KB of shared rings
    static constexpr int kMinCtas = kGlobal ? 8 : 10;            // CTAs per SM the registers have to allow
    static constexpr bool kGroups = true;                           // has surely()
    static constexpr int kMeta = 32 + 96 * NM;                      // state ints besides the ring
    __host__ __device__ static constexpr int ring_cells(int L) { return L - kMeta; }   // shared-memory ints per warp

    int lane;
    int T0, tau;             // t = T0 + tau, 0 <= tau < 32
    int cur;                 // V of this lane's round of chunk 0
    int rl;                  // that round - t
    int xr, x31;             // first and last round of far chunk `lane` (the (lane+1)-th chunk ahead) - t
    int nkt;                 // M + tau
    int A[NM], C[NM], U[NM];
    int acc;                 // sum of tau over the admissions
    i64 tel;                 // the rest of the sum of completion times
    int* ring;               // this lane's column
    int mask;                // ring ints - 1, without the lane bits

    __device__ __forceinline__ void attach(int* ring_, int L) {
        lane = kv_lane();
        ring = ring_ + lane;
        mask = (ring_cells(L) - 1) & ~31;
    }
    __device__ __forceinline__ int* cells_of(int x) const { return ring + KV_IDX(x & mask, mask + 32, 151); }
    __device__ __forceinline__ static int cell(const int* p) { return kGlobal ? __ldcg(p) : *p; }
    __device__ __forceinline__ void set_time(int t, int M) {
        T0 = t & ~31; tau = t & 31;
        rl = lane - tau; xr = 32 * (lane + 1) - tau; x31 = xr + 31; nkt = M + tau;
        acc = 0;
    }
    __device__ __forceinline__ int start() const { return T0 + tau; }      // of the request admitted last

    // nothing is resident at t or later
    __device__ __forceinline__ void reset(int M, int t = 0) {
        set_time(t, M);
        cur = lane; tel = 0;
#pragma unroll
        for (int m = 0; m < NM; ++m) { A[m] = 0; C[m] = 0; U[m] = 32 * (lane + 1) + 1024 * m + 31; }
        for (int k = 0; k <= mask; k += 32) ring[KV_IDX(k, mask + 32, 152)] = 0;
        __syncwarp();
    }

    // snapshot: cur[32], then A, C, U of every m [32 each], then the ring
    __device__ __forceinline__ void load(const int* __restrict__ snap, const SnapHeader& h, int M, int left) {
        set_time(h.t, M);
        tel = (((i64)h.tel_hi << 32) | (i64)(unsigned)h.tel_lo) + (i64)T0 * left;
        const int4* src = reinterpret_cast<const int4*>(snap + kMeta) + lane;
        int4* dst = reinterpret_cast<int4*>(ring - lane) + lane;
        const int groups = (mask + 32) >> 2;
        for (int g = 0; g + lane < groups; g += 32) dst[KV_IDX(g, groups - lane, 153)] = src[g];
        cur = snap[lane];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            A[m] = snap[32 + 96 * m + lane]; C[m] = snap[64 + 96 * m + lane]; U[m] = snap[96 + 96 * m + lane];
        }
        __syncwarp();
    }
    // tel_before: sum of completion times of the requests admitted so far
    __device__ __forceinline__ void store(int* __restrict__ snap, SnapHeader* hdr, i64 tel_before) const {
        __syncwarp();
        const int4* src = reinterpret_cast<const int4*>(ring - lane) + lane;
        int4* dst = reinterpret_cast<int4*>(snap + kMeta) + lane;
        const int groups = (mask + 32) >> 2;
        for (int g = 0; g + lane < groups; g += 32) dst[g] = src[KV_IDX(g, groups - lane, 154)];
        __syncwarp();
        snap[lane] = cur;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            snap[32 + 96 * m + lane] = A[m]; snap[64 + 96 * m + lane] = C[m]; snap[96 + 96 * m + lane] = U[m];
        }
        if (lane == 0) {
            SnapHeader h; h.t = T0 + tau;
            h.tel_lo = (int)(tel_before & 0xffffffffll); h.tel_hi = (int)(tel_before >> 32);
            *hdr = h;
        }
    }
    // sum of the completion times of all requests; sum_o: decode lengths of those admitted here
    __device__ __forceinline__ i64 total(i64 sum_o) const { return tel + acc + sum_o; }

    // t has left chunk 0: the first far chunk takes its place, the others move down by one lane
    __device__ __forceinline__ void rotate(int left) {
        T0 += 32; tau -= 32; rl += 32; xr += 32; x31 += 32; nkt -= 32;
        tel += 32ll * left;
        int* p = cells_of(T0);
        const int from = (lane + 1) & 31;
        int ra[NM], rc[NM], ru[NM];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            rc[m] = __shfl_sync(KV_FULL, C[m], from);
            ra[m] = __shfl_sync(KV_FULL, A[m], from) + 32 * rc[m];
            ru[m] = __shfl_sync(KV_FULL, U[m], from) - 32;
        }
        // lane 31 has just received the values of the chunk that becomes chunk 0
        const int a = __shfl_sync(KV_FULL, ra[0], 31), c = __shfl_sync(KV_FULL, rc[0], 31) + 1;
        cur = cell(p) + a + c * lane;
        *p = 0;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int m1 = m + 1 < NM ? m + 1 : m;
            const bool last = lane == 31;
            A[m] = last ? (m + 1 < NM ? ra[m1] : 0) : ra[m];
            C[m] = last ? (m + 1 < NM ? rc[m1] : 0) : rc[m];
            U[m] = last ? (m + 1 < NM ? ru[m1] : 1024 * (m + 1) + 31) : ru[m];
        }
    }

    // far chunks of the window whose bound exceeds nk: exact maximum into U, wait bound of their cells
    __device__ __forceinline__ int far_need(int om, int nk) {
        int d = 0;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            unsigned todo = __ballot_sync(KV_FULL, xr + 1024 * m <= om && U[m] > nk);
            while (todo) {
                const int j = __ffs(todo) - 1;
                todo &= todo - 1;
                const int x0 = 32 * (j + 1) + 1024 * m;              // counted from T0
                const int a = __shfl_sync(KV_FULL, A[m], j), c = __shfl_sync(KV_FULL, C[m], j) + 1;
                const int v = cell(cells_of(T0 + x0)) + a + c * (x0 + lane);
                const int vmax = kv_warp_max(v);
                if (lane == j) U[m] = vmax;
                if (x0 + rl <= om) d = max(d, __viaddmin_s32(v, -nk, x0 + rl + 1));
            }
        }
        return kv_warp_max(d);
    }

    // One reduction answers for all lanes: above 0 the wait that chunk 0 asks for, 0 where a far bound
    // says "perhaps" (or a round fits exactly), below 0 everything is clear
    __device__ __forceinline__ int ask(int sp, int om) const {
        const int nk = nkt - sp;                         // it fits  <=>  V[x] <= nk in every round of the window
        int v = (unsigned)rl <= (unsigned)om ? __viaddmin_s32(cur, -nk, rl + 1) : INT_MIN;
        if (kShort && tau + om <= 31) return kv_warp_max(v);
        if (xr <= om && U[0] > nk) v = max(v, 0);
        if (NM > 1 && tau + om >= 1024 + 32) {
#pragma unroll
            for (int m = 1; m < NM; ++m) if (xr + 1024 * m <= om && U[m] > nk) v = max(v, 0);
        }
        return kv_warp_max(v);
    }
    // 0: (sp, om) fits at t; otherwise a lower bound of the rounds it has to wait
    __device__ __forceinline__ int test(int sp, int om) {
        const int d = ask(sp, om);
        if (d < 0) return 0;
        return d > 0 ? d : far_need(om, nkt - sp);
    }
    // t moves on by d rounds
    __device__ __forceinline__ void advance(int d, int left) {
        tau += d; rl -= d; xr -= d; x31 -= d; nkt += d;
        while (tau >= 32) rotate(left);
    }
    // the same for any d: a gap longer than every window leaves nothing resident
    __device__ __forceinline__ void skip(int d, int M) {
        if (d > mask + 64) reset(M, T0 + tau + d);
        else advance(d, 0);
    }
    // (sp, om) starts at t
    __device__ __forceinline__ void add(int sp, int om) {
        if ((unsigned)rl <= (unsigned)om) cur += sp + rl;
        if (kShort && tau + om <= 31) return;
        if (xr <= om) U[0] += sp + x31;
        if (x31 < om) { A[0] += sp - tau; C[0] += 1; }
        if (NM > 1 && tau + om >= 1024 + 32) {
#pragma unroll
            for (int m = 1; m < NM; ++m) {
                if (xr + 1024 * m <= om) U[m] += sp + x31 + 1024 * m;
                if (x31 + 1024 * m < om) { A[m] += sp - tau; C[m] += 1; }
            }
        }
        const int last = tau + om, back = (last & 31) - lane;       // the chunk the window ends in
        // an atomic without a result, by every lane: nothing waits for the old value, and adding zero costs
        // less than a branch around it (a window that ends in chunk 0 meets that chunk's own slot, unused)
        atomicAdd(cells_of(T0 + last), last > 31 && back >= 0 ? sp + om - back : 0);
    }

    // Takes back what is left (from t on) of a window whose ramp is a + x in round x, counted from T0, and
    // whose last round is `last`.  The bounds fall by the least the ramp has in a chunk it covers whole.
    __device__ __forceinline__ void remove(int a, int last) {
        if (rl >= 0 && lane <= last) cur -= a + lane;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int x = 32 * (lane + 1) + 1024 * m;
            if (x + 31 <= last) U[m] -= a + x;
            if (x + 31 < last) { A[m] -= a; C[m] -= 1; }
        }
        const int x = (last & ~31) + lane;                          // the chunk the window ends in
        if (last > 31 && x <= last) atomicAdd(cells_of(T0 + last), -(a + x));
    }

    // Whether requests of `size` tokens in all (s + o each), the longest with om = o - 1, certainly fit at t
    // one beside the other: none of them uses more than its s + o in any round.
    __device__ __forceinline__ bool surely(int size, int om) const {
        const int nk = nkt - size;
        bool over = (unsigned)rl <= (unsigned)om && cur > nk;
        over = over || (xr <= om && U[0] > nk);
        if (NM > 1 && tau + om >= 1024 + 32) {
#pragma unroll
            for (int m = 1; m < NM; ++m) over = over || (xr + 1024 * m <= om && U[m] > nk);
        }
        return !__any_sync(KV_FULL, over);
    }

    // The same result for a run that stands alone: one branch where the request does not wait.
    __device__ __forceinline__ bool admit_alone(int sp, int om, int left, int* status) {
        int v = ask(sp, om);
        const bool waited = v >= 0;                      // or a far bound had to be looked at
        if (waited) {
            for (int guard = 0;; ++guard) {
                const int d = v > 0 ? v : far_need(om, nkt - sp);
                if (d <= 0) break;
                advance(d, left);
                if (guard > kv_loop_cap(32 * mask + 2048)) { if (lane == 0) atomicExch(status, KV_DEV_LOOP_CAP); return true; }
                v = ask(sp, om);
                if (v < 0) break;
            }
        }
        add(sp, om);
        acc += tau;
        return waited;
    }

    // Admit one request (sp = s + 1, om = o - 1) at the earliest start; all 32 lanes call this with
    // identical arguments.  left: requests still to be admitted, this one included.  Returns whether it
    // had to wait.
    __device__ __forceinline__ bool admit(int sp, int om, int left, int* status) {
        bool waited = false;
        for (int guard = 0;; ++guard) {
            const int d = test(sp, om);
            if (d <= 0) break;
            waited = true;
            advance(d, left);
            if (guard > kv_loop_cap(32 * mask + 2048)) { if (lane == 0) atomicExch(status, KV_DEV_LOOP_CAP); return true; }
        }
        add(sp, om);
        acc += tau;
        return waited;
    }
};

// Up to 32 consecutive requests of a list, (s, o) of the k-th in lane k, the list going on with
// left - cnt behind them.  Returns the start of the k-th in lane k.
//
// kGroups: where memory is not short, several requests start in the same round; four at a time are then
// asked for together, and if their sizes certainly fit they are added one behind the other without a test
// each, so that the additions overlap.  Tried only behind a request that did not wait.  For a run that
// stands alone, where the latency of an admission counts: 0.251 -> 0.226 ms for 1,000 requests, 1.83 ->
// 1.69 ms for 10,000.  Many runs side by side are bound by instructions, of which the tries cost more than
// they save (8.70 -> 9.49 ms for 16,384 moves of the 10,000), so they go without.
template <bool kGroups, class SIM>
__device__ __forceinline__ int sim_run_block(SIM& sim, int2 so, int cnt, int left, int* status) {
    const int lane = threadIdx.x & 31, sp = so.x + 1, om = so.y - 1;
    int mine = 0;
    if constexpr (kGroups && SIM::kGroups) {
        int size = so.x + so.y, longest = om;                       // of the aligned four this lane is in
        size += __shfl_xor_sync(KV_FULL, size, 1); size += __shfl_xor_sync(KV_FULL, size, 2);
        longest = max(longest, __shfl_xor_sync(KV_FULL, longest, 1));
        longest = max(longest, __shfl_xor_sync(KV_FULL, longest, 2));
        bool waited = false;
        int k = 0;
        for (; k + 4 <= cnt; k += 4) {
            int s4[4], o4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) { s4[j] = __shfl_sync(KV_FULL, sp, k + j); o4[j] = __shfl_sync(KV_FULL, om, k + j); }
            if (!waited && sim.surely(__shfl_sync(KV_FULL, size, k), __shfl_sync(KV_FULL, longest, k))) {
#pragma unroll
                for (int j = 0; j < 4; ++j) sim.add(s4[j], o4[j]);
                sim.acc += 4 * sim.tau;
                if ((lane & ~3) == k) mine = sim.start();
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    waited = sim.admit_alone(s4[j], o4[j], left - k - j, status);
                    if (lane == k + j) mine = sim.start();
                }
            }
        }
        for (; k < cnt; ++k) {
            sim.admit_alone(__shfl_sync(KV_FULL, sp, k), __shfl_sync(KV_FULL, om, k), left - k, status);
            if (lane == k) mine = sim.start();
        }
    } else {
        for (int k = 0; k < cnt; ++k) {
            sim.admit(__shfl_sync(KV_FULL, sp, k), __shfl_sync(KV_FULL, om, k), left - k, status);
            if (lane == k) mine = sim.start();
        }
    }
    return mine;
}

// Ring slots (32 cells each, a power of two) for the longest decode of a handle: a window that starts
// in the last round of its chunk ends (30 + omax) / 32 chunks further on.
static inline int sim_pick_slots(int omax) {
    const int far = (30 + omax) >> 5;
    int slots = 1;
    while (slots < far) slots <<= 1;
    return slots;
}
