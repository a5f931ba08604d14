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
//   two near chunks (the one t lies in, the next)   the exact V[x] - M, one round of each per lane, in registers.
//   far chunks                    an admission that covers a far chunk whole adds a constant and a
//       slope to it, so only their sums are kept: A = sum of (s+1-p), C = how many; the chunk in which
//       a window ends is the one chunk per admission whose 32 cells are written (a ring in shared
//       memory, one column per lane: own[x] = sum of (s+1-p) + x over the windows that end in the
//       chunk and reach x).  V[x] = own[x] + A + C x, where A starts from -M and C from 1.  Every lane holds A, C of one
//       of the 32 chunks behind the two (and of every 32nd behind that for decodes beyond 1,025 rounds: NM
//       registers of each); the chunk number modulo 32 says which lane, so nothing moves when time does.
//   W (per far chunk)             M less an upper bound of V over the chunk: every admission that reaches the
//       chunk lowers it by its ramp's value in the chunk's last round.  One compare per lane tests 32
//       chunks.  Where W says "perhaps", the chunk's cells are put together, W becomes exact
//       and the cells decide.  Occupancy falls behind the chunk t lies in, so this is rare.
//
// Wait of a request that does not fit: a round over budget by e > 0 at offset r from t rules out every
// start before t + min(e, r+1) (either the ramp has dropped by e or the window has moved past the
// round).  The largest of these bounds is the first start that every round of [t, t+o) allows, and only the rounds
// that come into the window at its other end are left.  So one reduction over the two chunks nearly always
// answers "when", not only "whether" (see ask).  A request that waits for longer than the two chunks
// takes its bound from A + C x of the far ones: a few steps, however long it waits.
//
// Rounds are counted from 0 throughout, so nothing that a lane keeps changes when t moves on (counted from the beginning of
// t's chunk, entering the next one had to correct A, W, X and both chunks: 26 instead of 19 instructions, 1.6 times per
// admission where memory is short).  A request is passed as sp = s + 1 and om = o - 1.
//
// What bounds it: instructions.  With one near chunk, tested again after every wait, an admission of k3_eval_moves took
// 75 to 95 of them; the exact wait, windows of 64 rounds and more without masks, and two turns of the loop in a row leave 60
// to 80.  Sweeps with a warp each: 16,384 moves of 10,000 requests (decodes to 1,024) 8.71 -> 7.26 ms, 16,000
// of 1,000 1.23 -> 1.01 ms, 7,000 of 100,000 (decodes to 4,096) 40.5 -> 35.9 ms.  One run
// that stands alone (run_alone) is bound by the latency of one admission: the part behind the two chunks is put while the
// next request's reduction is under way, and a branch on fresh data costs 28 cycles, so there is one.  Cycles per
// admission 367 -> 216 (1,000 requests, 13 rounds per request), 278 -> 150 (10,000, 3 rounds), 269 -> 155 (100,000, 1 round).
// Three kinds of backlog leave that loop for nearly every request, at the price of two branches and a second question, so
// they have loops of their own, which cost the others up to 0.03 (10,000 requests, cycles per admission with the loop
// for the rest -> theirs): nothing waits (run_together: decodes to 2,048 rounds 236 -> 155, to 1,024 148 -> 116); windows of less
// than 64 rounds wait inside the chunk (kBrief: up to 20 rounds, one beside the other, 758 -> 300; up to 64, 706 -> 433);
// windows of 1,025 rounds and more (kLengthy: half of them such, 0.05 / 1 rounds per request, 236 -> 202 / 336 -> 267).
// Tried without gain: two to eight requests in a row without a branch where some of them wait (their conditions cost more:
// 172 to 257 for the 10,000), t moving over several chunks at once (sweeps 82 -> 85 issue slots per admission).
//
// Sums may wrap; V itself fits 31 bits (the host checks M, sum of o and n), so arithmetic modulo 2^32
// gives it exactly.  U may exceed it by 31 for every request that is resident in a chunk's first round (chunk_sums_fit, api.cu).
#pragma once

#include "common.cuh"

// kGlobal: the rings are in device memory.  A simulator for decodes up to 4,097 rounds has 16 KB of ring,
// so shared memory holds 13 of them per SM and registers 32; the ring is written without waiting and read once per
// 32 rounds.  device_rings_fit (api.cu) has the rule and the figures.
//
// kShort: a window that ends in t's chunk leaves everything else alone.  Where nearly every decode is a few rounds,
// a sweep takes 0.78 to 0.95 of the time (mean 4 and 20); with longer ones it is no gain.  short_windows (api.cu) has the rule.
template <int NM, bool kGlobal_ = false, bool kShort = false>
struct ChunkSim {
    static constexpr bool kGlobal = kGlobal_;
    static constexpr int kWarps = NM == 1 || kGlobal ? 4 : NM == 2 ? 2 : 1;    // per CTA: 16 KB of shared rings
    static constexpr int kMinCtas = kGlobal ? 8 : 10;            // CTAs per SM the registers have to allow
    static constexpr int kMeta = 64 + 96 * NM;                      // state ints besides the ring
    __host__ __device__ static constexpr int ring_cells(int L) { return L - kMeta; }   // shared-memory ints per warp
    static constexpr int kAsk = 128;                                // "look closer": above every wait in the two chunks
    enum { kPlain, kBrief, kLengthy };                              // forms of run_alone, see there
    static constexpr int kLong = 64;                                // om from which every window covers what is left of the two chunks and ends behind them

    int lane;
    int t;                   // the round the next request may start at
    int tn;                  // first round of the chunk behind the one t lies in
    int M;
    int x0;                  // this lane's round of the chunk t lies in
    int cur, nxt;            // V - M of this lane's round of the two chunks
    int X;                   // first round of this lane's far chunk; register m: the chunk 1024 m rounds behind it
    int A[NM], C[NM], W[NM]; // W = M - U
    unsigned acc;            // of a block of up to 32 admissions: sum of their starts
    i64 tel;                 // sum of starts in front of the block
    int* ring;               // this lane's column
    int mask;                // ring ints - 1, without the lane bits

    __device__ __forceinline__ void attach(int* ring_, int L) {
        lane = kv_lane();
        ring = ring_ + lane;
        mask = (ring_cells(L) - 1) & ~31;
    }
    __device__ __forceinline__ int* cells_of(int x) const { return ring + KV_IDX(x & mask, mask + 32, 151); }
    __device__ __forceinline__ static int cell(const int* p) { return kGlobal ? __ldcg(p) : *p; }
    // *p += v where `on`: an atomic without a result, so nothing waits for the old value, and without a branch
    __device__ __forceinline__ static void raise(int* p, int v, bool on) {
        if (kGlobal) asm volatile("{ .reg .pred q; setp.ne.s32 q, %2, 0; @q red.global.add.s32 [%0], %1; }" :: "l"(p), "r"(v), "r"((int)on) : "memory");
        else atomicAdd(p, on ? v : 0);
    }
    __device__ __forceinline__ void set_time(int t_, int M_) {
        t = t_; M = M_;
        x0 = (t & ~31) + lane; tn = (t & ~31) + 32;
        X = tn + 32 + 32 * ((lane - (tn >> 5) - 1) & 31);
    }
    __device__ __forceinline__ int start() const { return t; }             // of the request admitted last

    // nothing is resident at t or later
    __device__ __forceinline__ void reset(int M_, int t_ = 0) {
        set_time(t_, M_);
        cur = x0 - M; nxt = cur + 32; tel = 0;
#pragma unroll
        for (int m = 0; m < NM; ++m) { A[m] = -M; C[m] = 1; W[m] = M - (X + 1024 * m + 31); }
        for (int k = 0; k <= mask; k += 32) ring[KV_IDX(k, mask + 32, 152)] = 0;
        __syncwarp();
    }

    // snapshot: the two chunks [32 each], then A, C, W of every m [32 each], then the ring
    __device__ __forceinline__ void load(const int* __restrict__ snap, const SnapHeader& h, int M_) {
        set_time(h.t, M_);
        tel = ((i64)h.tel_hi << 32) | (i64)(unsigned)h.tel_lo;
        const int4* src = reinterpret_cast<const int4*>(snap + kMeta) + lane;
        int4* dst = reinterpret_cast<int4*>(ring - lane) + lane;
        const int groups = (mask + 32) >> 2;
        for (int g = 0; g + lane < groups; g += 32) dst[KV_IDX(g, groups - lane, 153)] = src[g];
        cur = snap[lane]; nxt = snap[32 + lane];
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            A[m] = snap[64 + 96 * m + lane]; C[m] = snap[96 + 96 * m + lane]; W[m] = snap[128 + 96 * m + lane];
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
        snap[lane] = cur; snap[32 + lane] = nxt;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            snap[64 + 96 * m + lane] = A[m]; snap[96 + 96 * m + lane] = C[m]; snap[128 + 96 * m + lane] = W[m];
        }
        if (lane == 0) {
            SnapHeader h; h.t = t;
            h.tel_lo = (int)(tel_before & 0xffffffffll); h.tel_hi = (int)(tel_before >> 32);
            *hdr = h;
        }
    }
    // sum of the completion times of all requests; sum_o: decode lengths of those admitted here
    __device__ __forceinline__ i64 total(i64 sum_o) const { return tel + sum_o; }

    __device__ __forceinline__ static int pick(int on, int a, int b) {     // a select that stays one
        int r;
        asm("{ .reg .pred q; setp.ne.s32 q, %1, 0; selp.s32 %0, %2, %3, q; }" : "=r"(r) : "r"(on), "r"(a), "r"(b));
        return r;
    }
    // on: this lane's first far chunk is none any more.  With several registers as selects by all lanes: as a branch that one lane
    // takes alone it held up the other 31 (10,000 requests on short prefills, 20 rounds per request, 6,000 moves, decodes to
    // 2,048 / 4,096 / 8,192: 6.55 -> 6.26, 9.57 -> 7.29, 22.0 -> 14.6 ms).
    __device__ __forceinline__ void next_chunk(int on) {
        if (NM == 1) {
            if (on) { X += 1024; A[0] = -M; C[0] = 1; W[0] = M - (X + 31); }
            return;
        }
        X += on << 10;
#pragma unroll
        for (int m = 0; m + 1 < NM; ++m) { A[m] = pick(on, A[m + 1], A[m]); C[m] = pick(on, C[m + 1], C[m]); W[m] = pick(on, W[m + 1], W[m]); }
        A[NM - 1] = pick(on, -M, A[NM - 1]); C[NM - 1] = pick(on, 1, C[NM - 1]);
        W[NM - 1] = pick(on, M - (X + (1024 * (NM - 1) + 31)), W[NM - 1]);
    }
    // t has left its chunk: the next one takes its place, the first far chunk that one's, and the lane that held it
    // gets the chunk 1024 NM rounds further on
    __device__ __forceinline__ void rotate() {
        tn += 32; x0 += 32;
        const int j = (tn >> 5) & 31;
        int* const p = cells_of(tn);
        const int own = cell(p);
        *p = 0;
        const int a = __shfl_sync(KV_FULL, A[0], j), c = __shfl_sync(KV_FULL, C[0], j);
        cur = nxt;
        nxt = own + a + c * (x0 + 32);
        next_chunk(lane == j);
    }
    // t moves on by d rounds
    __device__ __forceinline__ void advance(int d) {
        t += d;
        while (t >= tn) rotate();
    }
    // the same for any d: a gap longer than every window leaves nothing resident
    __device__ __forceinline__ void skip(int d, int M) {
        if (d > mask + 128) reset(M, t + d);
        else advance(d);
    }
    // Lists whose schedules may go on for 2^30 rounds and more (orders with an id many times over, any start times) count
    // their rounds from a later one now and then: taken off t, a multiple of every ring's length and of the 32 lanes' chunks.
    __device__ __forceinline__ int rebase() {
        if (t < (1 << 29)) return 0;
        const int d = t & ~8191;
        t -= d; tn -= d; x0 -= d; X -= d; cur -= d; nxt -= d;
#pragma unroll
        for (int m = 0; m < NM; ++m) { A[m] += (C[m] - 1) * d; W[m] += d; }
        return d;
    }
    // far chunks of the window whose bound does not clear it: exact maximum into W, wait bound of their cells
    __device__ __forceinline__ int far_need(int a0, int last) {
        int d = 0;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            unsigned todo = __ballot_sync(KV_FULL, X + 1024 * m <= last && a0 > W[m]);
            while (todo) {
                const int j = __ffs(todo) - 1;
                todo &= todo - 1;
                const int x = __shfl_sync(KV_FULL, X, j) + 1024 * m + lane;
                const int a = __shfl_sync(KV_FULL, A[m], j), c = __shfl_sync(KV_FULL, C[m], j);
                const int v = cell(cells_of(x)) + a + c * x;
                const int vmax = kv_warp_max(v);
                if (lane == j) W[m] = -vmax;
                if (x <= last) d = max(d, __viaddmin_s32(v, a0, x - t + 1));
            }
        }
        return kv_warp_max(d);
    }
    // 0: (sp, om) fits at t; otherwise a lower bound of the rounds it has to wait.  A far chunk that may be over says
    // what the windows that cover it whole use in its last round of the window: a long wait is a few steps.
    __device__ __forceinline__ int test(int sp, int om) {
        const int a0 = sp - t, last = t + om;            // it fits  <=>  V[x] - M + a0 <= 0 in every round of the window
        const int r = x0 + 1 - t;
        int v = x0 <= last ? __viaddmin_s32(cur, a0, r) : 0;
        if (x0 + 32 <= last) v = max(v, __viaddmin_s32(nxt, a0, r + 32));
        bool far = false;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int x = X + 1024 * m;
            if (x <= last && a0 > W[m]) {
                const int e = min(x + 31, last);
                v = max(v, __viaddmin_s32(A[m] + C[m] * e, a0, e - t + 1));
                far = true;
            }
        }
        const int d = kv_warp_max(v);
        if (d > 0 || !__any_sync(KV_FULL, far)) return max(d, 0);
        return far_need(a0, last);
    }

    // One reduction answers for all lanes: 0 or less: (sp, om) fits at t; kAsk: a far bound says "perhaps"; otherwise
    // the rounds that the two chunks make it wait.  kWhole (om >= kLong): that wait is exact.  The request fits in the two
    // chunks from then on, and the far chunks that a wait of up to 64 rounds can bring into the window are
    // asked here, at the limit of t, which only rises.
    template <bool kWhole>
    __device__ __forceinline__ int ask(int sp, int om) const {
        const int a0 = sp - t, last = t + om, r = x0 + 1 - t;
        int v = __viaddmin_s32(cur, a0, kWhole || x0 <= last ? r : 0);             // rounds before t: 0 or less
        if (kShort && !kWhole && last < tn) return kv_warp_max(v);
        v = max(v, __viaddmin_s32(nxt, a0, kWhole || x0 + 32 <= last ? r + 32 : 0));
        if (X <= (kWhole ? tn + 32 + om : last) && a0 > W[0]) v = kAsk;
        if (kWhole && NM > 1 && om >= 1024) {
#pragma unroll
            for (int m = 1; m < NM; ++m) if (X + 1024 * m <= tn + 32 + om && a0 > W[m]) v = kAsk;
        }
        return kv_warp_max(v);
    }
    // the same for any window without a branch but for long ones: where one run stands alone a branch takes longer
    __device__ __forceinline__ int ask(int sp, int om) const {
        const int a0 = sp - t, last = t + om, r = x0 + 1 - t;
        int v = __viaddmin_s32(cur, a0, x0 <= last ? r : 0);
        v = max(v, __viaddmin_s32(nxt, a0, x0 + 32 <= last ? r + 32 : 0));
        if (X - tn <= om + 32 && a0 > W[0]) v = kAsk;
        if (NM > 1 && om >= 1024) {
#pragma unroll
            for (int m = 1; m < NM; ++m) if (X + 1024 * m - tn <= om + 32 && a0 > W[m]) v = kAsk;
        }
        return kv_warp_max(v);
    }
    // what `test` says, the far chunks looked at only where they have to be
    __device__ __forceinline__ int need(int sp, int om) {
        const int v = ask(sp, om);
        return v >= kAsk ? test(sp, om) : max(v, 0);
    }
    // (sp, om) starts at t
    template <bool kWhole>
    __device__ __forceinline__ void put(int sp, int om) {
        const int a = sp - t, last = t + om;
        if (kWhole ? x0 >= t : (unsigned)(x0 - t) <= (unsigned)om) cur += a + x0;
        if (kShort && !kWhole && last < tn) return;
        if (kWhole || x0 + 32 <= last) nxt += a + x0 + 32;
        if (!kWhole && last < tn + 32) return;
        if (X <= last) W[0] -= a + X + 31;
        if (kWhole) {                                                   // a short one covers no far chunk whole
            if (X + 31 < last) { A[0] += a; C[0] += 1; }
            if (NM > 1 && om >= 1024) {
#pragma unroll
                for (int m = 1; m < NM; ++m) {
                    if (X + 1024 * m <= last) W[m] -= a + (X + 1024 * m + 31);
                    if (X + 1024 * m + 31 < last) { A[m] += a; C[m] += 1; }
                }
            }
        }
        const int x = (last & ~31) + lane;                          // the chunk the window ends in
        raise(cells_of(last), a + x, x <= last);
    }
    __device__ __forceinline__ void add(int sp, int om) {                // the same for any window
        const int a = sp - t, last = t + om;
        if (x0 >= t && x0 <= last) cur += a + x0;
        if (x0 + 32 <= last) nxt += a + x0 + 32;
        if (X <= last) W[0] -= a + X + 31;
        if (X + 31 < last) { A[0] += a; C[0] += 1; }
        if (NM > 1 && om >= 1024) {
#pragma unroll
            for (int m = 1; m < NM; ++m) {
                if (X + 1024 * m <= last) W[m] -= a + (X + 1024 * m + 31);
                if (X + 1024 * m + 31 < last) { A[m] += a; C[m] += 1; }
            }
        }
        const int x = (last & ~31) + lane;
        raise(cells_of(last), a + x, last >= tn + 32 && x <= last);
    }

    // Whether a request of (size, om) certainly fits at t; or several, `size` the sum of their s + o, the longest with
    // om = o - 1, one beside the other: none of them uses more than its s + o in any round.
    __device__ __forceinline__ bool surely(int size, int om) const {
        const int a0 = size - t, last = t + om;
        bool over = x0 >= t && x0 <= last && cur > -a0;
        over = over || (x0 + 32 <= last && nxt > -a0) || (X <= last && a0 > W[0]);
        if (NM > 1 && om >= 1024) {
#pragma unroll
            for (int m = 1; m < NM; ++m) over = over || (X + 1024 * m <= last && a0 > W[m]);
        }
        return !__any_sync(KV_FULL, over);
    }

    // Starts (sp, om) at t if it fits there: a vote, since no wait is asked for, and no second chunk for a window that is put
    // in the first.  Windows of 64 rounds and more take a path of their own as long as their bounds are one register (with more of
    // them, on fewer warps, it was no gain).  2,000 schedules of 1,000 requests, decodes to 20 / 256 / 1,024 / 4,096, with the
    // question that answers a wait -> this: 428 -> 304, 366 -> 311, 367 -> 331, 522 -> 510 us.
    __device__ __forceinline__ bool put_if_fits(int sp, int om) {
        const int a0 = sp - t, last = t + om;
        if (NM == 1 && om >= kLong) {
            const bool over = (x0 >= t && cur > -a0) || nxt > -a0 || (X <= last && a0 > W[0]);
            if (__any_sync(KV_FULL, over) && test(sp, om) > 0) return false;
            put<true>(sp, om);
            return true;
        }
        if (!surely(sp, om) && test(sp, om) > 0) return false;
        if (NM == 1) put<false>(sp, om); else add(sp, om);
        return true;
    }

    // Takes back what is left (from t on) of a window whose ramp is a + x in round x and whose last round is `last`.  The
    // bounds fall by the least the ramp has in a chunk it covers whole.
    __device__ __forceinline__ void remove(int a, int last) {
        if (x0 >= t && x0 <= last) cur -= a + x0;
        if (x0 + 32 <= last) nxt -= a + x0 + 32;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int x = X + 1024 * m;
            if (x + 31 <= last) W[m] += a + x;
            if (x + 31 < last) { A[m] -= a; C[m] -= 1; }
        }
        const int x = (last & ~31) + lane;                          // the chunk the window ends in
        raise(cells_of(last), -(a + x), last >= tn + 32 && x <= last);
    }

    // The request at hand stays where `run` has left it: t moves on to the next round that is worth a question (false), or it
    // fits although a far bound does not clear it and has been admitted (true).  v: the answer that was neither
    // "fits" nor a wait that ends in t's chunk.
    __device__ __forceinline__ bool step(int sp, int om, int v) {
        if (v >= kAsk) v = test(sp, om);
        else if (om >= kLong) { advance(v); put<true>(sp, om); return true; }
        if (v <= 0) { add(sp, om); return true; }
        advance(v);
        return false;
    }

    // acc counts modulo 2^32; the starts of a block lie less than 2^27 rounds apart
    __device__ __forceinline__ void add_block(int t_first, int cnt) {
        const unsigned base = (unsigned)t_first * (unsigned)cnt;
        tel += (i64)t_first * cnt + (i64)(acc - base);
    }

    // Up to 32 consecutive requests of a list, each at its earliest start: (s, o) of the k-th in lane k.  Returns
    // the start of the k-th in lane k.
    __device__ __forceinline__ int run(int2 so, int cnt, int* status) {
        const int sp_l = so.x + 1, om_l = so.y - 1, t_first = t;
        const int cap = kv_loop_cap(32 * mask + 2048);
        int mine = 0, k = 0, turns = 0;
        acc = 0;
        for (;;) {
            int sp = 0, om = 0, v = 0;
#pragma unroll 2
            for (; k < cnt; ++k) {                   // as long as t stays in its chunk and no far bound is in the way
                sp = __shfl_sync(KV_FULL, sp_l, k); om = __shfl_sync(KV_FULL, om_l, k);
                if (om >= kLong) {
                    v = ask<true>(sp, om);
                    const int at = __viaddmax_s32(v, t, t);
                    if (at >= tn) break;
                    t = at;
                    put<true>(sp, om);
                } else {
                    for (;;) {                       // a wait inside the chunk: ask again from there
                        v = ask<false>(sp, om);
                        if (kGlobal || v <= 0 || t + v >= tn) break;
                        t += v;
                    }
                    if (v > 0) break;
                    put<false>(sp, om);
                }
                acc += (unsigned)t;
                if (lane == k) mine = t;
            }
            if (k >= cnt) break;
            if (step(sp, om, v)) {
                acc += (unsigned)t;
                if (lane == k) mine = t;
                ++k;
                turns = 0;
            } else if (++turns > cap) { if (lane == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }
        }
        add_block(t_first, cnt);
        return mine;
    }

    // The same for a run that stands alone: one branch for a request that neither waits for another chunk nor meets a far
    // bound.  What leaves the loop otherwise, and stays in it by kForm: kBrief: a window of less than 64 rounds that
    // waits inside the chunk; kLengthy: windows of 1,025 rounds and more.
    template <int kForm>
    __device__ __forceinline__ int run_alone(int2 so, int cnt, int* status) {
        constexpr bool kBriefs = kForm == kBrief, kFar = NM > 1 && kForm == kLengthy;
        const int sp_l = so.x + 1, om_l = so.y - 1, t_first = t;
        const int cap = kv_loop_cap(32 * mask + 2048);
        // far rounds that may matter, from tn on: a short window ends om + 31 rounds behind the chunk's beginning at the
        // latest, a long one waits for up to 64.
        // From the lane that has it: worked out in every turn it lies in front of the reduction.
        const int far_l = om_l + (om_l >= kLong ? 32 : -1);
        int mine = 0, k = 0, turns = 0;
        acc = 0;
        int sp = __shfl_sync(KV_FULL, sp_l, 0), om = __shfl_sync(KV_FULL, om_l, 0), far_to = kBriefs ? __shfl_sync(KV_FULL, far_l, 0) : 0;
        int pa = 0, plast = -1;                          // the admission whose part behind the two chunks is still to be put
        auto put_far = [&]() {
            if (X + 31 < plast) { A[0] += pa; C[0] += 1; }
            const int x = (plast & ~31) + lane;
            raise(cells_of(plast), pa + x, plast >= tn + 32 && x <= plast);
        };
        while (kForm == kPlain || k < cnt) {             // of the two ways to write it the faster one for each form, by up to a half
            int v, sp_next, om_next, far_next = 0;
            for (;;) {
                const int a0 = sp - t, end = t + om, r = x0 + 1 - t;
                v = __viaddmin_s32(cur, a0, x0 <= end ? r : 0);
                v = max(v, __viaddmin_s32(nxt, a0, x0 + 32 <= end ? r + 32 : 0));
                if (X - tn <= (kBriefs ? far_to : om + 32) && a0 > W[0]) v = kAsk;
                if (kFar && om >= 1024) {
#pragma unroll
                    for (int m = 1; m < NM; ++m) if (X + 1024 * m - tn <= om + 32 && a0 > W[m]) v = kAsk;
                }
                v = kv_warp_max(v);
                put_far();
                plast = -1;
                sp_next = __shfl_sync(KV_FULL, sp_l, (k + 1) & 31); om_next = __shfl_sync(KV_FULL, om_l, (k + 1) & 31);
                if (kBriefs) far_next = __shfl_sync(KV_FULL, far_l, (k + 1) & 31);
                const int most = NM > 1 && !kFar && om >= 1024 ? t - 1 : om >= kLong ? tn - 1 : t;
                const int at = __viaddmax_s32(v, t, t);
                if (at > most) {
                    if (!kBriefs || om >= kLong || at >= tn) break;
                    t = at;                            // asked again from there
                    continue;
                }
                t = at;
                pa = sp - t; plast = t + om;
                if (x0 >= t && x0 <= plast) cur += pa + x0;
                if (x0 + 32 <= plast) nxt += pa + (x0 + 32);
                if (X <= plast) W[0] -= pa + (X + 31);
                if (kFar && om >= 1024) {
#pragma unroll
                    for (int m = 1; m < NM; ++m) {
                        if (X + 1024 * m <= plast) W[m] -= pa + (X + 1024 * m + 31);
                        if (X + 1024 * m + 31 < plast) { A[m] += pa; C[m] += 1; }
                    }
                }
                if (lane == k) mine = t;
                acc += (unsigned)t;
                turns = 0;
                sp = sp_next; om = om_next; far_to = far_next;
                if (++k >= cnt) break;
            }
            if (k >= cnt) break;
            bool in = false;
            if (NM > 1 && !kFar && om >= 1024) {
                v = ask<true>(sp, om);
                in = t + v < tn;
                if (in) { t += max(v, 0); put<true>(sp, om); }
            }
            if (in || step(sp, om, v)) {
                if (lane == k) mine = t;
                acc += (unsigned)t;
                turns = 0;
                sp = sp_next; om = om_next; far_to = far_next;
                ++k;
                if (kForm == kPlain && k >= cnt) break;
            } else if (++turns > cap) { if (lane == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }
        }
        put_far();
        add_block(t_first, cnt);
        return mine;
    }

    // The same where nothing has waited for a while: four at a time are asked for together and put without a question each, as
    // long as that goes well; calm tells afterwards whether it did.
    __device__ __forceinline__ int run_together(int2 so, int cnt, bool& calm, int* status) {
        constexpr int kMost = (1 << 29) - 1;             // four of them fit 31 bits; a group of so much is none
        const int sp_l = so.x + 1, om_l = so.y - 1, t_first = t;
        int size = min(so.x + so.y, kMost), longest = om_l;                  // of the aligned four this lane is in
        size += __shfl_xor_sync(KV_FULL, size, 1); size += __shfl_xor_sync(KV_FULL, size, 2);
        if (size >= kMost) size = INT_MAX;
        longest = max(longest, __shfl_xor_sync(KV_FULL, longest, 1));
        longest = max(longest, __shfl_xor_sync(KV_FULL, longest, 2));
        int mine = 0, k = 0, turns = 0;
        acc = 0;
        for (; calm && k + 4 <= cnt; k += 4) {
            int s4[4], o4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) { s4[j] = __shfl_sync(KV_FULL, sp_l, k + j); o4[j] = __shfl_sync(KV_FULL, om_l, k + j); }
            calm = surely(__shfl_sync(KV_FULL, size, k), __shfl_sync(KV_FULL, longest, k));
            if (!calm) break;
#pragma unroll
            for (int j = 0; j < 4; ++j) add(s4[j], o4[j]);
            acc += 4u * (unsigned)t;
        }
        if (lane < k) mine = t_first;
        while (k < cnt) {
            const int sp = __shfl_sync(KV_FULL, sp_l, k & 31), om = __shfl_sync(KV_FULL, om_l, k & 31), v = need(sp, om);
            if (v <= 0) {
                add(sp, om);
                if (lane == k) mine = t;
                acc += (unsigned)t;
                ++k;
                turns = 0;
            } else {
                calm = false;
                advance(v);
                if (++turns > kv_loop_cap(32 * mask + 2048)) { if (lane == 0) atomicExch(status, KV_DEV_LOOP_CAP); break; }
            }
        }
        add_block(t_first, cnt);
        return mine;
    }
};

// Ring slots (32 cells each, a power of two) for the longest decode of a handle: a window that starts
// in the last round of its chunk ends (30 + omax) / 32 chunks further on.
static inline int sim_pick_slots(int omax) {
    const int far = (30 + omax) >> 5;
    int slots = 1;
    while (slots < far) slots <<= 1;
    return slots;
}
static inline int sim_state_ints(int nm, int slots) { return 64 + 96 * nm + 32 * slots; }
