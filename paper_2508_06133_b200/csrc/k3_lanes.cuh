// K3, many candidates: one THREAD per candidate move.  Same rule, same results as k3_eval_moves
// (sim_chunk.cuh has the rule; V[x] is the tokens in use in round x, plus x).
//
// k3_eval_moves gives a warp to a candidate; nearly all of its 77 instructions per admission are the same
// in every lane.  Here the 32 candidates of a warp are neighbours in the launch order (first moved
// positions next to each other), so they start from the same state of the base run and meet about the
// same requests in about the same rounds: they are moved through time together, chunk by chunk of CH
// rounds, and within a chunk each lane admits and waits at its own pace.
//
// State of a candidate, x counted from the beginning T0 of the chunk that time is in:
//   cells     of this chunk and the next one, as they were when time entered the chunk before: base[x]
//       (shared memory, a column per thread).  Admissions since then add d_A + d_C x to a whole chunk;
//       a window that ends inside one of the two takes its share back from the cells behind its end.
//   events    for the chunks behind these: per round x, the requests whose last round is x, their sum of
//       s+o and their number in one word (global memory, a ring of NCH chunks; a lane's chunk is one
//       line of 128 or 256 bytes), and the running totals A = sum of (s+1-p), C = how many over the requests
//       that run into them.  An admission is two additions and at most one word, whatever its window; a
//       chunk's words are read once, when its cells are put together from the totals.
//   bounds    W0, W1 of V over the two chunks, U[c] over the NF behind them (registers), Uall their
//       maximum: each raised by a ramp's value in the chunk's last round.  All below the limit: it fits.
// Where W0 says "perhaps", one walk back over the chunk's cells gives the first round from which the
// request fits (the maximum of V behind a round falls along the chunk, the limit rises), hence the wait,
// so a turn nearly always ends with an admission in every lane (1.25 turns per admission).  W1 is
// answered from the next chunk's cells, U (2 of 1,000 turns) from the events.
//
// What bounds it: integer issue, as in the kernel with a warp per candidate, but by the work of a chunk (two
// builds of 32 cells, 34 event words) and not by that of an admission: it pays when few rounds pass per
// admission.  Measured, kernel against k3_eval_moves: 10,000 requests, budget 262,144 (2.9 rounds per
// request), 64,000 moves 33.0 -> 23.6 ms; 3,000 requests, budget 400,000 (1.9), 256,000 moves 36.6 -> 18.9 ms.
// lanes_fit (api.cu) has the rule and the other side.
#pragma once

#include "common.cuh"
#include "k3_eval.cuh"

struct LaneParams {
    MoveEvalParams m;
    int omax;                // largest decode length, <= CH * NCH - CH + 1
    int shift;               // events: sum of (s+o - least) in the low `shift` bits, number above them
    int least;               // smallest s+o
    void* rings;             // per resident warp: NCH * 32 * CH words
    unsigned* counter;       // next group of 32 candidates
    int groups;
};

template <typename WORD_>
struct LaneSim {
    typedef WORD_ WORD;
    static constexpr int CH = 32, NF = 32, NCH = NF + 2;
    static constexpr int kWarps = 4;
    static constexpr size_t kRingWords = (size_t)NCH * 32 * CH;            // per warp
    static constexpr size_t kSmem = (size_t)2 * CH * 32 * kWarps * sizeof(int);
};

template <typename WORD>
__global__ void __launch_bounds__(128, 5)
k3_lane_moves(const LaneParams P) {
    typedef LaneSim<WORD> S;
    constexpr int CH = S::CH, NF = S::NF, NCH = S::NCH, VS = 32 * S::kWarps;           // cell x of a chunk: [x * VS]
    constexpr int PER = 16 / (int)sizeof(WORD);                            // words per 16-byte load
    extern __shared__ __align__(16) int lane_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* b0 = lane_smem + threadIdx.x;
    int* b1 = b0 + CH * VS;
    WORD* const ring = (WORD*)P.rings + ((size_t)blockIdx.x * S::kWarps + warp) * S::kRingWords + (size_t)lane * CH;
    const int n = P.m.n, M = P.m.M, least = P.least, shift = P.shift;
    const WORD vmask = ((WORD)1 << shift) - 1, one = (WORD)1 << shift;
    auto unpack = [](const uint4& v, WORD* ev) {                           // the words of 16 bytes
        if (sizeof(WORD) == 4) { ev[0] = (WORD)v.x; ev[1] = (WORD)v.y; ev[2] = (WORD)v.z; ev[3] = (WORD)v.w; }
        else { ev[0] = (WORD)((u64)v.x | ((u64)v.y << 32)); ev[1] = (WORD)((u64)v.z | ((u64)v.w << 32)); }
    };
    auto line_of = [&](int k) -> WORD* {                                   // this lane's words of slot k (k < 2 NCH)
        if (k >= NCH) k -= NCH;
        return ring + (size_t)KV_IDX(k, NCH, 421) * (32 * CH);
    };
    // the word of the x-th round behind the beginning of slot `slot`
    auto word_of = [&](int slot, int x) -> WORD* { return line_of(slot + x / CH) + (x & (CH - 1)); };
    for (;;) {
        unsigned group = 0;
        if (lane == 0) group = atomicAdd(P.counter, 1u);
        group = __shfl_sync(KV_FULL, group, 0);
        if (group >= (unsigned)P.groups) break;
        const i64 slot_c = (i64)group * 32 + lane;
        const bool mine = slot_c < P.m.count;
        const i64 cand = mine ? KV_IDX(P.m.launch_order[slot_c], P.m.count, 422) : 0;
        Move mv = {-1, n, n};
        if (mine) mv = k4_move_of(P.m.src, n, cand);
        const bool valid = mine && (unsigned)mv.i < (unsigned)n && (unsigned)mv.j < (unsigned)n;
        const int first_pos = kv_warp_min(valid ? min(mv.i, mv.j) : n);
        i64* const dst = P.m.tel_out + (P.m.tel_by_slot ? slot_c : cand);
        if (mine && !valid) *dst = INT64_MAX;                              // a code outside the neighbourhood
        if (first_pos >= n) continue;
        const int snap = (int)KV_IDX(first_pos / P.m.stride, P.m.snap_count, 423);
        const SnapHeader hdr = P.m.snap_hdr[snap];
        int q = snap * P.m.stride;                                         // this lane's next position
        const int T0 = hdr.t & ~(CH - 1);

        // ---- the base run's state in front of q: events, totals and bounds of the requests that still run
        for (int c = 0; c < NCH; ++c) {
            uint4* z = reinterpret_cast<uint4*>(line_of(c));
            for (int k = 0; k < CH / PER; ++k) __stcg(z + k, make_uint4(0, 0, 0, 0));
        }
        int A = 0, C = 0;                                                  // from the beginning of the chunk built next
        int U[NF];                                                         // U[c]: chunk c + 2
#pragma unroll
        for (int c = 0; c < NF; ++c) U[c] = CH * (c + 3) - 1;
        {
            int lo = 0, hi = q;                                            // first position that can still run at t
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (P.m.base_starts_pos[mid] + P.omax > hdr.t) hi = mid; else lo = mid + 1; }
            for (int k = lo; k < q; ++k) {
                const int2 so = P.m.tbl_base[k];
                const int p = P.m.base_starts_pos[k] - T0, last = p + so.y - 1;
                if (last < hdr.t - T0) continue;
                const int a = so.x + 1 - p;
                A += a; ++C;
                WORD* w = word_of(0, last);
                __stcg(w, __ldcg(w) + (WORD)(so.x + so.y - least) + one);
#pragma unroll
                for (int c = 0; c < NF; ++c) if (last >= CH * (c + 2)) U[c] += a + CH * (c + 3) - 1;
            }
        }
        // cells of the chunk whose events are in `slot`, from the totals; the totals move on to the next
        // one.  Returns the maximum of V, x counted from the chunk's own beginning.
        auto build = [&](int* cells, int slot) -> int {
            WORD* line = line_of(slot);
            int w = INT_MIN;
#pragma unroll 4
            for (int x0 = 0; x0 < CH; x0 += PER) {
                const uint4 v = __ldcg(reinterpret_cast<const uint4*>(line + x0));
                __stcg(reinterpret_cast<uint4*>(line + x0), make_uint4(0, 0, 0, 0));
                WORD ev[4];
                unpack(v, ev);
#pragma unroll
                for (int k = 0; k < PER; ++k) {
                    const int x = x0 + k, cell = A + C * x;
                    cells[x * VS] = cell;
                    w = max(w, cell + x);
                    const int num = (int)(ev[k] >> shift);
                    A -= (int)(ev[k] & vmask) + num * (least - x);
                    C -= num;
                }
            }
            A += CH * C;
            return w;
        };
        int W0 = build(b0, 0), W1 = build(b1, 1) + CH;
        int slot = 2;                                                      // events of the chunk behind the two
        int dA0 = 0, dC0 = 0, dA1 = 0, dC1 = 0;
        int tau = hdr.t - T0;
        i64 tel = (((i64)hdr.tel_hi << 32) | (i64)(unsigned)hdr.tel_lo) + (i64)T0 * (n - q);
        int acc = 0;                                                       // sum of tau + o
        // kv_map_pos without branches: position x1 holds y1, x2 holds y2, those in between are shifted
        const int d_in = mv.type == 1 ? (mv.i < mv.j ? 1 : -1) : 0;
        const int x1 = mv.j, y1 = mv.i, x2 = mv.type == 0 ? mv.i : n, y2 = mv.j;
        const int in_lo = min(mv.i, mv.j), in_len = max(mv.i, mv.j) - in_lo;
        auto fetch = [&](int at, int& sp_, int& om_) {
            int q = (unsigned)(at - in_lo) <= (unsigned)in_len ? at + d_in : at;
            q = at == x1 ? y1 : at == x2 ? y2 : q;
            const int2 so = P.m.tbl_base[KV_IDX(at < n ? q : 0, n, 424)];
            sp_ = so.x + 1; om_ = so.y - 1;
        };
        if (!valid) q = n;
        int sp = 2, om = 0, sp1 = 2, om1 = 0;                              // the request at q and the one behind it
        fetch(q, sp, om);
        fetch(q + 1, sp1, om1);

        for (i64 chunk = 0;; ++chunk) {
            int Uall = INT_MIN;
#pragma unroll
            for (int c = 0; c < NF; ++c) Uall = max(Uall, U[c]);
            // ---- every lane admits and waits until it leaves the chunk
            for (int guard = 0;; ++guard) {
                const bool act = q < n && tau < CH;
                if (!__any_sync(KV_FULL, act)) break;
                const int lim = M - sp;                                    // fits at t  <=>  V[x] <= lim + t over the window
                bool fits = act;
                const bool ask0 = act && W0 > lim + tau;
                if (__any_sync(KV_FULL, ask0)) {
                    const int x_lo = kv_warp_min(ask0 ? tau : CH - 1) & ~3;
                    const int lim0 = lim - dA0, slope = dC0 + 1;
                    int mx = INT_MIN, best = CH, best_w = 0;
                    for (int x4 = CH - 4; x4 >= x_lo; x4 -= 4) {
#pragma unroll
                        for (int k = 3; k >= 0; --k) {
                            const int x = x4 + k;
                            mx = max(mx, b0[x * VS] + slope * x);
                            if (mx <= lim0 + x) { best = x; best_w = mx; }
                        }
                    }
                    const bool cut = ask0 && tau + om < CH - 1;            // the window ends inside the chunk
                    if (ask0 && !cut) {
                        if (best < CH) { tau = max(tau, best); W0 = best_w + dA0; }
                        else { tau = CH; fits = false; }
                    }
                    if (__any_sync(KV_FULL, cut)) {
                        int d = 0;
                        if (cut)
                            for (int x = tau; x <= tau + om; ++x)
                                d = max(d, __viaddmin_s32(b0[x * VS] + slope * x, -(lim0 + tau), x - tau + 1));
                        if (d > 0) { tau += d; fits = false; }
                    }
                }
                const bool ask1 = fits && W1 > lim + tau && tau + om >= CH;
                if (__any_sync(KV_FULL, ask1 || (fits && Uall > lim + tau && tau + om >= 2 * CH))) {
                if (__any_sync(KV_FULL, ask1)) {
                    const int lim1 = lim + tau - dA1 - CH, slope = dC1 + 1, end = tau + om - CH;
                    int w = INT_MIN, d = 0;
#pragma unroll 4
                    for (int x = 0; x < CH; ++x) {
                        const int v = b1[x * VS] + slope * x;
                        w = max(w, v);
                        if (x <= end) d = max(d, __viaddmin_s32(v, -lim1, x + CH + 1 - tau));
                    }
                    if (ask1) {
                        W1 = w + dA1 + CH;
                        if (d > 0) { tau += d; fits = false; }
                    }
                }
                const bool far = fits && Uall > lim + tau && tau + om >= 2 * CH;
                if (__any_sync(KV_FULL, far)) {
                    // which far chunks of the window may be over?
                    const int nk = lim + tau, last = tau + om;
                    int c_hi = -1, all = INT_MIN;
#pragma unroll
                    for (int c = 0; c < NF; ++c) {
                        all = max(all, U[c]);
                        if (far && U[c] > nk && last >= CH * (c + 2)) c_hi = c;
                    }
                    if (far) Uall = all;
                    const int c_end = kv_warp_max(c_hi);
                    int a = A, cn = C, d = 0;                              // from the beginning of the chunk at hand
                    for (int c = 0; c <= c_end; ++c) {
                        const int base = CH * (c + 2);
                        const WORD* line = line_of(slot + c);
                        int w = INT_MIN;
#pragma unroll 4
                        for (int x0 = 0; x0 < CH; x0 += PER) {
                            const uint4 l = __ldcg(reinterpret_cast<const uint4*>(line + x0));
                            WORD ev[4];
                            unpack(l, ev);
#pragma unroll
                            for (int j = 0; j < PER; ++j) {
                                const int x = x0 + j, v = a + (cn + 1) * x + base;
                                w = max(w, v);
                                if (c <= c_hi && base + x <= last) d = max(d, __viaddmin_s32(v, -nk, base + x - tau + 1));
                                const int num = (int)(ev[j] >> shift);
                                a -= (int)(ev[j] & vmask) + num * (least - x);
                                cn -= num;
                            }
                        }
                        a += CH * cn;
                        all = INT_MIN;
#pragma unroll
                        for (int k = 0; k < NF; ++k) { if (k == c) U[k] = w; all = max(all, U[k]); }
                        Uall = all;
                    }
                    if (far && d > 0) { tau += d; fits = false; }
                }
                }
                const int a = sp - tau, last = tau + om;
                const int reach_max = kv_warp_max(fits ? last : 0);
                const bool far1 = fits && last >= CH, far2 = fits && last >= 2 * CH;
                if (fits) { dA0 += a; ++dC0; W0 += a + CH - 1; acc += last + 1; }
                if (far1) { dA1 += a + CH; ++dC1; W1 += a + 2 * CH - 1; }
                if (far2) {
                    A += a + 2 * CH; ++C;
                    atomicAdd(word_of(slot, last - 2 * CH), (WORD)(sp + om - least) + one);
                }
                if (__any_sync(KV_FULL, fits && !far2)) {                  // a window that ends in one of the two chunks
                    if (far1 && !far2) { for (int x = last + 1 - CH; x < CH; ++x) b1[x * VS] -= a + CH + x; }
                    if (fits && !far1) { for (int x = last + 1; x < CH; ++x) b0[x * VS] -= a + x; }
                }
                const int reach = fits ? last : 0;
                if (fits) {
                    sp = sp1; om = om1;
                    ++q;
                }
                fetch(q + 1, sp1, om1);
                // bounds of the far chunks the new windows reach
#pragma unroll
                for (int c0 = 0; c0 < NF; c0 += 8) {
                    if (reach_max < CH * (c0 + 2)) break;
#pragma unroll
                    for (int c = c0; c < c0 + 8; ++c)
                        if (reach >= CH * (c + 2)) { U[c] += a + CH * (c + 3) - 1; Uall = max(Uall, U[c]); }
                }
                if (guard > kv_loop_cap(1 << 28)) { if (lane == 0) atomicExch(P.m.status, KV_DEV_LOOP_CAP); break; }
            }
            if (!__any_sync(KV_FULL, q < n)) break;
            if (chunk > kv_loop_cap((i64)(1 << 30))) { if (lane == 0) atomicExch(P.m.status, KV_DEV_LOOP_CAP); break; }
            // ---- the next chunk
            tau -= CH;
            tel += (i64)CH * (n - q);
            int* const x = b0; b0 = b1; b1 = x;
            dA0 = dA1; dC0 = dC1; dA1 = 0; dC1 = 0;
            W0 = W1 - CH;
            W1 = build(b1, slot) + CH;
            slot = slot + 1 == NCH ? 0 : slot + 1;
#pragma unroll
            for (int c = 0; c + 1 < NF; ++c) U[c] = U[c + 1] - CH;
            U[NF - 1] = CH * (NF + 2) - 1;
        }
        if (valid) *dst = tel + acc;
        __syncwarp();
    }
}
