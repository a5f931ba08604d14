// K3, many candidates: one THREAD per candidate move.  Same rule, same results as k3_eval_moves
// (sim_chunk.cuh has the rule; V[x] is the tokens in use in round x, plus x).
//
// k3_eval_moves gives a warp to a candidate; nearly all of its 60 to 80 instructions per admission are the same
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
//       s+o and their number in one word (global memory, a ring of NCH chunks), and the running totals
//       A = sum of (s+1-p), C = how many over the requests that run into them.  An admission is two
//       additions and at most one word, whatever its window; a chunk's words are read once, when its
//       cells are put together from the totals.
//   bounds    W0, W1 of V over the two chunks, U[c] over the NF behind them (registers), Uall their
//       maximum: each raised by a ramp's value in the chunk's last round.  All below the limit: it fits.
// Where W0 says "perhaps", one walk back over the chunk's cells gives the first round from which the
// request fits (the maximum of V behind a round falls along the chunk, the limit rises), hence the wait,
// so a turn nearly always ends with an admission in every lane.  A request whose window covers the rest of the chunk and that
// the chunk's last cell keeps out whatever its start leaves the chunk before the turn begins (its last cell is kept in a register):
// 1.25 to 1.6 turns per admission, 1.4 to 2.2 where the walk had to find that out.  W1 is
// answered from the next chunk's cells, U (2 of 1,000 turns) from the events.
//
// What bounds it: instructions at 20 warps per SM (registers and the cells of two chunks allow no more), 0.72 of the issue
// slots and 0.68 of the integer pipe; below a full chip, latency.  A turn is about 330 instructions, a chunk 400 more: the
// walk takes four cells with one maximum (their slopes differ by one, two and three), a chunk's cells follow from
// the one before by two additions, the bounds' maximum two at a time, and the state in front of a group's first position is summed by
// reductions with a request per lane instead of by every lane for itself.  The event rings of all resident candidates are
// 412 MB and do not stay in L2 (126 MB), so a chunk's words are read with eight 16-byte loads in flight, laid out so
// that a warp's load is 512 contiguous bytes, called to L2 one chunk ahead, and cleared only where they are not zero; the
// request behind the next is on its way a turn early.
// 499,500 moves of 1,000 requests, budget 65,536: 13.45 -> 10.45 ms (blocked requests leave early 12.15, the walk by fours and
// the cells by additions 10.75); 65,536 moves of 10,000, budget 262,144: 14.9 -> 12.2 ms alone on the chip, of which 65,536 threads fill
// 0.7, so sweeps of several handles overlap (7.8 ms each).  A handle's first sweep also allocates the rings, which can
// take the driver several ms.  lanes_from (api.cu) has the rule and the other side.
#pragma once

#include "common.cuh"
#include "k3_eval.cuh"

struct LaneParams {
    MoveEvalParams m;
    int omax;                // largest decode length, at most CH * NF + 1
    int shift;               // events: sum of (s+o - least) in the low `shift` bits, number above them
    int least;               // smallest s+o
    void* rings;             // per resident warp: NCH * 32 * CH words
    unsigned* counter;       // next group of 32 candidates
    int groups;
};

template <int CH_, typename WORD_>
struct LaneSim {
    typedef WORD_ WORD;
    static constexpr int CH = CH_, NF = 32, NCH = NF + 2;
    static constexpr int kWarps = 4, kCtas = CH == 32 ? 5 : 3;            // CTAs per SM: shared memory
    static constexpr size_t kRingWords = (size_t)NCH * 32 * CH;            // per warp
    static constexpr size_t kSmem = (size_t)2 * CH * 32 * kWarps * sizeof(int);
};

template <int CH, typename WORD>
__global__ void __launch_bounds__(128, LaneSim<CH, WORD>::kCtas)
k3_lane_moves(const LaneParams P) {
    typedef LaneSim<CH, WORD> S;
    constexpr int NF = S::NF, NCH = S::NCH, VS = 4 * 32 * S::kWarps;
    constexpr int GROUP = 8;                                               // 16-byte loads of events in flight
    constexpr int PER = 16 / (int)sizeof(WORD);                            // words per 16-byte load
    extern __shared__ __align__(16) int lane_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* b0 = lane_smem + 4 * threadIdx.x;                                 // cells in fours: at(x)
    int* b1 = b0 + CH / 4 * VS;
    auto at = [](int x) -> int { const int c = (int)KV_IDX(x, CH, 425); return (c >> 2) * VS + (c & 3); };
    WORD* const ring = (WORD*)P.rings + ((size_t)blockIdx.x * S::kWarps + warp) * S::kRingWords + lane * PER;
    const int n = P.m.n, M = P.m.M, least = P.least, shift = P.shift;
    const WORD vmask = ((WORD)1 << shift) - 1, one = (WORD)1 << shift;
    const int most_turns = kv_loop_cap(1 << 28);
    auto unpack = [](const uint4& v, WORD* ev) {                           // the words of 16 bytes
        if (sizeof(WORD) == 4) { ev[0] = (WORD)v.x; ev[1] = (WORD)v.y; ev[2] = (WORD)v.z; ev[3] = (WORD)v.w; }
        else { ev[0] = (WORD)((u64)v.x | ((u64)v.y << 32)); ev[1] = (WORD)((u64)v.z | ((u64)v.w << 32)); }
    };
    // words of slot k (k < 2 NCH): 16 bytes of each lane side by side, then the next 16 bytes
    auto line_of = [&](int k) -> WORD* {
        if (k >= NCH) k -= NCH;
        return ring + (size_t)KV_IDX(k, NCH, 421) * (32 * CH);
    };
    // the word of the x-th round behind the beginning of slot `slot`
    auto word_of = [&](int slot, int x) -> WORD* {
        x = (int)KV_IDX(x, NCH * CH, 426);
        return line_of(slot + x / CH) + (x & (CH - 1)) / PER * (32 * PER) + (x & (PER - 1));
    };
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
            for (int k = 0; k < CH / PER; ++k) __stcg(z + 32 * k, make_uint4(0, 0, 0, 0));
        }
        int A = 0, C = 0;                                                  // from the beginning of the chunk built next
        int U[NF];                                                         // U[c]: chunk c + 2
#pragma unroll
        for (int c = 0; c < NF; ++c) U[c] = CH * (c + 3) - 1;
        {
            int lo = 0, hi = q;                                            // first position that can still run at t
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (P.m.base_starts_pos[mid] + P.omax > hdr.t) hi = mid; else lo = mid + 1; }
            // the same for all lanes: one running request each, its sums by reductions, its event in every lane's ring
            for (int k0 = lo; k0 < q; k0 += 32) {
                const int k = k0 + lane < q ? k0 + lane : lo;
                const int2 so = P.m.tbl_base[k];
                const int p = P.m.base_starts_pos[k] - T0, last = p + so.y - 1;
                const bool runs = k0 + lane < q && last >= hdr.t - T0;
                const int a = so.x + 1 - p, size = so.x + so.y - least, reach = runs ? last : -1;
                unsigned todo = __ballot_sync(KV_FULL, runs);
                A += __reduce_add_sync(KV_FULL, runs ? a : 0);
                C += __popc(todo);
#pragma unroll
                for (int c = 0; c < NF; ++c) U[c] += __reduce_add_sync(KV_FULL, reach >= CH * (c + 2) ? a + CH * (c + 3) - 1 : 0);
                for (; todo; todo &= todo - 1) {
                    const int j = __ffs(todo) - 1, at_round = __shfl_sync(KV_FULL, last, j);
                    atomicAdd(word_of(0, at_round), (WORD)__shfl_sync(KV_FULL, size, j) + one);
                }
            }
        }
        // cells of the chunk whose events are in `slot`, from the totals; the totals move on to the next
        // one.  Returns the maximum of V, x counted from the chunk's own beginning.
        int end0 = 0, end1 = 0;                                            // the last cell of either chunk
        auto build = [&](int* cells, int slot) -> int {
            WORD* line = line_of(slot);
            int w = INT_MIN;
            for (int x0 = 0; x0 < CH; x0 += GROUP * PER) {
                uint4 v[GROUP];
#pragma unroll
                for (int g = 0; g < GROUP; ++g) v[g] = __ldcg(reinterpret_cast<const uint4*>(line + 32 * x0) + 32 * g);
#pragma unroll
                for (int g = 0; g < GROUP; ++g)                            // without a branch
                    asm volatile("{ .reg .pred q; setp.ne.u32 q, %1, 0; @q st.global.cg.v4.u32 [%0], {%2, %2, %2, %2}; }"
                                 :: "l"(reinterpret_cast<uint4*>(line + 32 * x0) + 32 * g), "r"(v[g].x | v[g].y | v[g].z | v[g].w), "r"(0) : "memory");
                WORD ev[GROUP * PER];
#pragma unroll
                for (int g = 0; g < GROUP; ++g) unpack(v[g], ev + g * PER);
#pragma unroll
                for (int x4 = 0; x4 < GROUP * PER; x4 += 4) {
                    int cell[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        cell[k] = A;
                        w = __viaddmax_s32(A, x0 + x4 + k, w);
                        // those whose last round this is take their s+o with them, the others use one more each
                        const int num = (int)(ev[x4 + k] >> shift);
                        C -= num;
                        A += C - (sizeof(WORD) == 4 ? (int)ev[x4 + k] - num * ((1 << (shift & 31)) - least) : (int)ev[x4 + k] + num * least);
                    }
                    *reinterpret_cast<int4*>(cells + at(x0 + x4)) = make_int4(cell[0], cell[1], cell[2], cell[3]);
                    end1 = cell[3];
                }
            }
            // the words that are read next: the admissions of a chunk are time enough to have them in L2
#pragma unroll
            for (int x = 0; x < CH; x += 128 / (int)sizeof(WORD))
                asm volatile("prefetch.global.L2 [%0];" :: "l"(line_of(slot + 1) + lane * (CH - PER) + x));
            return w;
        };
        int W0 = build(b0, 0);
        end0 = end1;
        int W1 = build(b1, 1) + CH;
        int slot = 2;                                                      // events of the chunk behind the two
        int dA0 = 0, dC0 = 0, dA1 = 0, dC1 = 0;
        int tau = hdr.t - T0;
        i64 tel = (((i64)hdr.tel_hi << 32) | (i64)(unsigned)hdr.tel_lo) + (i64)T0 * (n - q);
        int acc = 0;                                                       // sum of tau + o
        // kv_map_pos without branches: position x1 holds y1, x2 holds y2, those in between are shifted
        const int d_in = mv.type == 1 ? (mv.i < mv.j ? 1 : -1) : 0;
        const int x1 = mv.j, y1 = mv.i, x2 = mv.type == 0 ? mv.i : n, y2 = mv.j;
        const int in_lo = min(mv.i, mv.j), in_len = max(mv.i, mv.j) - in_lo;
        auto fetch = [&](int pos) -> int2 {
            int from = (unsigned)(pos - in_lo) <= (unsigned)in_len ? pos + d_in : pos;
            from = pos == x1 ? y1 : pos == x2 ? y2 : from;
            return P.m.tbl_base[KV_IDX(pos < n ? from : 0, n, 424)];
        };
        if (!valid) q = n;
        // the request at q, and the one behind it as it was read: nothing waits for it before it is needed
        const int2 so0 = fetch(q);
        int sp = so0.x + 1, om = so0.y - 1;
        int2 next = fetch(q + 1);

        for (i64 chunk = 0;; ++chunk) {
            int Uall = INT_MIN;
#pragma unroll
            for (int c = 0; c < NF; c += 2) Uall = __vimax3_s32(Uall, U[c], U[c + 1]);
            // ---- every lane admits and waits until it leaves the chunk
            for (int guard = 0;; ++guard) {
                const int lim = M - sp;                                    // fits at t  <=>  V[x] <= lim + t over the window
                // where the window reaches the chunk's last round and that one is over for every start, none is in this chunk
                if (tau + om >= CH - 1 && end0 + dA0 + (CH - 1) * dC0 > lim) tau = max(tau, CH);
                const bool act = q < n && tau < CH;
                if (!__any_sync(KV_FULL, act)) break;
                bool fits = act;
                const bool ask0 = act && W0 > lim + tau;
                const int from = kv_warp_min(ask0 ? tau : CH);
                if (from < CH) {
                    const int x_lo = from & ~3;
                    const int lim0 = lim - dA0;
                    // y: maximum of V behind a round, less the round; grows strictly towards the front.  First the
                    // four cells in which it passes the limit, then the cell.
                    const int rise = dC0;
                    int y = INT_MIN / 2, y_in = y, x_in = CH - 4;
#pragma unroll 2
                    for (int x4 = CH - 4; x4 >= x_lo; x4 -= 4) {
                        const int4 four = *reinterpret_cast<const int4*>(b0 + at(x4));
                        if (y <= lim0) { y_in = y; x_in = x4; }
                        const int m = __viaddmax_s32(four.w, 3 * (rise + 1), __viaddmax_s32(four.z, 2 * (rise + 1), __viaddmax_s32(four.y, rise + 1, four.x)));
                        y = __viaddmax_s32(y, 4, m + rise * x4);
                    }
                    int best = x_in + 4, best_w;
                    {
                        const int4 four = *reinterpret_cast<const int4*>(b0 + at(x_in));
                        const int cell[4] = {four.x, four.y, four.z, four.w};
                        y = y_in;
#pragma unroll
                        for (int k = 3; k >= 0; --k) {
                            y = __viaddmax_s32(y, 1, cell[k] + rise * (x_in + k));
                            if (y <= lim0) { y_in = y; best = x_in + k; }
                        }
                        best_w = y_in + best;
                    }
                    const bool cut = ask0 && tau + om < CH - 1;            // the window ends inside the chunk
                    if (ask0 && !cut) {
                        if (best < CH) { tau = max(tau, best); W0 = best_w + dA0; }
                        else { tau = CH; fits = false; }
                    }
                    if (__any_sync(KV_FULL, cut)) {
                        int d = 0;
#pragma unroll 2
                        for (int x4 = x_lo; x4 < CH; x4 += 4) {
                            const int4 four = *reinterpret_cast<const int4*>(b0 + at(x4));
                            const int cell[4] = {four.x, four.y, four.z, four.w};
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int x = x4 + k - tau;
                                if (cut && (unsigned)x <= (unsigned)om)
                                    d = max(d, __viaddmin_s32(cell[k] + (dC0 + 1) * (x4 + k), -(lim0 + tau), x + 1));
                            }
                        }
                        if (d > 0) { tau += d; fits = false; }
                    }
                }
                const bool ask1 = fits && W1 > lim + tau && tau + om >= CH;
                if (__any_sync(KV_FULL, ask1 || (fits && Uall > lim + tau && tau + om >= 2 * CH))) {
                if (__any_sync(KV_FULL, ask1)) {
                    const int lim1 = lim + tau - dA1 - CH, slope = dC1 + 1, end = tau + om - CH;
                    int w = INT_MIN, d = 0;
#pragma unroll 4
                    for (int x4 = 0; x4 < CH; x4 += 4) {
                        const int4 four = *reinterpret_cast<const int4*>(b1 + at(x4));
                        const int m = __viaddmax_s32(four.w, 3 * slope, __viaddmax_s32(four.z, 2 * slope, __viaddmax_s32(four.y, slope, four.x)));
                        w = max(w, m + slope * x4);
                    }
                    if (ask1) W1 = w + dA1 + CH;
                    const bool over1 = ask1 && w > lim1;                   // somewhere in the chunk: in the window?
                    if (__any_sync(KV_FULL, over1)) {
#pragma unroll 2
                        for (int x4 = 0; x4 < CH; x4 += 4) {
                            const int4 four = *reinterpret_cast<const int4*>(b1 + at(x4));
                            const int cell[4] = {four.x, four.y, four.z, four.w};
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int x = x4 + k;
                                if (x <= end) d = max(d, __viaddmin_s32(cell[k] + slope * x, -lim1, x + CH + 1 - tau));
                            }
                        }
                        if (over1 && d > 0) { tau += d; fits = false; }
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
                            const uint4 l = __ldcg(reinterpret_cast<const uint4*>(line + 32 * x0));
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
                    if (far1 && !far2) {
                        for (int x = last + 1 - CH; x < CH; ++x) b1[at(x)] -= a + CH + x;
                        if (last < 2 * CH - 1) end1 -= a + 2 * CH - 1;
                    }
                    if (fits && !far1) {
                        for (int x = last + 1; x < CH; ++x) b0[at(x)] -= a + x;
                        if (last < CH - 1) end0 -= a + CH - 1;
                    }
                }
                const int reach = fits ? last : 0;
                if (fits) {
                    sp = next.x + 1; om = next.y - 1;
                    ++q;
                }
                next = fetch(q + 1);
                // bounds of the far chunks the new windows reach
#pragma unroll
                for (int c0 = 0; c0 < NF; c0 += 4) {
                    if (reach_max < CH * (c0 + 2)) break;
#pragma unroll
                    for (int c = c0; c < c0 + 4; c += 2) {
                        if (reach >= CH * (c + 2)) U[c] += a + CH * (c + 3) - 1;
                        if (reach >= CH * (c + 3)) U[c + 1] += a + CH * (c + 4) - 1;
                        Uall = __vimax3_s32(Uall, U[c], U[c + 1]);
                    }
                }
                if (guard > most_turns) { if (lane == 0) atomicExch(P.m.status, KV_DEV_LOOP_CAP); break; }
            }
            if (!__any_sync(KV_FULL, q < n)) break;
            if (chunk > kv_loop_cap((i64)(1 << 30))) { if (lane == 0) atomicExch(P.m.status, KV_DEV_LOOP_CAP); break; }
            // ---- the next chunk
            tau -= CH;
            tel += (i64)CH * (n - q);
            int* const x = b0; b0 = b1; b1 = x;
            dA0 = dA1; dC0 = dC1; dA1 = 0; dC1 = 0;
            W0 = W1 - CH;
            end0 = end1;
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
