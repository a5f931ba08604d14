"""Kernel variants at the sizes where one takes over from another, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_2508_06133_b200 import binding as kv
from paper_2508_06133_b200 import workloads as W

pytestmark = pytest.mark.gpu


def kernels_of(f):
    """What f returns, and the names of the kernels that it launched."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as prof:
        out = f()
        torch.cuda.synchronize()
    return out, " ".join(" ".join([e.key] * e.count) for e in prof.key_averages())


def oracle_moves(s, o, M, base, codes):
    mv = [orc.decode_move(len(s), int(c)) for c in codes]
    return orc.eval_moves(s, o, M, base, [m[0] for m in mv], [m[1] for m in mv], [m[2] for m in mv])


@pytest.mark.parametrize("omax", [1, 2, 31, 32, 33, 34, 65, 1025, 1026, 2049, 2050, 4097, 4098, 8193, 8194])
def test_timeline_sizes(omax):
    """The longest decode at and beside the numbers of far chunks and far registers a timeline is built
    for, and the first length of the simulator that keeps every cell: explicit orders with starts, moves
    from snapshots (n = 70 has five), the starts checked again and one of them broken."""
    rng = np.random.default_rng(7 * omax)
    n, M = 70, 5 * omax + 40
    s = rng.integers(1, M - omax, n).astype(np.int32)
    o = rng.integers(1, omax + 1, n).astype(np.int32)
    o[:4] = omax
    s[:2] = 1
    s[::9] = M - o[::9]
    s[4:40:3] = 1                                            # several fit beside each other
    orders = np.stack([rng.permutation(n) for _ in range(3)]).astype(np.int32)
    codes = np.arange(0, 3 * n * (n - 1) // 2, 61, dtype=np.int64)
    with kv.Scheduler(s, o, M) as h:
        tel, _, starts = h.eval_batch(kv.CAND_ORDER, orders, want_starts=True)
        broken = starts.copy()
        broken[:, orders[0][n - 1]] = starts[:, 0]            # two requests at the start of the first
        again, ok, _ = h.eval_batch(kv.CAND_START_TIMES, np.concatenate([starts, broken]), want_feasible=True)
        h.set_base_order(orders[0])
        mtel, _, _ = h.eval_batch(kv.CAND_MOVE, codes)
        mtel2, _, mstarts = h.eval_batch(kv.CAND_MOVE, codes[:5], want_starts=True)
    for c in range(3):
        p, t, _ = orc.list_schedule_rounds(s, o, M, orders[c])
        assert tel[c] == t and (starts[c] == p).all()
        assert again[c] == t and ok[c]
        ref = orc.check_schedule(s, o, M, broken[c])
        assert again[3 + c] == ref["tel"] and bool(ok[3 + c]) == ref["feasible"]
    ref = oracle_moves(s, o, M, orders[0], codes)
    assert (mtel == ref).all() and (mtel2 == ref[:5]).all()
    assert (mstarts.astype(np.int64).sum(1) + int(o.sum()) == ref[:5]).all()


@pytest.mark.parametrize("omax", [98, 1025, 2049, 4097, 8193])
@pytest.mark.parametrize("beside", [1.5, 4, 30])
def test_waits_in_and_behind_the_near_chunks(omax, beside):
    """Windows of 63 to 66 and 94 to 98 rounds (the shortest that covers the two exact chunks wherever it begins, and
    those that end on the last round of the next one) among the shortest and the longest, budgets for 1.5 to 30 requests beside
    each other, so that waits end in the first chunk, in the second and many chunks further on: orders with starts, the same
    through the run that stands alone, and moves."""
    rng = np.random.default_rng(omax + int(10 * beside))
    n = 160
    o = rng.choice(np.array([1, 2, 31, 32, 33, 62, 63, 64, 65, 66, 67, 94, 95, 96, 97, 98, omax]), n).astype(np.int32)
    o[0] = omax
    s = np.where(rng.random(n) < 0.15, rng.integers(1, 6000, n), rng.integers(1, 300, n)).astype(np.int32)
    M = max(int((s + o).max()), int(beside * (s + o).mean()))
    orders = np.stack([rng.permutation(n) for _ in range(3)]).astype(np.int32)
    codes = np.arange(0, 3 * n * (n - 1) // 2, 149, dtype=np.int64)
    with kv.Scheduler(s, o, M) as h:
        tel, _, starts = h.eval_batch(kv.CAND_ORDER, orders, want_starts=True)
        ok = h.eval_batch(kv.CAND_START_TIMES, starts, want_feasible=True)[1]
        h.set_base_order(orders[0])
        mtel = h.eval_batch(kv.CAND_MOVE, codes)[0]
        final, ftel, _, _ = h.local_search(kv.NBHD_SWAP, 0, order=orders[1])
    for c in range(3):
        p, t, _ = orc.list_schedule_rounds(s, o, M, orders[c])
        assert tel[c] == t and (starts[c] == p).all()
    assert ok.all() and (final == orders[1]).all() and ftel == tel[1]
    assert (mtel == oracle_moves(s, o, M, orders[0], codes)).all()


@pytest.mark.parametrize("omax,beside", [(1, 1), (20, 1), (20, 3), (64, 2), (64, 400), (300, 1), (1024, 400), (2049, 400), (4097, 60),
                                         (8193, 400), (8194, 20)])
def test_runs_that_stand_alone(omax, beside):
    """The base run where nothing waits (requests go four at a time), where a burst of large requests ends that and small
    ones begin it again, and where nearly every request waits for a few rounds: TEL, and moves from its snapshots."""
    rng = np.random.default_rng(omax + beside)
    n = 397
    o = rng.integers(1, omax + 1, n).astype(np.int32)
    s = rng.integers(1, 40, n).astype(np.int32)
    o[100:110] = o[301] = omax
    s[100:110] += 20 * omax
    M = max(int((s + o).max()), int(beside * (s + o).mean()))
    codes = np.arange(0, 3 * n * (n - 1) // 2, 1999, dtype=np.int64)
    for base in (np.arange(n, dtype=np.int32), rng.permutation(n).astype(np.int32)):
        with kv.Scheduler(s, o, M) as h:
            final, tel, _, _ = h.local_search(kv.NBHD_SWAP, 0, order=base)
            mtel = h.eval_batch(kv.CAND_MOVE, codes)[0]
        assert (final == base).all() and tel == orc.list_schedule_rounds(s, o, M, base)[1]
        assert (mtel == oracle_moves(s, o, M, base, codes)).all()


@pytest.mark.parametrize("share", [0.05, 0.099, 0.101])
@pytest.mark.parametrize("omax,median", [(64, 20), (1025, 200), (2049, 200), (2049, 1500), (4097, 20), (4097, 400), (8193, 4000)])
def test_runs_that_stand_alone_by_share_of_the_budget(omax, median, share):
    """Every form of the base run on both sides of the budget from which requests are asked for four at a time."""
    rng = np.random.default_rng(omax + median)
    n = 333
    o = np.clip(rng.lognormal(np.log(median), 1.0, n), 1, omax).astype(np.int32)
    o[50] = omax
    s = rng.integers(1, 200, n).astype(np.int32)
    M = max(int((s + o).max()), int(share * float((s + o).sum())))
    base = rng.permutation(n).astype(np.int32)
    codes = np.arange(0, 3 * n * (n - 1) // 2, 4999, dtype=np.int64)
    with kv.Scheduler(s, o, M) as h:
        final, tel, _, _ = h.local_search(kv.NBHD_SWAP, 0, order=base)
        mtel = h.eval_batch(kv.CAND_MOVE, codes)[0]
    assert (final == base).all() and tel == orc.list_schedule_rounds(s, o, M, base)[1]
    assert (mtel == oracle_moves(s, o, M, base, codes)).all()


@pytest.mark.parametrize("part", [2, 3, 8])
def test_runs_that_stand_alone_on_the_largest_budget(part):
    """Four requests in a row hold more tokens than 31 bits count."""
    M, n = (1 << 30) - 1, 70
    rng = np.random.default_rng(part)
    s = (M // part - rng.integers(20, 60, n)).astype(np.int32)
    o = rng.integers(1, 20, n).astype(np.int32)
    base = rng.permutation(n).astype(np.int32)
    with kv.Scheduler(s, o, M) as h:
        assert h.local_search(kv.NBHD_SWAP, 0, order=base)[1] == orc.list_schedule_rounds(s, o, M, base)[1]


@pytest.mark.parametrize("n", [1, 31, 33, 127, 128, 129, 400, 4096])
def test_amin_running_lists(n):
    """Evictions from lists of running requests at and beside the multiples of what the warps of a CTA look at
    side by side, and the largest ids; nearly everything starts at once, on estimates of one round."""
    rng = np.random.default_rng(n)
    s = rng.integers(1, 4, n).astype(np.int32)
    o = rng.integers(1, 40, n).astype(np.int32)
    lower = np.where(rng.random(n) < 0.98, 1, o).astype(np.int32)
    M = max(int((s + o).max()), int(s.sum()) + 2 * n)
    order = rng.permutation(n).astype(np.int32)
    starts, tel, ev, peak, _ = kv.amin_simulate([n], s[None], lower[None], o[None], M, order[None])
    p, rtel, rev, rpeak = orc.amin_schedule_rounds(s, lower, o, M, order)
    assert (starts[0] == p).all() and (tel[0], ev[0], peak[0]) == (rtel, rev, rpeak)
    assert n < 100 or rev > n // 8


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1024, 1025, 2049, 12000, 20000])
def test_sorting_and_batch_selection_sizes(n):
    """One tile, its edges, several, and sizes beyond what the solvers keep in shared memory."""
    inst = W.mixed_backlog(n, 5 + n, 70000)
    s, o, M = inst.s, inst.o, inst.M
    s[: n // 3] = 17; o[: n // 3] = 9                         # ties in size and in decode length
    with kv.Scheduler(s, o, M) as h:
        order, offs, tel = h.sorted_f()
    r_order, r_offs = orc.sorted_f_prefix(s, o, M)
    assert (order == r_order).all() and (offs == r_offs).all()
    assert tel == orc.list_schedule_rounds(s, o, M, r_order)[1]


@pytest.mark.parametrize("n", [32768, 32769, 40000, 70001, 1048577])
def test_sorting_in_several_merges(n):
    """The last length that one merge sorts, the first that takes two, groups of runs that do not come out even,
    and the first that takes three; rows of start times, and through the Phase-1 sorts where n is not too large."""
    rng = np.random.default_rng(n)
    s = rng.integers(1, 50, n).astype(np.int32)
    o = rng.integers(1, 6, n).astype(np.int32)
    M = 1 << 28                                              # everything fits beside each other
    with kv.Scheduler(s, o, M) as h:
        order, _, tel = h.sorted_f()
        # one batch of everything, by ascending (o, index)
        assert (order == np.lexsort((np.arange(n), o))).all() and tel == int(o.astype(np.int64).sum())
        starts = np.stack([rng.integers(0, 300, n), rng.integers(0, 300, n)]).astype(np.int32)
        for budget in (M, 2000):                             # the second one is exceeded
            if budget < M:
                h2 = kv.Scheduler(s, o, budget)
            got, ok, _ = (h if budget == M else h2).eval_batch(kv.CAND_START_TIMES, starts, want_feasible=True)
            ref = [orc.check_schedule(s, o, budget, st) for st in starts]
            assert [int(x) for x in got] == [r["tel"] for r in ref]
            assert [bool(x) for x in ok] == [r["feasible"] for r in ref]
        h2.close()


@pytest.mark.parametrize("n", [2, 63, 65, 513, 1500])
@pytest.mark.parametrize("weight", [0, 1])
def test_local_swap_sizes(n, weight):
    """Blocks of the prefix minima and their edges; a large prefill weight (many swaps)."""
    rng = np.random.default_rng(n)
    M = 4000
    s = rng.integers(1, 900, n).astype(np.int32)
    o = rng.integers(1, 400, n).astype(np.int32)
    with kv.Scheduler(s, o, M) as h:
        if weight:
            h.set_prefill_weight(3, 2)
        order, offs, _ = h.sorted_f_local_swap()
    ref = orc.sorted_g_local_swap(s, o, M, 3, 2) if weight else orc.sorted_f_local_swap(s, o, M)
    assert (order == ref[0]).all() and (offs == ref[1]).all()


def test_solvers_beyond_shared_memory():
    """Local swap and quantile selection where their arrays are in global memory (more than 11,000)."""
    inst = W.mixed_backlog(12500, 3, 1 << 22)
    with kv.Scheduler(inst.s, inst.o, inst.M) as h:
        order, offs, _ = h.sorted_f_quantile(9)
    ref = orc.sorted_f_quantile(inst.s, inst.o, inst.M, 9)
    assert (order == ref[0]).all() and (offs == ref[1]).all()
    rng = np.random.default_rng(8)
    n, M = 12500, 1 << 21                                    # few batches and swaps: the oracle walks every pair
    s = np.full(n, 200, dtype=np.int32)
    o = np.sort(rng.integers(100, 400, n)).astype(np.int32)
    with kv.Scheduler(s, o, M) as h:
        order, offs, _ = h.sorted_f_local_swap()
    ref = orc.sorted_f_local_swap(s, o, M)
    assert (order == ref[0]).all() and (offs == ref[1]).all()


@pytest.mark.parametrize("n,M,alone", [(2047, 30000, False), (2048, 30000, False), (3000, (1 << 21) - 1, False),
                                       (3000, 1 << 21, False), (2100, 4000, True)])
def test_quantile_sizes(n, M, alone):
    """The first length whose keys are made beforehand and the last that goes without, sums of a tile in 32 and in 64 bits, and
    a list with more batches (one request each) than keys are made for."""
    rng = np.random.default_rng(n + M)
    s = rng.integers(M // 2 + 1, M // 2 + 400, n).astype(np.int32) if alone else rng.integers(1, M // 20, n).astype(np.int32)
    o = rng.integers(1, 300, n).astype(np.int32)
    with kv.Scheduler(s, o, M) as h:
        order, offs, _ = h.sorted_f_quantile(11)
    ref = orc.sorted_f_quantile(s, o, M, 11)
    assert (order == ref[0]).all() and (offs == ref[1]).all()
    assert not alone or len(offs) == n + 1


@pytest.mark.parametrize("n,M,beforehand", [(2048, 20000, True), (20000, 60000, False), (16000, 400000, True)])
def test_quantile_keys_where_they_cover_the_batches(monkeypatch, n, M, beforehand):
    """Keys are made beforehand where 64 MiB hold those of all batches there may well be (20,000 requests at a budget of 60,000:
    some 900 batches of 80 KB), and the same batches come without memory for them."""
    inst = W.mixed_backlog(n, 3, M)
    with kv.Scheduler(inst.s, inst.o, M) as h:
        (order, offs, tel), names = kernels_of(lambda: h.sorted_f_quantile(5))
    assert ("k2q_leading" in names) == beforehand, names
    with kv.Scheduler(inst.s, inst.o, M) as h:
        monkeypatch.setenv("KVSCHED_REFUSE_MB", "1")
        (order2, offs2, tel2), names = kernels_of(lambda: h.sorted_f_quantile(5))
    assert "k2q_leading" not in names, names
    assert (order == order2).all() and (offs == offs2).all() and tel == tel2
    if n <= 16000:
        ref = orc.sorted_f_quantile(inst.s, inst.o, M, 5)
        assert (order == ref[0]).all() and (offs == ref[1]).all()


def test_sweeps_without_memory_for_rings(monkeypatch):
    """The forms that keep state in device memory, with memory and without: the same TELs from a warp per candidate."""
    for inst, count, kernel in ((W.mixed_backlog(1000, 4, 65536), 60000, "k3_lane_moves"),
                                (W.mixed_backlog(3000, 4, 4194304, **dict(chat_o=(5.5, 1.0, 8, 4096))), 6000, "ChunkSim<4, true")):
        best = torch.zeros(2, dtype=torch.int64, device="cuda")
        tels = []
        for refuse in (False, True):
            tel = torch.empty(count, dtype=torch.int64, device="cuda")
            with kv.Scheduler(inst.s, inst.o, inst.M) as h:
                h.sorted_f()
                h.sweep_dev(64, best, sampled=True, seed=3, iteration=1)
                h.sync()
                if refuse:
                    monkeypatch.setenv("KVSCHED_REFUSE_MB", "4")
                _, names = kernels_of(lambda: (h.sweep_dev(count, best, sampled=True, seed=3, iteration=1, tel_out=tel), h.sync()))
            monkeypatch.delenv("KVSCHED_REFUSE_MB", raising=False)
            assert (kernel in names) != refuse, names
            tels.append(tel)
        assert torch.equal(*tels)


@pytest.mark.parametrize("n,M", [(9, 200), (40, 600), (24, 1100), (24, 1250)])
def test_dynamic_programme_sizes(n, M):
    """The last tables that fit shared memory and the first that do not."""
    rng = np.random.default_rng(n + M)
    s = rng.integers(1, M // 3, n).astype(np.int32)
    o = rng.integers(1, M // 4, n).astype(np.int32)
    with kv.Scheduler(s, o, M) as h:
        order, offs, _ = h.sorted_f_dp()
    ref = orc.sorted_f_exact(s, o, M, orc.DP)
    assert (order == ref[0]).all() and (offs == ref[1]).all()


@pytest.mark.parametrize("lookahead", [127, 128, 129, 400])
def test_online_windows(lookahead):
    """A burst of arrivals: windows up to and beyond what a plan keeps in registers, plans that live so
    long that several of their batches, the requests behind the window and late arrivals are used."""
    rng = np.random.default_rng(lookahead)
    n, M = 420, 3000
    s = rng.integers(1, 500, n).astype(np.int32)
    o = rng.integers(1, 120, n).astype(np.int32)
    a = np.sort(np.where(rng.random(n) < 0.7, 0, rng.integers(0, 2000, n))).astype(np.int32)
    for period in (10, 100000):
        starts, lat, _ = kv.online_simulate([n], a[None], s[None], o[None], M, kv.POLICY_SORTED_F, period, lookahead)
        p, tot = orc.online_schedule(a, s, o, M, kv.POLICY_SORTED_F, period, lookahead)
        assert (starts[0] == p).all() and lat[0] == tot


@pytest.mark.parametrize("n", [2, 40, 1170, 1171, 1531])
def test_host_candidates_are_checked(n):
    """An order with a repeated id, one with an id outside 0 .. n-1, a negative start and one of 2^30 are
    refused, wherever they stand, and not evaluated; the handle goes on.  1,170 are the most that the host checks."""
    rng = np.random.default_rng(n)
    s = rng.integers(1, 50, n).astype(np.int32)
    o = rng.integers(1, 50, n).astype(np.int32)
    good = np.stack([rng.permutation(n) for _ in range(7)]).astype(np.int32)
    with kv.Scheduler(s, o, 4000) as h:
        tel, _, starts = h.eval_batch(kv.CAND_ORDER, good, want_starts=True)
        for row, col, value in ((6, n - 1, good[6, 0]), (0, 0, n), (3, n // 2, -1)):
            bad = good.copy()
            bad[row, col] = value
            before = h.stats()[1]
            with pytest.raises(kv.SchedError) as e:
                h.eval_batch(kv.CAND_ORDER, bad, want_starts=True)
            assert e.value.code == kv.E_NOT_PERMUTATION and h.stats()[1] == before
        for row, col, value in ((6, n - 1, -1), (0, 0, 1 << 30)):
            bad = starts.copy()
            bad[row, col] = value
            before = h.stats()[1]
            with pytest.raises(kv.SchedError) as e:
                h.eval_batch(kv.CAND_START_TIMES, bad, want_feasible=True)
            assert e.value.code == kv.E_INVAL and h.stats()[1] == before
        again, ok, _ = h.eval_batch(kv.CAND_START_TIMES, starts, want_feasible=True)
    assert ok.all() and (again == tel).all()


@pytest.mark.parametrize("least", [1, 300])
@pytest.mark.parametrize("omax", [1, 31, 32, 33, 64, 65, 1024, 1025, 1026, 2049])
def test_moves_by_lanes(omax, least):
    """One thread per candidate: every move of 150 requests (33,525, four times over: short decodes keep the warp
    up to 94,000) with a budget that lets 1.5 to 3.3 rounds pass per request, event words of both widths, decodes at the
    edges of its chunks."""
    rng = np.random.default_rng(omax + least)
    n = 150
    s = rng.integers(least, 3000, n).astype(np.int32)
    o = rng.integers(1, omax + 1, n).astype(np.int32)
    o[::20] = omax
    s[0], o[0] = least, 1
    volume = int((s.astype(np.int64) * o + o.astype(np.int64) ** 2 // 2).sum())
    for rounds in (1.5, 3.3):
        M = max(int((s + o).max()), int(volume / (rounds * n)) + n)
        base = rng.permutation(n).astype(np.int32)
        codes = np.arange(3 * n * (n - 1) // 2, dtype=np.int64)
        with kv.Scheduler(s, o, M) as h:
            h.set_base_order(base)
            (tel, _, _), names = kernels_of(lambda: h.eval_batch(kv.CAND_MOVE, np.tile(codes, 4)))
        assert "k3_lane_moves<%d," % (32 if omax <= 1025 else 64) in names, names
        tel = tel.reshape(4, -1)
        assert (tel == tel[0]).all()
        assert (tel[0, ::11] == oracle_moves(s, o, M, base, codes[::11])).all()
        with kv.Scheduler(s, o, M) as h:                     # the same in calls that take a warp per candidate
            h.set_base_order(base)
            parts, names = kernels_of(lambda: [h.eval_batch(kv.CAND_MOVE, c)[0] for c in np.array_split(codes, 3)])
        assert "k3_lane_moves" not in names, names
        assert (tel[0] == np.concatenate(parts)).all()


@pytest.mark.parametrize("M,omax,thread", [(1 << 23, 2, True), (1 << 24, 3, True), (1 << 26, 2, False), (1 << 27, 40, False),
                                           ((1 << 30) - 1, 2, False), ((1 << 30) - 1, 1500, False), (1 << 28, 1500, True)])
def test_moves_on_the_largest_budgets(M, omax, thread):
    """Prefills of a third of the budget and less, with decodes of one and more rounds: the tokens of all that starts in the
    rounds of one chunk pass 32 bits.  Those backlogs keep the warp; the others (the last one has no decode below 700) are
    counted right by a thread each."""
    rng = np.random.default_rng(omax)
    n = 150
    least, most = (M // 60, M // 40) if omax == 1500 else (M // 5, M // 3)
    s = rng.integers(least, most, n).astype(np.int32)
    o = rng.integers(700 if thread and omax == 1500 else 1, omax + 1, n).astype(np.int32)
    o[::20] = omax
    base = rng.permutation(n).astype(np.int32)
    codes = np.arange(3 * n * (n - 1) // 2, dtype=np.int64)
    with kv.Scheduler(s, o, M) as h:
        h.set_base_order(base)
        (tel, _, _), names = kernels_of(lambda: h.eval_batch(kv.CAND_MOVE, np.tile(codes, 5)))
    assert ("k3_lane_moves" in names) == thread, names
    tel = tel.reshape(5, -1)
    assert (tel == tel[0]).all()
    assert (tel[0, ::11] == oracle_moves(s, o, M, base, codes[::11])).all()


@pytest.mark.parametrize("omax,median,smax,rounds,count,thread", [
    (1024, 200, 4000, 3.0, 24000, True), (1024, 200, 4000, 3.0, 18000, False),
    (64, 16, 2000, 2.0, 40000, False), (64, 16, 2000, 2.0, 95000, True),      # short decodes
    (1024, 256, 20, 6.0, 95000, False), (1024, 256, 20, 0.5, 40000, True),    # short prefills: memory grows
    (2048, 512, 20, 6.0, 95000, False), (2048, 512, 2000, 3.0, 40000, True),
    (1024, 200, 4000, 24.0, 62000, True), (1024, 200, 20, 1.0, 60000, True), (2048, 512, 2000, 0.5, 20000, True),
    (256, 20, 2000, 0.5, 28000, False)])
def test_which_form_a_sweep_takes(omax, median, smax, rounds, count, thread):
    """Backlogs on which a thread per candidate is slower than a warp (by up to ten times) keep the warp."""
    rng = np.random.default_rng(omax + median + smax)
    n = 2000
    s = rng.integers(1, smax, n).astype(np.int32)
    o = np.clip(np.round(rng.lognormal(np.log(median), 0.8, n)), 1, omax).astype(np.int32)
    o[0] = omax
    volume = (s.astype(np.float64) * o + o.astype(np.float64) ** 2 / 2).sum()
    M = max(int((s.astype(np.int64) + o).max()), int(volume / (rounds * n)))
    best = torch.zeros(2, dtype=torch.int64, device="cuda")
    with kv.Scheduler(s, o, M) as h:
        order = h.sorted_f()[0]
        _, names = kernels_of(lambda: (h.sweep_dev(count, best, sampled=True, seed=3, iteration=2), h.sync()))
    assert ("k3_lane_moves" in names) == thread and ("k3_eval_moves" in names) != thread, names
    value, m = best.tolist()
    i = orc.sample_move(n, 3, 2, m)
    assert orc.eval_moves(s, o, M, order, [i[0]], [i[1]], [i[2]])[0] == value


@pytest.mark.parametrize("omax", [2050, 4097])
def test_moves_from_device_rings(omax):
    """A warp per candidate with its ring in device memory: every move of 80 requests (9,480), budgets that let 1
    and 1.8 rounds pass per request."""
    rng = np.random.default_rng(omax)
    n = 80
    s = rng.integers(1, 3000, n).astype(np.int32)
    o = rng.integers(1, omax + 1, n).astype(np.int32)
    o[::20] = omax
    volume = int((s.astype(np.int64) * o + o.astype(np.int64) ** 2 // 2).sum())
    for rounds in (1.0, 1.8):
        M = max(int((s + o).max()), int(volume / (rounds * n)) + n)
        base = rng.permutation(n).astype(np.int32)
        codes = np.arange(3 * n * (n - 1) // 2, dtype=np.int64)
        with kv.Scheduler(s, o, M) as h:
            h.set_base_order(base)
            tel, _, _ = h.eval_batch(kv.CAND_MOVE, codes)
            parts = [h.eval_batch(kv.CAND_MOVE, c)[0] for c in np.array_split(codes, 4)]
        assert (tel[::7] == oracle_moves(s, o, M, base, codes[::7])).all()
        assert (tel == np.concatenate(parts)).all()


@pytest.mark.parametrize("n,M", [(7577, 65536), (8118, 65536), (5981, 1 << 22), (6313, 1 << 22)])
def test_longest_lists_of_the_policy_sweep(n, M):
    """The longest lists that the policies of one instance fit shared memory with, prefix sums of 32 and of 64
    bits, and two lengths in front of them; one request more is refused."""
    inst = W.mixed_backlog(n + 1, 5, M)
    pols = np.array([kv.POLICY_FCFS, kv.POLICY_SOF, kv.POLICY_TOTAL_SIZE, kv.POLICY_SORTED_F], dtype=np.int32)
    s, o = inst.s[:n].copy(), inst.o[:n].copy()
    with kv.Scheduler(s, o, M) as h:
        tel, _, starts = h.eval_batch(kv.CAND_POLICY, pols, want_starts=True)
    refs = [orc.policy_order(s, o, orc.FCFS), orc.policy_order(s, o, orc.SHORTEST_OUTPUT_FIRST),
            orc.policy_order(s, o, orc.TOTAL_SIZE_FIRST), orc.sorted_f_prefix(s, o, M)[0]]
    for k in range(4):
        p, t, _ = orc.list_schedule_rounds(s, o, M, refs[k])
        assert tel[0, k] == t and (starts[0, k] == p).all()
    if n in (8118, 6313):
        with kv.Scheduler(inst.s, inst.o, M) as h:
            with pytest.raises(kv.SchedError) as e:
                h.eval_batch(kv.CAND_POLICY, pols)
        assert e.value.code == kv.E_UNSUPPORTED


@pytest.mark.parametrize("far", [1, 2, 3, 4, 5, 8, 9, 225])
def test_windows_beyond_the_registers(far):
    """Decodes whose window ends in the first, second, ... chunk behind the 33 that the long-decode simulator
    keeps in registers, and beside it: orders, starts and moves (n = 60 has eight states to resume from)."""
    rng = np.random.default_rng(far)
    n, top = 60, 32 * (33 + far)
    o = np.where(rng.random(n) < 0.5, rng.integers(top - 63, top + 1, n), rng.integers(1, top, n)).astype(np.int32)
    o[0], o[1:3] = 8300, (top, top - 31)                     # the first asks for this simulator
    s = rng.integers(1, 4000, n).astype(np.int32)
    M = 2 * int((s.astype(np.int64) + o).max())
    orders = np.stack([rng.permutation(n) for _ in range(3)]).astype(np.int32)
    codes = np.arange(0, 3 * n * (n - 1) // 2, 37, dtype=np.int64)
    with kv.Scheduler(s, o, M) as h:
        tel, _, starts = h.eval_batch(kv.CAND_ORDER, orders, want_starts=True)
        h.set_base_order(orders[0])
        mtel, _, _ = h.eval_batch(kv.CAND_MOVE, codes)
    for c in range(3):
        p, t, _ = orc.list_schedule_rounds(s, o, M, orders[c])
        assert tel[c] == t and (starts[c] == p).all()
    assert (mtel == oracle_moves(s, o, M, orders[0], codes)).all()


@pytest.mark.parametrize("omax", [1, 12, 33, 40])
def test_moves_of_short_windows(omax):
    """The simulator for windows that mostly end in the chunk they begin in, and beside them windows that end on
    its last round and in the two chunks behind it; with a longer mean decode the other one is taken."""
    rng = np.random.default_rng(omax)
    n, M = 300, 5000
    s = rng.integers(1, 2000, n).astype(np.int32)
    o = rng.integers(1, min(omax, 12) + 1, n).astype(np.int32)
    o[::30] = omax
    codes = rng.integers(0, 3 * n * (n - 1) // 2, 3000).astype(np.int64)
    base = rng.permutation(n).astype(np.int32)
    with kv.Scheduler(s, o, M) as h:
        h.set_base_order(base)
        (tel, _, _), names = kernels_of(lambda: h.eval_batch(kv.CAND_MOVE, codes))
    assert "ChunkSim<1, false, true>" in names, names
    assert (tel[::5] == oracle_moves(s, o, M, base, codes[::5])).all()
    with kv.Scheduler(s, 40 * o, M) as h:
        _, names = kernels_of(lambda: h.eval_batch(kv.CAND_MOVE, codes))
    assert ("ChunkSim<1, false, false>" if 40 * omax <= 1025 else "ChunkSim<2, false, false>") in names, names


@pytest.mark.parametrize("median,short", [(12, True), (16, True), (32, False)])
def test_backlogs_that_take_the_simulator_of_short_windows(median, short):
    """Log-normal decodes: shares of short ones of 0.98, 0.96 and 0.84."""
    rng = np.random.default_rng(median)
    n = 3000
    s = rng.integers(1, 500, n).astype(np.int32)
    o = np.clip(np.round(rng.lognormal(np.log(median), 0.8, n)), 1, 512).astype(np.int32)
    codes = rng.integers(0, 3 * n * (n - 1) // 2, 3000).astype(np.int64)
    base = rng.permutation(n).astype(np.int32)
    with kv.Scheduler(s, o, 30000) as h:
        h.set_base_order(base)
        (tel, _, _), names = kernels_of(lambda: h.eval_batch(kv.CAND_MOVE, codes))
    assert ("ChunkSim<1, false, true>" in names) == short, names
    assert (tel[::300] == oracle_moves(s, o, 30000, base, codes[::300])).all()


@pytest.mark.parametrize("count", [5000, 32768, 32769, 80000])
def test_launches_of_moves_from_device_rings(count):
    """32,768 rings of 16 KB per launch: every launch counts, and the candidates of all of them agree with a call
    that holds them in shared memory."""
    rng = np.random.default_rng(count)
    n = 40
    s = rng.integers(1000, 3000, n).astype(np.int32)
    o = rng.integers(1, 4098, n).astype(np.int32)
    o[0] = 4097
    M = int((s.astype(np.int64) * o + o.astype(np.int64) ** 2 // 2).sum() // n)
    total = 3 * n * (n - 1) // 2
    codes = np.arange(count, dtype=np.int64) % total
    with kv.Scheduler(s, o, M) as h:
        few, _, _ = h.eval_batch(kv.CAND_MOVE, np.arange(total, dtype=np.int64))
        before = h.stats()[0]
        (tel, _, _), names = kernels_of(lambda: h.eval_batch(kv.CAND_MOVE, codes))
        launches = h.stats()[0] - before
    assert names.count("k3_eval_moves<ChunkSim<4, true") == -(-count // 32768), names
    assert launches == names.count("k3_eval_moves<") + names.count("k4_"), names
    assert (tel == few[codes]).all()


@pytest.mark.parametrize("omax", [1000, 4000])
def test_kernel_time_without_the_search_for_memory(omax):
    """The first large sweep of a handle allocates its rings of a few hundred MB; the kernel's time leaves that out."""
    rng = np.random.default_rng(omax)
    n, count = 100, 60000
    s = rng.integers(1000, 3000, n).astype(np.int32)
    o = rng.integers(omax // 2, omax + 1, n).astype(np.int32)
    M = int((s.astype(np.int64) * o).sum() // n)
    best = torch.zeros(2, dtype=torch.int64, device="cuda")
    for _ in range(2):                                       # the first handle loads the kernels
        kv.release_cached_memory()
        with kv.Scheduler(s, o, M) as h:
            ms = []
            for k in range(3):
                h.sweep_dev(count, best, sampled=True, seed=1, iteration=0)
                h.sync()
                ms.append(h.last_eval_kernel_ms())
    assert ms[0] <= 1.5 * min(ms[1:]) + 0.05, ms


def test_orders_that_do_not_pass_through_pinned_memory():
    """4,300,000 requests: the order and the offsets of a solver and a search's order in and out."""
    n, M = 4300000, 1 << 28
    rng = np.random.default_rng(4)
    s = rng.integers(1, 8, n).astype(np.int32)
    o = rng.integers(1, 4, n).astype(np.int32)
    total = int(o.astype(np.int64).sum())
    with kv.Scheduler(s, o, M) as h:                         # everything fits beside each other
        order, offsets, tel = h.sorted_f()
        assert (order == np.lexsort((np.arange(n), o))).all() and list(offsets) == [0, n] and tel == total
        given = rng.permutation(n).astype(np.int32)
        final, tel, done, trace = h.local_search(kv.NBHD_SAMPLED, 1, order=given, seed=1, samples_per_iter=64)
        assert (final == given).all() and tel == total and done == 1 and trace[0, 1] == total
        assert (h.get_base_order() == given).all()
        with pytest.raises(kv.SchedError) as e:
            h.local_search(kv.NBHD_SAMPLED, 1, order=np.zeros(n, dtype=np.int32), seed=1, samples_per_iter=64)
        assert e.value.code == kv.E_NOT_PERMUTATION


@pytest.mark.parametrize("omax", [1, 300, 1500, 5000])
def test_schedules_of_more_rounds_than_a_permutation_has(omax):
    """Device form: orders that repeat one long request (they are not detected) and start times up to 2^31, sparse and one behind the
    other, in rounds that the permutations of the list never reach."""
    n, M, far = 700, 40000, (1 << 31) - 1 - omax
    s = np.full(n, M // 3, np.int32)
    o = np.full(n, omax, np.int32)
    rng = np.random.default_rng(omax)
    gap = omax if omax > 1 else 2
    rows = np.stack([np.sort(rng.integers(0, far, n)), far - gap * np.arange(n - 1, -1, -1), far - (gap - 1) * np.arange(n - 1, -1, -1),
                     (1 << 29) - 350 * gap + gap * np.arange(n), np.full(n, far)]).astype(np.int32)
    starts = torch.from_numpy(rows).cuda()
    tel = torch.zeros(len(rows), dtype=torch.int64, device="cuda")
    ok = torch.zeros(len(rows), dtype=torch.uint8, device="cuda")
    with kv.Scheduler(s, o, M) as h:
        h.eval_batch_dev(kv.CAND_START_TIMES, len(rows), starts, tel, ok, None)
        h.sync()
    for r, good, total in zip(rows.astype(np.int64), ok.tolist(), tel.tolist()):
        ends = r + omax                                       # memory is fullest in somebody's last round
        beside = (r[None] < ends[:, None]) & (ends[:, None] <= ends[None])
        most = np.where(beside, s[0] + ends[:, None] - r[None], 0).sum(1).max()
        assert bool(good) == (most <= M) and total == int((r + omax).sum())


def test_orders_that_go_on_for_two_to_the_thirty_rounds():
    """Device form: one request of 8,000 rounds 150,000 times over, each alone in the memory, between others that run once."""
    n, M = 150000, 16000
    s, o = np.full(n, 10, np.int32), np.full(n, 7, np.int32)
    s[0], o[0] = 8000, 8000
    order = np.zeros(n, np.int32)
    order[-40:] = np.arange(1, 41)
    with kv.Scheduler(s, o, M) as h:
        tel = torch.zeros(1, dtype=torch.int64, device="cuda")
        starts = torch.zeros((1, n), dtype=torch.int32, device="cuda")
        h.eval_batch_dev(kv.CAND_ORDER, 1, torch.from_numpy(order[None]).cuda(), tel, None, starts)
        h.sync()
    p = 8000 * np.arange(n, dtype=np.int64)
    p[-40:] = p[-41]                                          # 40 requests of 17 tokens fit beside the last long one at once
    assert p[-1] > 1 << 30
    assert (starts.cpu().numpy()[0, 1:41] == p[-1]).all()
    assert tel.item() == int(p.sum()) + 8000 * (n - 40) + 7 * 40
