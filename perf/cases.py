"""The work that users of the framework have it do, as timed cases.

A case names an operation (a call, or the few calls of one program, on the public Python binding of
the C library) and the backlog it runs on:

    plan        a small backlog planned in full: Sorted-F, the exact dynamic programme, 2-swap search
    sorted_f    Sorted-F with prefix-F batch selection, results on the host
    local_swap  Sorted-F with Algorithm 3 (Local Swap Search)
    quantile    Sorted-F with Algorithm 4 (Quantile Greedy Selection)
    sweep       one sampled swap + insert neighbourhood of the Sorted-F order, on the device
    search      order-level local search from the Sorted-F order, every swap in every iteration
    policy      many small instances under the four order policies
    orders      explicit orders scored through host memory, their start times checked again
    online      arrival streams simulated under one policy
    amin        Sorted-F + A_min executed against many outcomes of the decode lengths

Backlogs are the seeded synthetic ones of the framework: `mixed` (short chats and long documents,
decodes up to 1,024), `heavy` (longer tail, decodes up to 4,096), `paper` (the paper's own lengths,
decodes up to 2,048), `uniform` (short lengths up to `hi`).  All results are integers and do not depend
on the order in which anything is computed, so two correct implementations agree exactly.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_06133_b200 import binding as kv
from paper_2508_06133_b200 import workloads as W

HEAVY = dict(frac_long=0.3, chat_s=(6.0, 1.0, 16, 8192), chat_o=(5.5, 1.0, 8, 4096),
             doc_s=(8192, 32768), doc_o=(256, 1024))
PAPER = dict(chat_s=(2.48, 1.58, 1, 4096), chat_o=(3.76, 1.17, 1, 2048), doc_s=(500, 4800), doc_o=(30, 560))
MIXTURES = {"mixed": {}, "heavy": HEAVY, "paper": PAPER}

# mean decode length of each mixture (of a uniform backlog it is (1 + hi) / 2)
MEAN_O = {"mixed": 235.0, "heavy": 470.0, "paper": 128.0}

# cells of the occupancy timeline that the largest listed sweep updates; drawn sweeps and searches stay below
MOST_CELLS = 2.2e11


def listed():
    return [
        # one user's handful of requests: every call is launches and latency
        {"name": "plan_tiny_16", "op": "plan", "lengths": "uniform", "hi": 32, "n": 16, "M": 256, "iters": 16},
        # ordering an ordinary backlog before serving it
        {"name": "sorted_f_mixed_1k", "op": "sorted_f", "lengths": "mixed", "n": 1000, "M": 65536},
        # ordering the largest backlog
        {"name": "sorted_f_heavy_100k", "op": "sorted_f", "lengths": "heavy", "n": 100000, "M": 4194304},
        # the paper's experiment: n = 2,000 with Local Swap Search in Phase 1
        {"name": "local_swap_paper_2k", "op": "local_swap", "lengths": "paper", "n": 2000, "M": 16492},
        # the paper's other Phase-1 heuristic on the ten-thousand-request backlog
        {"name": "quantile_mixed_10k", "op": "quantile", "lengths": "mixed", "n": 10000, "M": 262144},
        # one iteration of a sampled local search on the ten-thousand-request backlog
        {"name": "sweep_mixed_10k", "op": "sweep", "lengths": "mixed", "n": 10000, "M": 262144, "moves": 65536, "tels": False},
        # the same on the largest backlog (decodes up to 4,096), every TEL kept
        {"name": "sweep_heavy_100k", "op": "sweep", "lengths": "heavy", "n": 100000, "M": 4194304, "moves": 7000, "tels": True},
        # 2-swap local search on the thousand-request backlog, its first iterations
        {"name": "search_mixed_1k", "op": "search", "lengths": "mixed", "n": 1000, "M": 65536, "iters": 2},
        # comparing policies over thousands of small instances
        {"name": "policy_4096x256", "op": "policy", "lengths": "mixed", "B": 4096, "n": 256, "M": 32768},
        # a user's own orders, scored and checked through host memory; sizes that divide nothing
        {"name": "orders_paper_1531x777", "op": "orders", "lengths": "paper", "n": 1531, "M": 16492, "count": 777},
        # the paper's Poisson experiment: ten rates, five streams each, Sorted-F-Online
        {"name": "online_sorted_f_50", "op": "online", "lengths": "paper", "policy": "sorted_f", "B": 50, "horizon": 4000, "M": 16492},
        # Sorted-F + A_min at the paper's scale, many outcomes of the decode lengths
        {"name": "amin_paper_2k_x64", "op": "amin", "lengths": "paper", "B": 64, "n": 2000, "M": 16492, "gamma": 0.5},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _backlog(rng, n):
    """Lengths and budget for n requests: budgets grow with the backlog, as in the framework's workloads."""
    kinds = ["mixed", "paper"] if n < 5000 else ["mixed"] if n < 20000 else ["mixed", "heavy"]
    kind = rng.choice(kinds)
    if kind == "paper":
        return {"lengths": kind, "n": n, "M": _log(rng, 12000, 40000)}
    if kind == "heavy":
        return {"lengths": kind, "n": n, "M": _log(rng, 1 << 20, 1 << 22)}
    return {"lengths": kind, "n": n, "M": _log(rng, 40000, 400000)}


def draw(rng):
    op = rng.choice(["plan", "sorted_f", "sorted_f", "local_swap", "quantile", "sweep", "sweep", "sweep", "search",
                     "policy", "orders", "online", "amin"])
    if op == "plan":
        return {"op": op, "lengths": "uniform", "hi": _log(rng, 16, 64), "n": rng.randint(9, 40), "M": rng.randint(200, 600),
                "iters": 8}
    if op == "sorted_f":
        return {"op": op, **_backlog(rng, _log(rng, 100, 100000))}
    if op == "local_swap":
        return {"op": op, **_backlog(rng, _log(rng, 200, 10000))}
    if op == "quantile":
        return {"op": op, **_backlog(rng, _log(rng, 200, 10000))}
    if op == "sweep":
        c = {"op": op, **_backlog(rng, _log(rng, 300, 100000))}
        per_move = 2.0 / 3.0 * c["n"] * MEAN_O[c["lengths"]]
        c["moves"] = max(64, min(1 << 20, int(_log(rng, 10 ** 9, int(MOST_CELLS)) / per_move)))
        c["tels"] = rng.random() < 0.5
        return c
    if op == "search":
        n = _log(rng, 64, 1000)
        return {"op": op, "lengths": "mixed", "n": n, "M": _log(rng, 40000, 130000), "iters": 2 if n > 400 else rng.randint(2, 6)}
    if op == "policy":
        return {"op": op, "lengths": "mixed", "B": _log(rng, 64, 8192), "n": _log(rng, 40, 512), "M": rng.choice([32768, 65536])}
    if op == "orders":
        n = _log(rng, 100, 4000)
        c = {"op": op, **_backlog(rng, n)}
        c["count"] = max(1, min(4000, _log(rng, 10000, 1200000) // n))
        return c
    if op == "online":
        return {"op": op, "lengths": "paper", "policy": rng.choice(["fcfs", "sof", "sorted_f"]), "B": _log(rng, 1, 120),
                "horizon": _log(rng, 300, 3500), "M": 16492}
    return {"op": op, "lengths": "paper", "B": _log(rng, 1, 600), "n": _log(rng, 200, 2000), "M": 16492,
            "gamma": rng.choice([0.3, 0.5, 0.8, 1.0])}


def _lengths(case, n, seed):
    if case["lengths"] == "uniform":
        return W.uniform_backlog(n, seed, 1, case["hi"], case["M"])
    return W.mixed_backlog(n, seed, case["M"], **MIXTURES[case["lengths"]])


def prepare(case, seed):
    op = case["op"]
    if op == "policy":
        inst = _lengths(case, case["B"] * case["n"], seed)
        h = kv.Scheduler.batch(inst.s.reshape(case["B"], -1), inst.o.reshape(case["B"], -1), case["M"])
        policies = torch.tensor([kv.POLICY_SORTED_F, kv.POLICY_FCFS, kv.POLICY_SOF, kv.POLICY_TOTAL_SIZE],
                                dtype=torch.int32, device="cuda")
        return {"op": op, "h": h, "policies": policies, "tel": torch.empty(case["B"] * 4, dtype=torch.int64, device="cuda")}
    if op == "online":
        # rates from well below to about three times what the memory sustains, as in the paper's experiment
        rates = np.linspace(0.03, 0.30, 10)
        streams = [W.online_poisson(float(rates[b % 10]), case["horizon"], seed=1000 * seed + b, M=case["M"])
                   for b in range(case["B"])]
        n_each = np.array([x.n for x in streams], dtype=np.int32)
        busiest = 0.30 * case["horizon"]                           # rows as long as the busiest stream may get
        n_max = max(int(busiest + 6 * math.sqrt(busiest)) + 8, int(n_each.max()))
        rows = np.zeros((3, case["B"], n_max), dtype=np.int32)
        for b, x in enumerate(streams):
            rows[:, b, :x.n] = x.a, x.s, x.o
        policy = {"fcfs": kv.POLICY_FCFS, "sof": kv.POLICY_SOF, "sorted_f": kv.POLICY_SORTED_F}[case["policy"]]
        return {"op": op, "args": (n_each, rows[0], rows[1], rows[2], case["M"], policy)}
    inst = _lengths(case, case["n"], seed)
    if op == "amin":
        # the planner knows a lower bound of every decode length; the outcomes lie between it and the upper bound
        B, n = case["B"], case["n"]
        lower = np.maximum(1, (inst.o * case["gamma"]).astype(np.int32))
        u = W.uniform01(seed, 60, np.arange(B * n)).reshape(B, n)
        truth = (lower + np.floor(u * (inst.o - lower + 1))).astype(np.int32)
        with kv.Scheduler(inst.s, lower, case["M"]) as h:
            order = h.sorted_f()[0]
        return {"op": op, "args": (np.full(B, n, dtype=np.int32), np.tile(inst.s, (B, 1)), np.tile(lower, (B, 1)), truth,
                                   case["M"], np.tile(order, (B, 1)))}
    h = kv.Scheduler(inst.s, inst.o, case["M"])
    # arrays of a fixed size that receive the batch offsets and the search's trace, whose lengths differ
    state = {"op": op, "h": h, "seed": seed, "offsets": np.empty(case["n"] + 1, dtype=np.int32),
             "trace": np.empty((case.get("iters", 1), 2), dtype=np.int64)}
    if op in ("sweep", "search"):
        state["order"] = h.sorted_f()[0]
    if op == "sweep":
        state["moves"] = case["moves"]
        state["best"] = torch.zeros(2, dtype=torch.int64, device="cuda")
        state["tel"] = torch.empty(case["moves"], dtype=torch.int64, device="cuda") if case["tels"] else None
    if op in ("search", "plan"):
        state["iters"] = case["iters"]
    if op == "orders":
        keys = W.u64(seed, 70, np.arange(case["count"] * case["n"])).reshape(case["count"], case["n"])
        state["orders"] = np.argsort(keys, axis=1).astype(np.int32)
    return state


def _whole(buffer, values):
    """`values` at the front of `buffer`, which is handed back; -1 behind them."""
    buffer[:len(values)] = values
    buffer[len(values):] = -1
    return buffer


def run(state):
    op = state["op"]
    h = state.get("h")
    if op == "sweep":
        h.sweep_dev(state["moves"], state["best"], sampled=True, seed=state["seed"], iteration=1, tel_out=state["tel"])
        return state["best"], state["tel"]
    if op == "policy":
        h.eval_batch_dev(kv.CAND_POLICY, 4, state["policies"], state["tel"])
        return state["tel"]
    if op in ("sorted_f", "local_swap", "quantile"):
        order, offsets, tel = (h.sorted_f() if op == "sorted_f" else h.sorted_f_local_swap() if op == "local_swap"
                               else h.sorted_f_quantile(state["seed"]))
        return order, _whole(state["offsets"], offsets), tel
    if op in ("plan", "search"):
        exact = h.sorted_f_dp() if op == "plan" else None
        order, offsets, greedy = h.sorted_f() if op == "plan" else (state["order"], (), 0)
        final, tel, done, trace = h.local_search(kv.NBHD_SWAP, state["iters"], order=order)
        return (exact[0], exact[2]) if exact else 0, greedy, _whole(state["offsets"], offsets), final, tel, done, _whole(state["trace"], trace)
    if op == "orders":
        tel, _, starts = h.eval_batch(kv.CAND_ORDER, state["orders"], want_starts=True)
        checked, feasible, _ = h.eval_batch(kv.CAND_START_TIMES, starts, want_feasible=True)
        return tel, starts, checked, feasible
    if op == "online":
        return kv.online_simulate(*state["args"])[:2]              # the third value is a time
    return kv.amin_simulate(*state["args"])[:4]


def work(case):
    """Inputs read and outputs written once; two operations (a comparison and an addition) for every
    round of every request that has to be placed on a timeline of its own."""
    op, n = case["op"], case.get("n", 0)
    mean_o = (1 + case["hi"]) / 2 if case["lengths"] == "uniform" else MEAN_O[case["lengths"]]
    if op == "sweep":                                   # two uniform positions: two thirds of the list lie behind the first
        runs, cells = case["moves"], case["moves"] * 2.0 / 3.0 * n * mean_o
        data = 8 * n + (8 * case["moves"] if case["tels"] else 16)
    elif op == "search":
        runs = case["iters"] * n * (n - 1) / 2
        cells, data = runs * 2.0 / 3.0 * n * mean_o, 8 * n + 8 * n
    elif op == "plan":                                  # and a table of n x M x n for the dynamic programme
        cells = (3 * n * (n - 1) / 2 * 2.0 / 3.0 + 2) * n * mean_o + n * n * case["M"] / 2
        data = 8 * n + 16 * n
    elif op == "policy":
        cells, data = 4.0 * case["B"] * n * mean_o, 8 * case["B"] * n + 32 * case["B"]
    elif op == "orders":                                # placed once to find the starts, once more to check them
        cells, data = 2.0 * case["count"] * n * mean_o, 8 * n + case["count"] * (8 * n + 4 * n + 4 * n + 17)
    elif op == "online":
        requests = case["B"] * 0.165 * case["horizon"]  # mean rate of the ten
        cells, data = requests * mean_o, 16 * requests + 8 * case["B"]
    elif op == "amin":
        cells, data = case["B"] * n * mean_o, case["B"] * (16 * n + 4 * n + 24)
    else:                                               # a Phase-1 solver and one run of its order
        cells, data = n * mean_o, 8 * n + 4 * n + 8
    return {"bytes": float(data), "flops": 2.0 * cells}


def tolerance(case):
    return "exact"
