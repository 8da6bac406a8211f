"""Performance cases: the calls a user of the device-mapping search makes, over the sizes they are made at.

A case names an entry point of ``paper_2607_22242_gb300.bf`` (``call``), a workflow shape (``dag``, with ``dag_seed`` for
its random edges), the number of tools and the entry point's own arguments.  Tool profiles (latencies, transfers,
footprints) come from the seed handed to ``prepare``: the same workflow profiled anew, as a scheduler that re-profiles
its tools searches it.  The recipes are those of the package's standard workloads (``scenarios.py``): GPU latency
lognormal(40 ms, 0.8), CPU 0.5 to 20 times that (or the four scheduling zones), transfer 1 to 30 ms, load-in 40 us/MiB,
contention 1 + 0.35 (k - 1).
"""
import numpy as np
import torch

from paper_2607_22242_gb300 import bf
from paper_2607_22242_gb300.scenarios import Scenario

INFEASIBLE = 0xFFFFFFFF
COLUMNS = ("pred_mask", "cpu_us", "gpu_us", "xfer_us", "load_us", "vram_mib")


# ---- workflows ------------------------------------------------------------------------------------------------------

def _edges(dag, n, rng):
    """Predecessor masks of n topologically numbered tools."""
    pred = [0] * n
    if dag == "chain":
        for v in range(1, n):
            pred[v] = 1 << (v - 1)
    elif dag == "fan":  # one source, n - 2 branches, one sink
        for v in range(1, n - 1):
            pred[v] = 1
        if n > 2:
            pred[n - 1] = (1 << (n - 1)) - 2
        elif n == 2:
            pred[1] = 1
    elif dag == "spine":  # a spine with a fan-out of 6 beside every third of its tools, cut after n tools
        tools, prev = [0], 0
        while len(tools) < n:
            head = len(tools)
            tools.append(1 << prev)
            first = len(tools)
            tools += [1 << head] * 7
            prev = len(tools)
            tools.append(sum(1 << v for v in range(first, first + 7)))
        pred = tools[:n]
    elif dag == "layered":  # layers of 4, an edge to each tool of the next layer with probability 0.4
        for v in range(4, n):
            for u in range((v // 4 - 1) * 4, v // 4 * 4):
                if rng.random() < 0.4:
                    pred[v] |= 1 << u
    elif dag == "sparse":  # any earlier tool with probability 0.2
        for v in range(1, n):
            for u in range(v):
                if rng.random() < 0.2:
                    pred[v] |= 1 << u
    else:
        raise ValueError(dag)
    return pred


# VRAM footprints (MiB) and budget of each shape: fan-outs and chains without pressure, spines mildly tight, layered and
# sparse workflows with tools of 2 to 16 GiB against a 24 GiB budget, where queueing and infeasible mappings dominate.
MEMORY = {"chain": (512, 6144, 81920), "fan": (512, 6144, 81920), "spine": (512, 6144, 32768),
          "layered": (2048, 16384, 24576), "sparse": (2048, 16384, 24576)}


def _workflow(dag, n, edge_rng, rng, budget=None):
    """One workflow's tables as plain lists."""
    lo, hi, default_budget = MEMORY[dag]
    g = np.clip(np.rint(rng.lognormal(np.log(40000.0), 0.8, n)), 1, 2_000_000)
    x = np.rint(rng.uniform(1000.0, 30000.0, n))
    m = rng.integers(lo, hi, n, endpoint=True)
    if dag == "spine":  # the four scheduling zones: GPU-preferred, ambiguous, CPU-preferred, neutral (11 : 4 : 1 : 3)
        zone = rng.permutation(np.resize(np.repeat(np.arange(4), (11, 4, 1, 3)), n))
        x = np.where(zone == 2, np.rint(g * rng.uniform(1.5, 3.0, n)), np.where(zone == 3, np.rint(x / 30), x))
        m = np.where(zone == 3, m // 48, m)
        c = np.select([zone == 0, zone == 1, zone == 2],
                      [g * rng.uniform(5.0, 70.0, n), g * rng.uniform(0.8, 1.5, n), (g + x) * rng.uniform(0.3, 0.5, n)],
                      g * rng.uniform(0.95, 1.05, n))
    else:
        c = g * rng.uniform(0.5, 20.0, n)
    c = np.clip(np.rint(c), 1, 40_000_000)
    as_list = lambda a: a.astype(np.int64).tolist()
    return dict(n=n, pred_mask=_edges(dag, n, edge_rng), cpu_us=as_list(c), gpu_us=as_list(g), xfer_us=as_list(x),
                load_us=as_list(40 * m), vram_mib=as_list(m), vram_budget_mib=int(budget or default_budget),
                slowdown_q10=[0] + [(1024 * (100 + (0 if dag == "chain" else 35) * (k - 1)) + 50) // 100
                                    for k in range(1, max(n, 20) + 1)])


def _single(case, seed):
    return _workflow(case["dag"], case["n"], np.random.default_rng(case["dag_seed"]),
                     np.random.default_rng([seed, case["n"], case["dag_seed"]]))


def _batch(case, seed):
    """`scenarios` workflows, each with its own edges, budget and (n_lo < n_hi) size."""
    rng = np.random.default_rng([seed, case["scenarios"], case["n_lo"], case["n_hi"]])
    out = []
    for _ in range(case["scenarios"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"], endpoint=True))
        dag = case["dag"] if case["dag"] != "mixed" else str(rng.choice(["chain", "fan", "spine", "layered", "sparse"]))
        budget = int(rng.integers(16384, 49152, endpoint=True)) if dag in ("layered", "sparse") else None
        out.append(_workflow(dag, n, rng, rng, budget))
    return out


def _sizes(case, seed=0):
    """Tools of each scenario of a batch whose sizes vary: only their mean matters for `work`."""
    lo, hi, s = case["n_lo"], case["n_hi"], case["scenarios"]
    return {n: s / (hi - lo + 1) for n in range(lo, hi + 1)}


# ---- the cases ------------------------------------------------------------------------------------------------------

def listed():
    return [
        # The smallest search: a short serial workflow on a kept handle, re-searched in a scheduler's loop.  Latency.
        {"name": "best_chain8", "call": "best", "dag": "chain", "n": 8, "dag_seed": 0},
        # One-off search of a new fan-out/fan-in workflow: no handle kept, so its set-up is part of the call.
        {"name": "once_fan12", "call": "once", "dag": "fan", "n": 12, "dag_seed": 0},
        # Full search of a layered workflow under a tight VRAM budget.
        {"name": "best_layered16", "call": "best", "dag": "layered", "n": 16, "dag_seed": 3},
        # The largest standard search: all 3^19 mappings of a spine with two fan-outs.
        {"name": "best_spine19", "call": "best", "dag": "spine", "n": 19, "dag_seed": 0},
        # One rank's ragged share of a sharded search.
        {"name": "range_layered16", "call": "range", "dag": "layered", "n": 16, "dag_seed": 3, "first": 14_348_908,
         "count": 14_348_909},
        # Every makespan of a ragged range of a large space written out (statistics of a workflow's mappings).
        {"name": "eval_spine19", "call": "eval", "dag": "spine", "n": 19, "dag_seed": 0, "first": 400_000_001,
         "count": 33_554_467},
        # Scattered candidate mappings (a sampler's or a heuristic's) scored together.
        {"name": "list_layered16", "call": "list", "dag": "layered", "n": 16, "dag_seed": 3, "count": 2_000_003},
        # The runtime monitor's what-if round around a mapping of a 28-tool workflow.  Latency.
        {"name": "whatif_spine28", "call": "whatif", "dag": "spine", "n": 28, "dag_seed": 0},
        # The largest batch: 4096 layered 10-tool workflows, each with its own budget, in one call.
        {"name": "batch_layered10", "call": "batch", "dag": "layered", "n_lo": 10, "n_hi": 10, "scenarios": 4096},
        # A scheduler's round over the workflows at hand, of all shapes and sizes, without allocating.
        {"name": "noalloc_mixed5to13", "call": "noalloc", "dag": "mixed", "n_lo": 5, "n_hi": 13, "scenarios": 200},
        # Exact optimum by branch and bound where full enumeration takes long.
        {"name": "pruned_layered18", "call": "pruned", "dag": "layered", "n": 18, "dag_seed": 3},
        # Exact optimum of the largest workflow the library takes.
        {"name": "tree_spine32", "call": "tree", "dag": "spine", "n": 32, "dag_seed": 0, "space": 3, "prune": True},
    ]


# Sizes of the drawn cases, per call and shape: up to what costs no more than the largest listed case.
DRAWN = {
    "best": {"chain": (1, 17), "fan": (2, 15), "spine": (6, 19), "layered": (5, 16), "sparse": (3, 15)},
    "range": {"chain": (6, 16), "fan": (6, 15), "spine": (8, 18), "layered": (6, 16), "sparse": (6, 15)},
    "eval": {"chain": (4, 17), "fan": (4, 16), "spine": (8, 19), "layered": (5, 17), "sparse": (4, 16)},
    "list": {"chain": (4, 32), "fan": (4, 24), "spine": (8, 32), "layered": (5, 32), "sparse": (4, 28)},
    "whatif": {"chain": (4, 32), "fan": (4, 24), "spine": (8, 32), "layered": (5, 32), "sparse": (4, 32)},
    "pruned": {"chain": (6, 20), "fan": (6, 14), "spine": (8, 20), "layered": (6, 18), "sparse": (6, 16)},
    "tree": {"chain": (6, 32), "fan": (6, 14), "spine": (8, 32), "layered": (6, 18), "sparse": (6, 16)},
}
DRAWN["once"] = DRAWN["best"]


def draw(rng):
    call = rng.choice(["best", "best", "once", "range", "eval", "list", "whatif", "batch", "noalloc", "pruned", "tree"])
    log_uniform = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))
    if call in ("batch", "noalloc"):
        n_lo = rng.randint(3, 12)
        n_hi = min(14, n_lo + rng.randint(0, 5))
        most = 241_864_704 // sum(3 ** n for n in range(n_lo, n_hi + 1)) * (n_hi - n_lo + 1)
        return {"call": call, "dag": rng.choice(["layered", "mixed"]), "n_lo": n_lo, "n_hi": n_hi,
                "scenarios": max(1, log_uniform(1, max(1, min(most, 4096 if call == "batch" else 1024))))}
    dag = rng.choice(sorted(DRAWN[call]))
    case = {"call": call, "dag": dag, "n": rng.randint(*DRAWN[call][dag]), "dag_seed": rng.randint(0, 1000)}
    total = 3 ** case["n"]
    if call in ("range", "eval"):
        case["count"] = min(total, log_uniform(min(total, 1000), min(total, 50_000_000)))
        case["first"] = rng.randint(0, total - case["count"])
    elif call == "list":
        case["count"] = log_uniform(1, 4_000_000)
    elif call == "tree":
        case["space"] = rng.choice([2, 3])
        case["prune"] = not (3 ** case["n"] < 10 ** 8 and rng.random() < 0.3)
    return case


# ---- preparation and one pass ---------------------------------------------------------------------------------------

def _scenario(tables):
    return Scenario(**tables)


def _random_indices(case, seed):
    rng = np.random.default_rng([seed, case["count"], 1])
    return rng.integers(0, 3 ** case["n"], case["count"], dtype=np.int64)


def _base_mapping(case, tables):
    """A plausible current mapping: each tool on its isolated-faster device."""
    return sum(3 ** v for v in range(case["n"])
               if tables["gpu_us"][v] + tables["xfer_us"][v] < tables["cpu_us"][v])


def prepare(case, seed):
    call = case["call"]
    state = {"case": case}
    if call in ("batch", "noalloc"):
        state["scenarios"] = [_scenario(t) for t in _batch(case, seed)]
        if call == "batch":
            state["packed"] = bf.pack_descs(state["scenarios"])
        return state
    tables = _single(case, seed)
    if call == "once":
        state["scenario"] = _scenario(tables)
        return state
    state["handle"] = bf.create_scenario(_scenario(tables))
    if call in ("eval", "list"):
        state["makespan"] = torch.empty(case["count"], dtype=torch.int32, device="cuda")
        state["feasible"] = torch.empty(case["count"], dtype=torch.uint8, device="cuda")
    if call == "list":
        state["indices"] = torch.from_numpy(_random_indices(case, seed)).cuda()
    if call == "whatif":
        state["base"] = _base_mapping(case, tables)
    return state


def _as_array(r):
    return np.array([r.index, r.makespan_us, int(r.feasible), *r.modes], dtype=np.int64)


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "best":
        return _as_array(bf.search_best(state["handle"]))
    if call == "once":
        return _as_array(bf.search_best(state["scenario"]))
    if call == "range":
        return _as_array(bf.search_range(state["handle"], case["first"], case["count"]))
    if call == "pruned":
        return _as_array(bf.search_pruned(state["handle"]))
    if call == "tree":
        return _as_array(bf.search_tree(state["handle"], case["space"], case["prune"])[0])
    if call == "eval":
        return bf.eval_mappings(state["handle"], case["first"], case["count"], state["makespan"], state["feasible"])
    if call == "list":
        return bf.eval_indices(state["handle"], state["indices"], state["makespan"], state["feasible"])
    if call == "whatif":
        probes = bf.whatif(state["handle"], state["base"])
        return np.array([(p.index, p.makespan_us, p.feasible, p.kind == "swap", p.tool, p.mode,
                          255 if p.other is None else p.other) for p in probes], dtype=np.int64)
    if call == "batch":
        res = bf.search_batch(state["scenarios"], packed=state["packed"])
    else:
        res = bf.search_batch_noalloc(state["scenarios"])
    return [np.array([r.index for r in res], dtype=np.int64), np.array([r.makespan_us for r in res], dtype=np.int64)]


DESC_BYTES = 908  # one scenario's tables as the library takes them


def work(case):
    """What one pass cannot do without.  A search forms every mapping's makespan (one addition to what it shares with
    others) and compares it; an evaluation writes 5 bytes per mapping; a branch and bound at least simulates its
    optimum (n events, each over up to n running and n waiting tools)."""
    call = case["call"]
    if call in ("batch", "noalloc"):
        sizes = _sizes(case)
        return {"bytes": case["scenarios"] * (DESC_BYTES + 16), "flops": 2 * sum(c * 3 ** n for n, c in sizes.items())}
    n = case["n"]
    if call in ("best", "once"):
        return {"bytes": DESC_BYTES + 16, "flops": 2 * 3 ** n}
    if call == "range":
        return {"bytes": DESC_BYTES + 16, "flops": 2 * case["count"]}
    if call == "eval":
        return {"bytes": DESC_BYTES + 5 * case["count"], "flops": case["count"]}
    if call == "list":
        return {"bytes": DESC_BYTES + 13 * case["count"], "flops": 2 * n * n * case["count"]}
    if call == "whatif":
        return {"bytes": DESC_BYTES + 24 * 2 * n, "flops": 2 * n * n * 2 * n}
    if call == "tree" and not case["prune"]:
        return {"bytes": DESC_BYTES + 16, "flops": 2 * case["space"] ** n}
    return {"bytes": DESC_BYTES + 16, "flops": 2 * n * n}


def tolerance(case):
    """Whole microseconds and mapping indices: nothing may differ."""
    return "exact"


# ---- the same in 64-bit integers, written from the model's rules ----------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _simulate(tabs, modes):
    """Makespans [S, B] (INFEASIBLE where a mapping is) of modes [S, n, B] under S scenarios of n tools each."""
    dev = modes.device
    S, n, B = modes.shape
    col = lambda name: torch.tensor([t[name][:n] for t in tabs], dtype=torch.int64, device=dev)[:, :, None]
    pred, c, g, x, load, m = (col(name) for name in COLUMNS)
    budget = torch.tensor([t["vram_budget_mib"] for t in tabs], dtype=torch.int64, device=dev)[:, None]
    slow = torch.tensor([t["slowdown_q10"][:n + 1] for t in tabs], dtype=torch.int64, device=dev)
    slow[:, 0] = 1024
    bit = (1 << torch.arange(n, dtype=torch.int64, device=dev))[None, :, None]
    order = torch.arange(n, dtype=torch.int64, device=dev)[None, :, None]
    FAR = 1 << 62
    cpu, now, que = modes == 0, modes == 1, modes == 2
    dead = (que & (m > budget[:, None])).any(1)
    pend = torch.ones((S, n, B), dtype=torch.bool, device=dev)
    run, wait = torch.zeros_like(pend), torch.zeros_like(pend)
    end = torch.zeros((S, n, B), dtype=torch.int64, device=dev)  # CPU: time; GPU: virtual clock; waiting: ready time
    T = torch.zeros((S, B), dtype=torch.int64, device=dev)
    V = torch.zeros_like(T)
    for _ in range(n + 1):
        open_ = ((pend | run | wait).to(torch.int64) * bit).sum(1, keepdim=True)
        ready = pend & ((pred & open_) == 0)
        pend = pend & ~ready
        end = torch.where(ready & cpu, T[:, None] + c, torch.where(ready & now, V[:, None] + (g + x) * 1024,
                          torch.where(ready & que, T[:, None].expand_as(end), end)))
        run = run | (ready & ~que)
        wait = wait | (ready & que)
        live = ((run & ~cpu).to(torch.int64) * m).sum(1)
        dead = dead | ((ready & now).any(1) & (live > budget))
        first = torch.where(wait, end * 64 + order, torch.full_like(end, FAR)).amin(1, keepdim=True)
        head = wait & (end * 64 + order == first) & ~(run & que).any(1, keepdim=True)
        head = head & (live[:, None] + m <= budget[:, None])
        end = torch.where(head, V[:, None] + (load + g + x) * 1024, end)
        run, wait = run | head, wait & ~head
        on_gpu = run & ~cpu
        k = on_gpu.sum(1)
        f = torch.gather(slow, 1, k)
        t_cpu = torch.where(run & cpu, end, torch.full_like(end, FAR)).amin(1)
        v_gpu = torch.where(on_gpu, end, torch.full_like(end, FAR)).amin(1)
        rem = torch.where(k > 0, v_gpu - V, torch.zeros_like(V))
        t_gpu = T + ((rem * f + (1 << 20) - 1) >> 20)
        gpu_event = (k > 0) & (t_gpu <= t_cpu)
        any_run = run.any(1)
        dt = torch.where(any_run & ~gpu_event, t_cpu - T, torch.zeros_like(T))
        V = torch.where(gpu_event, v_gpu, torch.where(k > 0, V + torch.div(dt << 20, f, rounding_mode="floor"), V))
        T = torch.where(gpu_event, t_gpu, T + dt)
        run = run & ~((run & cpu & (end == T[:, None])) | (on_gpu & gpu_event[:, None] & (end == V[:, None])))
    return torch.where(dead, torch.full_like(T, INFEASIBLE), T)


def _modes_of(index, n, radix=3):
    """Digits [n, B] of mapping numbers [B], tool 0 the least significant."""
    out = []
    for _ in range(n):
        out.append((index % radix).to(torch.int8))
        index = torch.div(index, radix, rounding_mode="floor")
    return torch.stack(out)


def _best(tabs, first, count, radix=3):
    """(index, makespan) of each scenario's best mapping among numbers [first, first + count); index in base 3."""
    dev, n = _device(), tabs[0]["n"]
    chunk = max(1, (1 << 25) // (n * len(tabs)))
    best = [(INFEASIBLE, first)] * len(tabs)
    for lo in range(first, first + count, chunk):
        idx = torch.arange(lo, min(lo + chunk, first + count), dtype=torch.int64, device=dev)
        modes = _modes_of(idx, n, radix)
        if radix == 2:
            idx = (modes.to(torch.int64) * (3 ** torch.arange(n, dtype=torch.int64, device=dev))[:, None]).sum(0)
        ms = _simulate(tabs, modes[None].expand(len(tabs), -1, -1))
        low = ms.amin(1)
        at = torch.where(ms == low[:, None], idx[None], torch.full_like(idx, 1 << 62)[None]).amin(1)
        for s, pair in enumerate(zip(low.tolist(), at.tolist())):
            best[s] = min(best[s], pair) if pair[0] != INFEASIBLE else best[s]
    return [(i, ms) for ms, i in best]


def _result(n, index, makespan):
    digits = [index // 3 ** v % 3 for v in range(n)]
    return np.array([index, makespan, int(makespan != INFEASIBLE), *digits], dtype=np.int64)


def _values(tabs, index):
    """Makespans and flags of listed mappings, as the evaluating entry points write them."""
    n, ms = tabs["n"], []
    for part in torch.split(index, (1 << 25) // n):
        ms.append(_simulate([tabs], _modes_of(part, n)[None])[0])
    ms = torch.cat(ms)
    return torch.where(ms >= 1 << 31, ms - (1 << 32), ms).to(torch.int32), (ms != INFEASIBLE).to(torch.uint8)


def exact(case, seed):
    call, dev = case["call"], _device()
    if call in ("batch", "noalloc"):
        scenarios = _batch(case, seed)
        found = [None] * len(scenarios)
        for n in sorted({t["n"] for t in scenarios}):
            ids = [i for i, t in enumerate(scenarios) if t["n"] == n]
            step = max(1, (1 << 24) // (n * 3 ** n))
            for at in range(0, len(ids), step):
                part = ids[at:at + step]
                for i, pair in zip(part, _best([scenarios[i] for i in part], 0, 3 ** n)):
                    found[i] = pair
        return [np.array([p[0] for p in found], dtype=np.int64), np.array([p[1] for p in found], dtype=np.int64)]
    tabs, n = _single(case, seed), case["n"]
    if call in ("best", "once", "pruned"):
        return _result(n, *_best([tabs], 0, 3 ** n)[0]) if n <= 17 else None
    if call == "range":
        return _result(n, *_best([tabs], case["first"], case["count"])[0])
    if call == "tree":
        return _result(n, *_best([tabs], 0, case["space"] ** n, case["space"])[0]) if case["space"] ** n <= 3 ** 17 else None
    if call == "eval":
        return _values(tabs, torch.arange(case["first"], case["first"] + case["count"], dtype=torch.int64, device=dev))
    if call == "list":
        return _values(tabs, torch.from_numpy(_random_indices(case, seed)).to(dev))
    base = _base_mapping(case, tabs)
    digits = [base // 3 ** v % 3 for v in range(n)]
    score = lambda idx: _values(tabs, torch.tensor(idx, dtype=torch.int64, device=dev))[0].tolist()
    rows = []
    for i in range(n):
        others = [a for a in range(3) if a != digits[i]]
        moved = [base + (a - digits[i]) * 3 ** i for a in others]
        for a, idx, ms in zip(others, moved, score(moved)):
            rows.append((idx, ms % (1 << 32), ms != -1, 0, i, a, 255))
            if a == 1 and ms == -1:  # moving it to the GPU exceeds the budget: swap with a tool there
                held = [j for j in range(n) if digits[j] == 1]
                swaps = [idx + 3 ** j for j in held]
                for j, idx2, ms2 in zip(held, swaps, score(swaps) if swaps else []):
                    rows.append((idx2, ms2 % (1 << 32), ms2 != -1, 1, i, 1, j))
    return np.array(rows, dtype=np.int64)
