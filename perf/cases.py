"""What this library is timed on: the passes its users make, over the sizes and options they make them with.

A pass goes through the public entry points only.  There are four kinds:
  step    a new trace arrives: load it, evaluate a policy grid on it, reduce, select (what bench.py calls a step);
  retune  the trace stays loaded and a new grid is evaluated on it: evaluate, reduce, select;
  shard   one request range of a larger trace, as each GPU of several does it: load, give the own tables out, take
          the whole trace's tables in, evaluate, export the accumulators, import the sum, reduce;
  sort    the allocation-free sort of one group's server TTFTs.

The distributions, endpoint profiles and grids are those of the library's workloads 0-5 (synth.py); traces are drawn on
the GPU so that a fresh one costs little.
"""
import math

import numpy as np
import torch

from paper_2502_11417_b200 import Trace, synth
from paper_2502_11417_b200.api import PAIR_FIELDS, policy_array, select_policy, sort_ttft_ticks_noalloc, stats_view

NOALLOC_MAX = 262144
PAIR_BYTES = 31               # the nine per-pair columns
STATS_BYTES = 152             # one policy's record
REQUEST_BYTES = 14            # prompt and output length, TTFT, two profile ids
SLO_S, CAP_FACTOR = 0.25, 1.25

# consumption rate (tokens/s) and estimated migration time (s): around the paper's reading pace first, then readers
# who outpace a phone's, a laptop's and finally the server's generation
PACES = [(5.0, 1.0), (4.0, 1.0), (8.0, 0.5), (12.0, 1.0), (20.0, 0.5), (30.0, 0.3)]
THETAS = [0.0, float("inf"), 0.05, 0.2, 0.02, 0.1, 0.4, 0.8]
MEAN_OUTPUT = {"chat": 200.0, "long": 830.0, "capped": 98.0}
GROUPS = {"fixed": 1, "basic": 1, "laptop": 1, "phone": 1, "mixed": 6, "paper": 6}


def _case(name, kind, n, fleet, outputs="chat", budgets=1, thetas=1, paces=1, rule="disco", inputs="device", rows=False,
          as_dicts=False):
    c = dict(kind=kind, n=n, fleet=fleet, outputs=outputs, budgets=budgets, thetas=thetas, paces=paces, rule=rule,
             inputs=inputs, rows=rows, as_dicts=as_dicts)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # one policy setting on a small trace held in ordinary numpy arrays, as in the README: all latency
        _case("one_policy_1k", "step", 1_000, "fixed", inputs="pageable", rows=True, as_dicts=True),
        # a budget curve with every pair written out for analysis (workload 1)
        _case("curve_100k_rows", "step", 100_000, "basic", budgets=64, rows=True),
        # budgets x migration thresholds on one commercial-API trace (workload 2)
        _case("grid_1m", "step", 1_000_000, "laptop", budgets=256, thetas=4),
        # long generations on a phone (workload 3)
        _case("long_4m", "step", 4_000_000, "phone", outputs="long", budgets=16),
        # the fleet: three server profiles, two devices, the full two-dimensional sweep (workload 4, bench.py's headline)
        _case("fleet_16m", "step", 16_000_000, "mixed", budgets=128, thetas=8),
        # the paper's phones, from page-locked host memory (workload 5, end to end)
        _case("phones_600k_pinned", "step", 600_000, "paper", outputs="capped", budgets=32, thetas=2, rule="expected",
              inputs="pinned"),
        # a day's ragged log from ordinary host arrays, a small grid
        _case("log_2m_pageable", "step", 1_999_993, "mixed", budgets=8, thetas=2, inputs="pageable"),
        # tuning against a loaded trace: several consumption rates at once, some faster than a device generates
        _case("retune_250k_paces", "retune", 250_007, "mixed", budgets=16, paces=5),
        # without the delivery buffer: tokens reach the reader as they are generated
        _case("unpaced_200k", "step", 200_000, "basic", budgets=32, rule="unpaced"),
        # the paper's baselines next to the method: random routing, the linear wait rule
        _case("baselines_300k", "step", 300_001, "mixed", budgets=16, rule="baselines"),
        # one of several GPUs' request ranges
        _case("shard_500k", "shard", 500_009, "mixed", budgets=32, thetas=2),
        # sorting without allocating, as between two launches of a serving loop
        _case("sort_100k", "sort", 100_003, "basic"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["step", "retune", "shard", "sort"], [7, 2, 1, 1])[0]
    if kind == "sort":
        return _case(None, "sort", _log_int(rng, 1_000, NOALLOC_MAX), "basic")
    fleet = rng.choice(["basic", "laptop", "phone", "mixed", "mixed", "paper"])
    outputs = "capped" if fleet == "paper" else rng.choice(["chat", "chat", "chat", "long"])
    rule = rng.choices(["disco", "unpaced", "baselines"], [8, 1, 1])[0]
    if fleet == "paper" and rule == "disco":
        rule = "expected"
    rows = kind == "step" and rng.random() < 0.25
    budgets = _log_int(rng, 1, 256 if rule in ("disco", "expected") else 32)
    thetas = rng.choice([1, 1, 2, 4, 8]) if rule in ("disco", "expected") else 1
    thetas = max(1, min(thetas, 1024 // budgets))
    paces = rng.choice([1, 1, 1, 2, 3, 5]) if kind == "retune" and rule in ("disco", "expected") and outputs != "long" else 1
    policies = budgets * thetas * paces * (3 if rule == "baselines" else 1)
    most = 16_000_000 if kind == "step" else 2_000_000
    if outputs == "long":
        most = min(most, 4_000_000)
    if rows:
        most = min(most, 8_000_000 // policies)
    if rule == "unpaced" or paces > 1:                   # every token of every stream counts
        most = min(most, int(400_000 * 200 / MEAN_OUTPUT[outputs]) // paces, 20_000_000 // policies)
    if rule == "baselines":                              # evaluated pair by pair
        most = min(most, 30_000_000 // policies)
    n = _log_int(rng, min(1_000, most), most)
    inputs = rng.choice(["device", "device", "pinned", "pageable"]) if kind == "step" else "device"
    return _case(None, kind, n, fleet, outputs, budgets, thetas, paces, rule, inputs, rows, as_dicts=policies <= 8)


def _lengths(gen, n, mu, sigma, lo, hi):
    z = torch.randn(n, generator=gen, device="cuda")
    return torch.exp(mu + sigma * z).round_().clamp_(lo, hi).to(torch.int32)


def _trace(case, gen, n):
    """Five trace columns of n requests on the GPU: prompt and output lengths, server TTFT, two profile ids."""
    fleet = case["fleet"]
    if fleet == "paper":
        prompt = _lengths(gen, n, 3.3, 0.8, 4, 512)
    else:
        prompt = _lengths(gen, n, 5.5, 1.0, 16, 4096)
    mu, sigma, lo, hi = {"chat": (5.0, 0.8, 8, 2048), "long": (6.5, 0.7, 64, 8192), "capped": (5.0, 0.8, 8, 128)}[case["outputs"]]
    output = _lengths(gen, n, mu, sigma, lo, hi)
    z = torch.randn(n, generator=gen, device="cuda")
    u = torch.rand(n, generator=gen, device="cuda")
    outlier = 5.0 + 10.0 * torch.rand(n, generator=gen, device="cuda")
    sp = torch.zeros(n, dtype=torch.uint8, device="cuda")
    dp = torch.zeros(n, dtype=torch.uint8, device="cuda")
    if fleet in ("fixed", "basic", "phone"):
        ttft = torch.exp(-1.0 + 0.6 * z)
        ttft = torch.where(u < 0.05, 4.0 * ttft, ttft)
    elif fleet in ("laptop", "paper"):
        ttft = torch.where(u < 0.02, outlier, torch.exp(-0.5 + 0.9 * z))
        if fleet == "paper":
            dp = torch.randint(0, 6, (n,), generator=gen, device="cuda", dtype=torch.uint8)
    else:
        sp = torch.randint(0, 3, (n,), generator=gen, device="cuda", dtype=torch.uint8)
        dp = torch.randint(0, 2, (n,), generator=gen, device="cuda", dtype=torch.uint8)
        k = sp.long()
        ttft = torch.exp(torch.tensor([-1.6, -0.5, 0.3], device="cuda")[k] + torch.tensor([0.3, 0.9, 1.1], device="cuda")[k] * z)
        ttft = torch.where((sp == 1) & (u < 0.02), outlier, ttft)
    return [prompt, output, ttft.clamp_(1e-3, 600.0), sp, dp]


def _endpoints(fleet):
    jitter_s, jitter_d = (0.0, 0.0) if fleet == "fixed" else (0.20, 0.05)
    if fleet == "paper":                                # the paper's three phones at two energy prices, GPT-4o-mini's prices
        phones = [(31.32, 13.93, 0.93, 0.82), (51.80, 20.14, 0.50, 0.42), (79.90, 21.47, 0.45, 0.37)]
        return ([synth.server(jitter=jitter_s, c_prefill=0.15e-6, c_decode=0.60e-6)],
                [synth.device(pf, dc, jitter=jitter_d, c_prefill=cp, c_decode=cd, lam=lam)
                 for lam in (0.3e-6, 5.0e-6) for pf, dc, cp, cd in phones])
    if fleet == "mixed":
        return ([synth.server(jitter=jitter_s) for _ in range(3)],
                [synth.device(1500.0, 40.0, jitter=jitter_d),
                 synth.device(200.0, 10.0, jitter=jitter_d, c_prefill=5.0e-3, c_decode=5.0e-3)])
    rates = {"laptop": (1500.0, 40.0), "phone": (200.0, 10.0)}.get(fleet, (500.0, 20.0))
    return [synth.server(jitter=jitter_s)], [synth.device(*rates, jitter=jitter_d)]


def _policies(case):
    grid = synth.budget_grid(case["budgets"])
    both = synth.FLAG_MIGRATION | synth.FLAG_PACING
    if case["rule"] == "unpaced":
        return [synth.policy(b, flags=synth.FLAG_MIGRATION) for b in grid]
    if case["rule"] == "baselines":
        return ([synth.policy(b, flags=both) for b in grid] +
                [synth.policy(b, flags=synth.FLAG_PACING | synth.FLAG_STOCHASTIC) for b in grid] +
                [synth.policy(b, flags=both | synth.FLAG_BETA_RULE, l_immediate=64) for b in grid])
    return [synth.policy(b, mig_threshold=th, r_c=rc, t_m_s=tm, expected_len=128 if case["rule"] == "expected" else 0)
            for rc, tm in PACES[:case["paces"]] for th in sorted(THETAS[:case["thetas"]]) for b in grid]


class State:
    pass


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    s = State()
    s.case, s.seed, n = case, int(seed), case["n"]
    if case["kind"] == "sort":
        s.ttft = _trace(case, gen, n)[2]
        s.ticks = torch.empty(n, dtype=torch.int32, device="cuda")
        return s
    columns = _trace(case, gen, n)
    if case["inputs"] == "pinned":
        columns = [c.cpu().pin_memory() for c in columns]
    elif case["inputs"] == "pageable":
        columns = [c.cpu().numpy() for c in columns]
    s.columns = columns
    s.servers, s.devices = _endpoints(case["fleet"])
    pols = _policies(case)
    s.policies = pols if case["as_dicts"] else policy_array(pols)
    s.trace = Trace()
    if case["kind"] == "retune":
        s.trace.load_trace(*columns, s.servers, s.devices)
    s.out = None
    if case["rows"]:
        s.out = {f: torch.empty((len(pols), n), dtype=getattr(torch, dt), device="cuda") for f, dt in PAIR_FIELDS}
    if case["kind"] == "shard":
        # what the other ranks' exchange brings: the tables of a further range of the same length
        other = Trace().load_trace(*_trace(case, gen, n), s.servers, s.devices, first_index=n)
        s.groups = other.n_groups
        s.other_cnt = [other.group_tables(g, 0)[0] for g in range(s.groups)]
        s.other_ticks = [other.sorted_ticks_device(g) for g in range(s.groups)]
        other.close()
        s.words = None
    return s


def _stats(stats):
    v = stats_view(stats)
    return {f: v[f] for f in v.dtype.names}


def run(s):
    kind = s.case["kind"]
    if kind == "sort":
        return sort_ttft_ticks_noalloc(s.ttft, s.ticks)
    tr = s.trace
    if kind == "shard":
        return _shard(s, tr)
    if kind == "step":
        tr.load_trace(*s.columns, s.servers, s.devices)
    tr.eval_policies(s.policies, s.seed, s.out)
    stats = tr.reduce_stats()
    status, best = select_policy(stats, CAP_FACTOR * float(stats_view(stats)["total_cost"].min()), SLO_S)
    result = {"stats": _stats(stats), "status": status, "best": best}
    if s.out is not None:                                # (unsigned columns as signed ones of the same width)
        signed = {torch.uint32: torch.int32, torch.uint16: torch.int16}
        result["pairs"] = {f: t.view(signed.get(t.dtype, t.dtype)) for f, t in s.out.items()}
    return result


def _shard(s, tr):
    tr.load_trace(*s.columns, s.servers, s.devices)
    cnt = np.stack([tr.group_tables(g, 0)[0] + s.other_cnt[g] for g in range(s.groups)])
    ticks = []
    for g in range(s.groups):
        ticks += [tr.sorted_ticks_device(g), s.other_ticks[g]]
    sizes = np.array([ticks[2 * g].numel() + ticks[2 * g + 1].numel() for g in range(s.groups)], dtype=np.uint64)
    tr.set_group_tables(cnt, torch.cat(ticks), sizes)
    tr.eval_policies(s.policies, s.seed)
    if s.words is None:
        s.words = torch.empty(tr.accumulator_words(), dtype=torch.int64, device="cuda")
    tr.export_accumulators(s.words)
    tr.import_accumulators(s.words)                      # (an all-reduce over the ranks lies between the two)
    return {"stats": _stats(tr.reduce_stats()), "words": s.words}


def work(case):
    n = case["n"]
    if case["kind"] == "sort":
        return {"bytes": 8 * n, "flops": 0}
    policies = len(_policies(case))
    total = STATS_BYTES * policies
    if case["kind"] == "retune":
        total += 9 * n                                   # a loaded request: ticks, two lengths, its group
    else:
        total += REQUEST_BYTES * n
    if case["rows"]:
        total += PAIR_BYTES * n * policies
    if case["kind"] == "shard":                          # the whole trace's ticks in, the accumulator words out and in
        total += 2 * 4 * n + 2 * 8 * policies * (GROUPS[case["fleet"]] * 12 + 2 * 864)
    # integer operations: about thirteen per token that has to be drawn (the hash, a range map, a sum).  With paced
    # delivery and generation that keeps up these are the tokens up to the hand-off, once the buffer is full; otherwise
    # every token of both streams.  Plus a dozen per request for dispatch and race.
    tokens = 10.0
    if case["rule"] == "unpaced":
        tokens = 2 * MEAN_OUTPUT[case["outputs"]]
    elif case["paces"] > 3:
        tokens = 10.0 * 3 + 2 * MEAN_OUTPUT[case["outputs"]] * (case["paces"] - 3)
    return {"bytes": total, "flops": n * (13 * tokens + 12)}


def tolerance(case):
    # times are whole ticks throughout, so counts, token totals, histogram bins and sorted ticks stay the same; the
    # per-pair columns are 32-bit floats, means and costs in 64 bits are formed from exact integer totals
    return "exact" if case["kind"] == "sort" else {"rel": 1e-6, "max": 1e-5}
