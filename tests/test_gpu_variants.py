"""Variants of the kernels that the library chooses by sizes and types: parity with the oracle where each one's range
begins and ends."""
import numpy as np
import pytest

from paper_2502_11417_b200 import synth
from parity import full_parity

pytestmark = pytest.mark.gpu

PACED = synth.FLAG_MIGRATION | synth.FLAG_PACING


@pytest.mark.parametrize("n", [1, 255, 257, 3000])
@pytest.mark.parametrize("buffer_tokens", [0, 1, 2, 11, 12, 200])
def test_handoff_search_by_one_thread_and_by_a_warp(n, buffer_tokens):
    # 20 tokens/s consumption against a server whose slowest token takes 42 ms: every token gains 8 ms or more, so the
    # search looks at (buffer - 1) * 50 / 8 + 1 tokens (64 is the last that one thread takes); a device generates at 40/s
    w = synth.tiny_workload(7 + n, n, max_prompt=300, max_out=500)
    w.servers = [synth.server(tbt_s=0.035, jitter=0.2)]
    w.devices = [synth.device(500.0, 40.0, jitter=0.05)]
    dear = [synth.device(500.0, 40.0, jitter=0.05, c_prefill=5e-3, c_decode=5e-3)]
    for devices in (w.devices, dear):
        w.devices = devices
        full_parity(w, [synth.policy(b, r_c=20.0, t_m_s=buffer_tokens * 0.05, mig_threshold=th, flags=PACED)
                        for b in (0.3, 1.0) for th in (0.0, 0.1)], select=False, tag=f"search {buffer_tokens}")


def _sample(kind, n, rng):
    if kind == "spread":                       # windows of many bins, up to the largest TTFT
        return np.exp(rng.uniform(np.log(1e-6), np.log(2000.0), n))
    if kind == "ties":                         # one value, and another in every sixteenth place
        return np.where(np.arange(n) % 16 == 3, 0.5, 600.0)
    if kind == "dense":                        # bins of more than 8,192 ticks spread over few values: counted
        return np.round(0.25 + 0.004 * rng.random(n), 6)
    if kind == "often":                        # ... a few of them very often
        return np.where(rng.random(n) < 0.9, 0.25, 0.25 + 1e-6 * rng.integers(0, 900, n))
    if kind == "few":                          # ... two in one bin, one in another
        return np.where(rng.random(n) < 0.4, 0.5, 0.25 + 1e-6 * rng.integers(0, 2, n))
    return 1000.0 + 100.0 * rng.random(n)      # "wide": bins of more than 8,192 ticks and 2^18 values: the radix sort


@pytest.mark.parametrize("kind", ["spread", "ties", "dense", "often", "few", "wide"])
@pytest.mark.parametrize("n", [1, 33, 4096, 4097, 8193, 70001, 260000])
def test_sorted_samples(kind, n):
    import torch
    from paper_2502_11417_b200 import Trace
    from paper_2502_11417_b200.api import sort_ttft_ticks_noalloc
    rng = np.random.default_rng(n)
    x = np.clip(_sample(kind, n, rng), 1e-6, 2000.0).astype(np.float32)
    ticks = np.rint(x.astype(np.float64) * 1e6).astype(np.int64)
    want = np.sort(ticks)
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    assert (sort_ttft_ticks_noalloc(torch.from_numpy(x).cuda(), out).cpu().numpy() == want).all()
    # two groups, loaded; then imported as a whole trace's tables would be
    dp = (np.arange(n) % 3 == 0).astype(np.uint8)
    devices = [synth.device(500.0, 20.0), synth.device(400.0, 20.0)]
    tr = Trace().load_trace(np.full(n, 7, np.int32), np.full(n, 5, np.int32), x, None, dp, [synth.server()], devices)
    groups = [ticks[dp == 0], ticks[dp == 1]]
    for _ in range(2):
        for g in range(2):
            cnt, knots, got = tr.group_tables(g)
            srt = np.sort(groups[g])
            assert got.shape == srt.shape and (got == srt).all()
            if len(srt):
                assert (knots == srt[np.arange(257, dtype=np.int64) * (len(srt) - 1) // 256]).all() and cnt[7] == len(srt)
        lengths = np.zeros((2, 4097), dtype=np.int64)
        lengths[:, 7] = [len(g) for g in groups]
        tr.set_group_tables(lengths, np.concatenate(groups).astype(np.int32), lengths[:, 7].astype(np.uint64))
    tr.close()


@pytest.mark.parametrize("shape", [(1, 7), (2, 4), (4, 5)])
@pytest.mark.parametrize("where", ["host", "pinned"])
def test_groups_whose_counters_fit_a_block_or_do_not(shape, where):
    import torch
    w = synth.tiny_workload(91, 5003, n_servers=shape[0], n_devices=shape[1], max_prompt=4096, max_out=60)
    if where == "pinned":
        for f in ("prompt_len", "output_len", "server_ttft_s", "server_profile", "device_profile"):
            setattr(w, f, torch.from_numpy(getattr(w, f)).pin_memory().numpy())
    full_parity(w, [synth.policy(b) for b in synth.budget_grid(9)], tag=f"{shape} groups")


@pytest.mark.parametrize("kind", ["spread", "ties", "dense", "wide"])
@pytest.mark.parametrize("n", [1, 2, 700, 40000])
def test_linear_wait_rule_on_samples(kind, n):
    # the slope of Eq. 1-2 is searched between positions in the sorted ticks: one tick, equal ticks, crowded bins
    rng = np.random.default_rng(n + 5)
    w = synth.tiny_workload(95, n, max_prompt=4096, max_out=20, device_dearer=True)
    w.server_ttft_s = np.clip(_sample(kind, n, rng) / (4.0 if kind == "wide" else 1.0), 1e-6, 500.0).astype(np.float32)
    flags = PACED | synth.FLAG_BETA_RULE | synth.MODE_DEVICE_CONSTRAINED
    pols = [synth.policy(b, flags=flags, l_immediate=li) for b in (0.0, 0.06, 0.3, 0.9, 1.0) for li in (0, 100, 4096)]
    if n <= 700:
        full_parity(w, pols, select=False, tag=f"{kind} {n}")
        return
    from oracle import Oracle
    from paper_2502_11417_b200 import Trace
    from parity import check_prep
    tr = Trace.from_workload(w)
    tr.eval_policies(pols, 1)
    check_prep(tr, Oracle.from_workload(w), pols, f"{kind} {n}")
    tr.close()


@pytest.mark.parametrize("n", [15, 8192, 8193, 32768, 32785, 70001, 1_200_003])
@pytest.mark.parametrize("profiles", ["both", "server", "device", "none"])
def test_pageable_traces_are_packed(n, profiles):
    # ordinary host arrays go to the device packed, chunk by chunk: the same tables and statistics as from device memory;
    # a value out of range is refused wherever it lies
    import torch
    from paper_2502_11417_b200 import DiscoError, Trace
    w = synth.tiny_workload(97, n, n_servers=3, n_devices=2, max_prompt=4096, max_out=30)
    sp = w.server_profile if profiles in ("both", "server") else None
    dp = w.device_profile if profiles in ("both", "device") else None
    cols = [w.prompt_len, w.output_len, w.server_ttft_s, sp, dp]
    dev = [None if c is None else torch.from_numpy(c).cuda() for c in cols]
    got = []
    for c in (cols, dev):
        tr = Trace().load_trace(*c, w.servers, w.devices)
        tr.eval_policies([synth.policy(0.4)], 3)
        got.append((bytes(tr.reduce_stats()), [t.tobytes() for g in range(tr.n_groups) for t in tr.group_tables(g)]))
        tr.close()
    assert got[0] == got[1]
    for k, bad in ((0, 4097), (0, 0), (1, 8193), (1, -1), (2, 0.0), (3, 3), (4, 2)):
        if cols[k] is None:
            continue
        at = (n * 2) // 3
        wrong = [None if c is None else c.copy() for c in cols]
        wrong[k][at] = bad
        with pytest.raises(DiscoError) as ei:
            Trace().load_trace(*wrong, w.servers, w.devices)
        assert ei.value.code == -1 and f"at request {at}" in str(ei.value)


@pytest.mark.parametrize("dearer", [False, True])
@pytest.mark.parametrize("n,budgets", [(1, 256), (31, 257), (700, 64), (700, 5), (5003, 256), (5003, 33)])
def test_few_requests_to_a_run(n, budgets, dearer):
    # small chunks under many thresholds are entered request by request, others run by run: both against the oracle, with
    # one overhead and with three, under Algorithm 2 (the device dearer) and 3
    w = synth.tiny_workload(99, n, n_servers=2, max_prompt=4096, max_out=60, device_dearer=dearer)
    grid = synth.budget_grid(budgets)
    full_parity(w, [synth.policy(b) for b in grid], select=False, tag=f"{n} {budgets}")
    full_parity(w, [synth.policy(b, mig_threshold=t) for b in grid[::3] for t in (0.0, 1e-6, 3e-5)], select=False,
                tag=f"{n} {budgets} x 3")


@pytest.mark.parametrize("dearer", [False, True])
@pytest.mark.parametrize("n", [257, 9000, 20011])
def test_eight_overheads(n, dearer):
    # the kernel of eight rows loads an iteration ahead, and runs are entered by the groups of bins they have counts in:
    # sweeps of a part of a block, of a whole one and of several, with budgets below the tail ratio (lists) under Algorithm 2
    w = synth.tiny_workload(101, n, max_prompt=64, max_out=60, device_dearer=dearer)
    thetas = (0.0, 1e-7, 1e-6, 4e-6, 1e-5, 3e-5, 1e-4, 1.0)
    full_parity(w, [synth.policy(b, mig_threshold=t) for b in (0.0, 0.01, 0.03, 0.4, 0.8) for t in thetas], select=False, tag=f"{n}")


@pytest.mark.parametrize("dearer", [False, True])
@pytest.mark.parametrize("overheads", [3, 4, 5, 8])
@pytest.mark.parametrize("n", [257, 9000])
def test_windows_under_several_overheads(n, overheads, dearer):
    # streams whose intervals are not all tau take their windows to every row of the grid, and the rows that migrate take
    # them back: without pacing, with a device slower than the reader, with either endpoint slower at times; and, for
    # comparison, even streams.  The overheads lie between the requests' savings: every level has some.
    w = synth.tiny_workload(103, n, max_prompt=64, max_out=60, device_dearer=dearer)
    thetas = (0.0, 0.004, 0.012, 0.02, 0.03, 0.06, 0.12, 1.0)[:overheads]
    grid = [(b, t) for b in (0.0, 0.01, 0.03, 0.4, 0.8) for t in thetas]
    for how in (dict(flags=synth.FLAG_MIGRATION), dict(r_c=25.0, t_m_s=0.2), dict(r_c=30.0, t_m_s=0.3), dict(t_m_s=0.4)):
        full_parity(w, [synth.policy(b, mig_threshold=t, **how) for b, t in grid], select=False, tag=f"{n} x {overheads} {how}")


@pytest.mark.parametrize("n,shape,kind,where", [(3_499_999, (1, 1), "spread", "device"), (3_500_000, (1, 1), "spread", "device"),
                                                (3_500_001, (1, 1), "one", "device"), (3_508_193, (3, 2), "spread", "pinned"),
                                                (3_600_013, (1, 7), "ties", "pageable"), (3_600_013, (2, 2), "dense", "unaligned"),
                                                (4_000_003, (1, 2), "wide", "device"), (3_600_013, (2, 4), "spread", "device"),
                                                (2 ** 24 + 17, (3, 2), "spread", "device")])
def test_large_traces_are_placed_by_way_of_buckets(n, shape, kind, where):
    # tables and statistics of traces from 3.5 M requests in up to seven groups on, and on the other side of both limits: full
    # and partly filled tiles and buckets, lengths and bins that take a bucket to themselves, samples left to the radix sort; beyond
    # 2^24 requests k_load places them in rounds
    import torch
    from oracle import Oracle
    from paper_2502_11417_b200 import DiscoError, Trace
    from parity import check_stats
    rng = np.random.default_rng(n)
    w = synth.tiny_workload(105, n, n_servers=shape[0], n_devices=shape[1], max_prompt=4096, max_out=6)
    if kind == "one":                              # one prompt length, one TTFT
        w.prompt_len[:] = 77
        w.server_ttft_s[:] = 0.25
    elif kind != "spread":
        w.server_ttft_s = np.clip(_sample(kind, n, rng), 1e-6, 2000.0).astype(np.float32)
        w.prompt_len[rng.random(n) < 0.3] = 900    # (more than a bucket's share)
    cols = [w.prompt_len, w.output_len, w.server_ttft_s, w.server_profile, w.device_profile]
    if where == "pinned":
        cols = [torch.from_numpy(c).pin_memory() for c in cols]
    elif where == "device":
        cols = [torch.from_numpy(c).cuda() for c in cols]
    elif where == "unaligned":
        cols = [torch.cat([torch.from_numpy(c[:1]), torch.from_numpy(c)]).cuda()[1:] for c in cols]
    tr = Trace()
    with pytest.raises(DiscoError) as ei:
        bad = w.output_len.copy()
        bad[n - 2] = 0
        tr.load_trace(w.prompt_len, bad, *[np.asarray(c) for c in (w.server_ttft_s, w.server_profile, w.device_profile)], w.servers, w.devices)
    assert f"at request {n - 2}" in str(ei.value)
    tr.load_trace(*cols, w.servers, w.devices)
    g_of = w.server_profile.astype(np.int64) * shape[1] + w.device_profile
    ticks = np.rint(w.server_ttft_s.astype(np.float64) * 1e6).astype(np.int64)
    for g in range(shape[0] * shape[1]):
        cnt, knots, srt = tr.group_tables(g)
        want = np.sort(ticks[g_of == g])
        assert (srt == want).all() and (cnt == np.bincount(w.prompt_len[g_of == g], minlength=4097)).all()
        assert (knots == want[np.arange(257, dtype=np.int64) * (len(want) - 1) // 256]).all()
    pols = [synth.policy(0.4)]
    if kind in ("spread", "one") and shape[0] * shape[1] in (1, 6):
        orc = Oracle.from_workload(w)
        out = tr.alloc_pair_outputs(1, ["ttft_s", "tok_server"])       # (rows: the requests' places are looked up)
        tr.eval_policies(pols, w.seed, out)
        stats, pairs = orc.eval(pols, w.seed, pairs=True)
        check_stats(tr.reduce_stats(), stats, tr.histograms, f"{n}")
        assert (out["tok_server"].cpu().numpy() == pairs["tok_server"]).all()
        assert np.allclose(out["ttft_s"].cpu().numpy(), pairs["ttft_s"], rtol=1e-6)
    tr.close()


def _crowded(kind, n, rng):
    x = np.exp(rng.normal(-0.5, 0.9, n))
    if kind == "pairs":                        # two neighbouring microseconds, thousands of each, in bins 8,192 and more wide
        at = (2 ** 20 * 2 ** (rng.permutation(3 * 128)[:300] / 128.0) + rng.integers(0, 4000, 300)).astype(np.int64)
        ticks = at[rng.integers(0, 300, n)] + rng.integers(0, 2, n)
        return np.where(rng.random(n) < 0.3, ticks * 1e-6, x)
    if kind == "two":
        return 0.25 + 1e-6 * rng.integers(0, 2, n)
    if kind == "narrow":
        return 0.25 + 0.004 * rng.random(n)
    step = {"1ms": 1e-3, "10ms": 1e-2, "0.1ms": 1e-4}[kind]
    return np.maximum(np.rint(x / step), 1) * step


@pytest.mark.parametrize("n,shape,kind", [(3_500_000, (1, 1), "1ms"), (3_500_000, (3, 2), "two"), (3_500_000, (3, 2), "narrow"), (4_000_003, (3, 2), "1ms"), (4_000_003, (1, 1), "10ms"), (4_000_003, (3, 2), "10ms"),
                                          (4_000_003, (1, 1), "0.1ms"), (4_000_003, (1, 1), "pairs"), (4_000_003, (1, 2), "pairs"), (16_000_000, (1, 1), "1ms"),
                                          (16_000_000, (3, 2), "10ms")])
def test_large_traces_by_a_coarse_clock(n, shape, kind):
    # buckets of ticks in which hundreds are equal, or take a few neighbouring values, and bins of one value or a few, very often: sorted
    # where they are, without further launches
    import torch
    from paper_2502_11417_b200 import Trace, api
    rng = np.random.default_rng(n + len(kind))
    x = np.clip(_crowded(kind, n, rng), 1e-6, 2000.0).astype(np.float32)
    g_of = rng.integers(0, shape[0] * shape[1], n).astype(np.uint8)
    cols = [np.full(n, 7, np.int32), np.full(n, 5, np.int32), x, g_of // shape[1], g_of % shape[1]]
    dev = [torch.from_numpy(c).cuda() for c in cols]
    ticks = np.rint(x.astype(np.float64) * 1e6).astype(np.int64)
    tr = Trace()
    before = api.lib().disco_kernel_launch_count()
    tr.load_trace(*dev, [synth.server()] * shape[0], [synth.device(500.0, 20.0)] * shape[1])
    assert api.lib().disco_kernel_launch_count() == before + 6
    for g in range(tr.n_groups):
        want = np.sort(ticks[g_of == g])
        cnt, knots, got = tr.group_tables(g)
        assert (got == want).all() and cnt[7] == len(want)
        assert (knots == want[np.arange(257, dtype=np.int64) * (len(want) - 1) // 256]).all()
    tr.close()


@pytest.mark.parametrize("shape", [(1, 1), (2, 3), (8, 8)])
@pytest.mark.parametrize("n", [1, 255, 257, 1500])
def test_rows_of_several_groups(n, shape):
    # a block writes the rows of neighbouring requests of any groups, with the rules of up to 16 policies for each: a partly
    # filled block and row of policies, up to 64 groups, with random routing and expected lengths among them and without
    w = synth.tiny_workload(107, n, n_servers=shape[0], n_devices=shape[1], max_prompt=300, max_out=60)
    plain = [synth.policy(b, mig_threshold=1e-6 * k) for k, b in enumerate(synth.budget_grid(17))]
    full_parity(w, plain, select=False, tag=f"{n} {shape}")
    full_parity(w, plain[:3] + [synth.policy(0.5, flags=PACED | synth.FLAG_STOCHASTIC), synth.policy(0.3, expected_len=20)], select=False, tag=f"{n} {shape} extras")


@pytest.mark.parametrize("n_policies", [1, 5, 31, 32, 150, 160, 400, 900])
@pytest.mark.parametrize("beta", [False, True])
def test_tables_of_the_policies_on_their_way(n_policies, beta):
    # the small tables go with a launch in one of three sizes, or lie in page-locked memory; evaluations follow each other without
    # a wait in between, so that the host must not write what a kernel has yet to read
    import torch
    from oracle import Oracle
    from paper_2502_11417_b200 import Trace
    from parity import check_prep, check_stats
    w = synth.tiny_workload(109, 700, n_servers=2, n_devices=2, max_prompt=300, max_out=40)
    rule = PACED | (synth.FLAG_BETA_RULE if beta else 0)
    pols = [synth.policy(b, flags=rule if k % 3 == 0 else PACED, mig_threshold=1e-6 * (k % 2)) for k, b in enumerate(synth.budget_grid(n_policies))]
    other = [synth.policy(0.9 - 0.001 * (k % 7), alpha=0.2) for k in range(n_policies)]
    orc, tr = Oracle.from_workload(w), Trace.from_workload(w)
    x = torch.randn(2048, 2048, device="cuda")
    for _ in range(20):                            # (work in front: the evaluations below queue up behind it)
        x = torch.tanh(x @ x)
    for _ in range(3):
        tr.eval_policies(other, 5)
    tr.eval_policies(pols, w.seed)
    stats = tr.reduce_stats()
    check_stats(stats, orc.eval(pols, w.seed)[0], tr.histograms, f"{n_policies}")
    check_prep(tr, orc, pols, f"{n_policies}")
    tr.close()


@pytest.mark.parametrize("n", [1, 300, 4000])
@pytest.mark.parametrize("rates", [(12.0, 20.0), (20.0, 5.0, 12.0), (5.0, 30.0, 12.0, 4.0, 20.0, 11.0), (12.0, 33.0, 20.0), tuple(12.0 + 0.4 * k for k in range(12)),
                                   tuple(3.0 + 0.2 * k for k in range(20))])
def test_classes_that_are_reduced_together(n, rates):
    # a slow device whose streams are delivered as they are generated at most of these rates, beside a server and a device that keep
    # the pace at some: such streams are played once for several classes (up to nine), classes without windows share a launch, sixteen
    # play-outs up to the hand-off do, and classes of any kind lie between them
    w = synth.tiny_workload(113 + n, n, n_servers=2, n_devices=2, max_prompt=300, max_out=200)
    w.servers = [synth.server(tbt_s=0.03, jitter=0.2), synth.server(tbt_s=0.03, jitter=0.0)]
    w.devices = [synth.device(1500.0, 40.0, jitter=0.05), synth.device(200.0, 10.0, jitter=0.05, c_prefill=5e-3, c_decode=5e-3)]
    pols = [synth.policy(b, r_c=r, t_m_s=0.5, mig_threshold=th, flags=PACED) for r in rates for b in (0.2, 0.7) for th in (0.0, 0.01)]
    full_parity(w, pols, select=False, tag=f"{rates}")
    more = [synth.policy(0.4, r_c=rates[0], flags=synth.FLAG_MIGRATION), synth.policy(0.4, r_c=rates[-1], flags=PACED | synth.FLAG_STOCHASTIC),
            synth.policy(0.6, r_c=rates[-1], flags=synth.FLAG_PACING), synth.policy(0.6, r_c=rates[1], flags=PACED | synth.FLAG_BETA_RULE, l_immediate=64)]
    full_parity(w, pols[::-1] + more, select=False, tag=f"{rates} and others")


@pytest.mark.parametrize("n", [1, 3, 9000, 30001])
@pytest.mark.parametrize("jitter", [0.0, 0.2])
@pytest.mark.parametrize("rate", [None, 12.0, 40.0])
def test_streams_delivered_as_they_are_generated(n, jitter, rate):
    # without pacing, with a slow device beside a server that keeps the pace, and with both endpoints slower than the reader or one of
    # them by groups: batches of two requests and more, partly filled, groups that are not played here between others
    w = synth.tiny_workload(127 + n, n, n_servers=2, n_devices=2, max_prompt=200, max_out=70)
    w.output_len[::17] = 900                       # (several rounds of a warp)
    w.servers = [synth.server(tbt_s=0.03, jitter=jitter), synth.server(tbt_s=0.045, jitter=jitter / 4)]
    w.devices = [synth.device(1500.0, 40.0, jitter=0.05), synth.device(200.0, 10.0, jitter=jitter / 2, c_prefill=5e-3, c_decode=5e-3)]
    flags = synth.FLAG_MIGRATION | (synth.FLAG_PACING if rate else 0)
    full_parity(w, [synth.policy(b, r_c=rate or 5.0, flags=flags) for b in (0.3, 0.8)], select=False, tag=f"{n} {jitter} {rate}")


@pytest.mark.parametrize("n", [1, 700, 20001])
@pytest.mark.parametrize("shape", [(1, 1), (3, 2)])
@pytest.mark.parametrize("plain", [0, 1, 9])
def test_grids_beside_the_slope_search(n, shape, plain):
    # plain policies are reduced while the slopes of the others are searched for: no plain ones, one, several rows, a column a policy
    # with overheads of its own, and searches that outlast or do not outlast the grid
    w = synth.tiny_workload(131 + n, n, n_servers=shape[0], n_devices=shape[1], max_prompt=2000, max_out=40)
    slopes = [synth.policy(b, flags=PACED | synth.FLAG_BETA_RULE | synth.MODE_DEVICE_CONSTRAINED, l_immediate=64) for b in (0.2, 0.5, 0.9)]
    rows = [synth.policy(b, mig_threshold=th) for b in synth.budget_grid(plain) for th in (0.0, 1e-5)]
    full_parity(w, slopes + rows, select=False, tag=f"{n} {shape} {plain}")
    full_parity(w, slopes[:1] + [synth.policy(b, mig_threshold=1e-6 * k) for k, b in enumerate(synth.budget_grid(plain))], select=False, tag="columns")


@pytest.mark.parametrize("n", [2, 1023, 1025, 5000])
@pytest.mark.parametrize("tbt", [0.0, 0.01, 0.0499, 0.05])
def test_tokens_that_are_certain_not_to_decide(n, tbt):
    # the tokens in front of the first that can fill a buffer or make a lag up are added up without a test: without jitter, where that
    # is all but the last, an interval of the reader's own pace, where none does, outputs that end among them, lags of one tick
    w = synth.tiny_workload(137 + n, n, n_servers=2, n_devices=2, max_prompt=1500, max_out=40)
    w.output_len[::5] = np.arange(len(w.output_len[::5])) % 9 + 1
    w.output_len[3::11] = 700
    w.servers = [synth.server(tbt_s=max(tbt, 1e-6), jitter=0.0), synth.server(tbt_s=0.04, jitter=0.2)]
    w.devices = [synth.device(20.0, 1.0 / max(tbt, 1e-6), jitter=0.0), synth.device(300.0, 25.0, jitter=0.2, c_prefill=5e-3, c_decode=5e-3)]
    full_parity(w, [synth.policy(b, r_c=20.0, t_m_s=t, flags=PACED) for b in (0.4, 1.0) for t in (0.05, 0.1, 0.4)], select=False, tag=f"{n} {tbt}")


@pytest.mark.parametrize("policies", [64, 2048])
def test_evaluations_in_a_row_wait_for_no_other_stream(policies):
    # beyond some 930 policies (of a budget each: 28 KB) their tables are read from page-locked memory, which the next evaluation writes again
    import torch
    from paper_2502_11417_b200 import Trace
    w = synth.tiny_workload(3, 5000)
    pols = [[synth.policy(top * k / (policies - 1)) for k in range(policies)] for top in (1.0, 0.5)]
    mine, other, done = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Event()
    t = Trace.from_workload(w, stream=mine)
    with torch.cuda.stream(mine):
        want = []
        for p in pols:
            t.eval_policies(p, 1)
            want.append([bytes(s) for s in t.reduce_stats()])
        with torch.cuda.stream(other):
            torch.cuda._sleep(1_000_000_000)                   # about half a second
            done.record()
        torch.cuda._sleep(20_000_000)                          # (the first evaluation's tables have not been read when the next one comes)
        for turn in range(8):
            t.eval_policies(pols[turn % 2], 1)
        got = [bytes(s) for s in t.reduce_stats()]
        assert not done.query()
        assert got == want[1] and got != want[0]
    done.synchronize()


@pytest.mark.parametrize("n", [1, 129, 700, 20001, 1_300_001])
@pytest.mark.parametrize("tbt", [0.03, 0.1999, 0.2])
def test_lags_behind_a_handoff_to_the_server(n, tbt):
    # many lags of a block are put in order by their lengths before they are made up: lags as widely spread as the server's TTFT, of no
    # token and of all that are left, intervals that make up hardly anything or nothing of them; a request a thread, and four
    w = synth.tiny_workload(139 + n, n, n_servers=2, max_prompt=300, max_out=500, device_dearer=True)
    w.server_ttft_s = np.clip(np.exp(np.random.default_rng(n).normal(0.0, 1.5, n)), 1e-3, 100.0).astype(np.float32)
    w.servers = [synth.server(jitter=0.2), synth.server(tbt_s=tbt, jitter=0.0)]
    pols = [synth.policy(b, flags=PACED) for b in (0.3, 1.0)]
    if n <= 20001:
        full_parity(w, pols, select=False, tag=f"{n} {tbt}")
        return
    from oracle import Oracle
    from paper_2502_11417_b200 import Trace
    from parity import check_stats
    tr = Trace.from_workload(w)
    tr.eval_policies(pols[1:], w.seed)
    check_stats(tr.reduce_stats(), Oracle.from_workload(w).eval(pols[1:], w.seed)[0], tr.histograms, f"{n} {tbt}")
    tr.close()


@pytest.mark.parametrize("n", [(1 << 20) - 1, 1 << 20, (1 << 20) + 1])
@pytest.mark.parametrize("lengths", [1, 900, 4096])
def test_linear_wait_rule_of_many_requests(n, lengths):
    # the slope search multiplies in 32 bits below 2^20 requests of a group, and takes the prompt lengths that occur
    from oracle import Oracle
    from paper_2502_11417_b200 import Trace
    from parity import check_prep
    w = synth.tiny_workload(149, n, max_prompt=lengths, max_out=4, device_dearer=True)
    w.prompt_len[:3] = 4096                        # (tokens of a length close to 2^32 where all but these have one)
    if lengths == 1:
        w.prompt_len[3:] = 4095
    pols = [synth.policy(b, flags=PACED | synth.FLAG_BETA_RULE | synth.MODE_DEVICE_CONSTRAINED, l_immediate=li) for b in (0.06, 0.5, 1.0) for li in (0, 100)]
    tr = Trace.from_workload(w)
    tr.eval_policies(pols, 1)
    check_prep(tr, Oracle.from_workload(w), pols, f"{n} {lengths}")
    tr.close()


@pytest.mark.parametrize("kinds", [1, 16, 17, 64, 65, 700])
def test_policies_of_many_kinds(kinds):
    # what policies share goes to the preparation once: kinds that come back, more of them than are looked up or lie close at hand,
    # with the launch and in page-locked memory
    w = synth.tiny_workload(151, 300, n_servers=2, max_prompt=300, max_out=30, device_dearer=True)
    pols = [synth.policy(0.001 * (k % 997), alpha=0.01 + 0.001 * (k % kinds), expected_len=k % 2 * 20) for k in range(max(kinds, 3))]
    full_parity(w, pols + pols[::2], select=False, tag=f"{kinds}")


@pytest.mark.parametrize("n", [5000, 30_001, 60_001])
@pytest.mark.parametrize("shape", [(1, 1), (2, 3)])
def test_narrow_grids_beside_wide_ones(n, shape):
    # a wide grid goes side by side, narrow ones run by run, and between them one whose overheads differ by budget (either): all in one
    # evaluation, with chunks of their own
    w = synth.tiny_workload(179 + n, n, n_servers=shape[0], n_devices=shape[1], max_prompt=700, max_out=40, device_dearer=True)
    of = lambda columns, rows, E: [synth.policy(b, flags=PACED, mig_threshold=1e-6 * k, expected_len=E) for b in synth.budget_grid(columns) for k in range(rows)]
    by_budget = [synth.policy(b, flags=PACED, mig_threshold=1e-6 * k, expected_len=3) for k, b in enumerate(synth.budget_grid(9))]
    full_parity(w, of(2, 1, 5) + of(48, 1, 0) + by_budget + of(2, 3, 7) + of(20, 3, 9) + of(1, 1, 11), select=False, tag=f"{n} {shape}")


@pytest.mark.parametrize("rate", [5.0, 40.0])
@pytest.mark.parametrize("rows", [1, 2])
def test_lists_that_fill_within_a_segment(rate, rows):
    # Algorithm 2 with a tail ratio so large that most requests of a segment wait longer in its first columns than the common wait
    # covers: chunks of some 4,800 requests and a few prompt lengths, whose lists are added to by run after run, fill and begin anew;
    # without windows and (a reader faster than either endpoint) with
    from oracle import Oracle
    from paper_2502_11417_b200 import Trace
    from parity import check_stats
    n = 1_400_001
    w = synth.tiny_workload(173, n, max_prompt=4, max_out=6, device_dearer=True)
    pols = [synth.policy(b, alpha=a, r_c=rate, flags=PACED, mig_threshold=1e-3 * k) for a in (0.55, 0.6, 0.65, 0.7) for b in (0.2, 0.5, 0.9) for k in range(rows)]
    tr = Trace.from_workload(w)
    tr.eval_policies(pols, w.seed)
    check_stats(tr.reduce_stats(), Oracle.from_workload(w).eval(pols, w.seed)[0], tr.histograms, f"{rate} {rows}")
    tr.close()


def test_evaluations_in_a_row_of_many_kinds():
    # Tables read from page-locked memory, with more kinds than a block of the preparation keeps: the call behind writes that memory
    # again (or gives it back for a larger piece) as soon as the last of it has been read.  Nothing is waited for between the calls.
    import torch
    from oracle import Oracle
    from paper_2502_11417_b200 import Trace
    from paper_2502_11417_b200.api import policy_array
    from parity import check_pairs, check_stats
    w = synth.tiny_workload(167, 300, n_servers=2, n_devices=3, max_prompt=300, max_out=30, device_dearer=True)
    t, orc = Trace.from_workload(w), Oracle.from_workload(w)
    cnt = np.stack([t.group_tables(g)[0] for g in range(t.n_groups)])
    ticks = torch.cat([t.sorted_ticks_device(g) for g in range(t.n_groups)])
    sizes = cnt.sum(axis=1).astype(np.uint64)
    kind = lambda k, e: dict(alpha=0.01 + 0.007 * ((k * (3 + 2 * e)) % 131), expected_len=(k + e) % 2 * 20)
    sets = [[synth.policy(0.001 * ((k * 7 + e) % 997), **kind(k, e)) for k in range(n)][::1 - 2 * (e % 2)] for e, n in enumerate([900, 700, 1300, 900, 1800, 1000])]
    arrays, outs = [policy_array(p) for p in sets], [t.alloc_pair_outputs(len(p)) for p in sets]
    again = [t.alloc_pair_outputs(len(p)) for p in sets]
    for tables in (False, True):
        torch.cuda.synchronize()
        for a, o in zip(arrays, again if tables else outs):
            t.eval_policies(a, w.seed, o)
            if tables:
                t.set_group_tables(cnt, ticks, sizes)
    t.eval_policies(arrays[-1], w.seed)
    stats = t.reduce_stats()
    for e, p in enumerate(sets):
        want, pairs = orc.eval(p, w.seed, pairs=True)
        check_pairs(outs[e], pairs, tag=f"evaluation {e}")
        check_pairs(again[e], pairs, tag=f"evaluation {e} in front of tables")
    check_stats(stats, want, t.histograms, "the last")
    t.close()


@pytest.mark.parametrize("n", [1, 256, 148 * 256, 148 * 256 + 1, 100_001])
@pytest.mark.parametrize("shape,policies", [((1, 1), 3), ((2, 3), 33), ((3, 3), 200)])
def test_pairs_in_whole_rounds_of_blocks(n, shape, policies):
    # policies with random routing take the pair kernel: a request to a multiprocessor's thread or one more, several tiles of
    # policies, and more groups times tiles than a round has blocks
    from oracle import Oracle
    from paper_2502_11417_b200 import Trace
    from parity import check_stats
    w = synth.tiny_workload(157, n, n_servers=shape[0], n_devices=shape[1], max_prompt=300, max_out=30)
    pols = [synth.policy(b, mig_threshold=1e-6 * (k % 2), flags=PACED | synth.FLAG_STOCHASTIC) for k, b in enumerate(synth.budget_grid(policies))]
    tr = Trace.from_workload(w)
    tr.eval_policies(pols, w.seed)
    check_stats(tr.reduce_stats(), Oracle.from_workload(w).eval(pols, w.seed)[0], tr.histograms, f"{n} {shape} {policies}")
    tr.close()


@pytest.mark.parametrize("n", [1, 700, 20_001, 60_000])
@pytest.mark.parametrize("shape", [(1, 1), (2, 3)])
def test_grids_beside_each_other(n, shape):
    # grids of one, five and two rows, with windows and without, and between them one whose overheads differ by budget (which runs
    # by itself)
    w = synth.tiny_workload(163 + n, n, n_servers=shape[0], n_devices=shape[1], max_prompt=500, max_out=60, device_dearer=True)
    of = lambda rate, rows: [synth.policy(b, r_c=rate, flags=PACED, mig_threshold=1e-6 * k) for b in (0.02, 0.2, 0.7) for k in range(rows)]
    full_parity(w, of(5.0, 1) + of(6.0, 5) + of(40.0, 2), select=False, tag=f"{n} {shape}")
    by_budget = [synth.policy(b, r_c=7.0, flags=PACED, mig_threshold=1e-6 * k) for k, b in enumerate(synth.budget_grid(9))]
    full_parity(w, of(40.0, 1) + by_budget + of(6.0, 1) + of(5.0, 3), select=False, tag=f"{n} {shape} and one apart")


@pytest.mark.parametrize("n,shape,kind,where", [(2_199_999, (3, 2), "spread", "device"), (2_200_000, (3, 2), "spread", "device"), (2_200_001, (1, 1), "one", "pageable"),
                                                (2_300_017, (1, 7), "ties", "unaligned"), (2_999_999, (1, 1), "spread", "pinned"), (3_000_000, (1, 2), "dense", "pinned")])
def test_where_buckets_begin(n, shape, kind, where):
    test_large_traces_are_placed_by_way_of_buckets(n, shape, kind, where)


@pytest.mark.parametrize("shape,kind", [((1, 1), "10ms"), ((3, 2), "pairs"), ((3, 2), "narrow")])
def test_smallest_traces_by_way_of_buckets_by_a_coarse_clock(shape, kind):
    test_large_traces_by_a_coarse_clock(2_200_000, shape, kind)
