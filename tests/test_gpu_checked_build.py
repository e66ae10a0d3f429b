"""The checked build (-DDISCO_DEBUG): the same kernels with every derived index tested against its bound before the
access.  The tiny and edge-case parity cases must run through it with no index refused and still match the oracle;
and the checks must be live (needs a GPU).  Each part runs in a process of its own, because a process loads either
the ordinary or the checked library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CASES = ("test_config0_full or test_config1_shape or test_config3_shape or test_config4_shape or test_config5_shape "
         "or test_edge_cases or test_empty_trace or test_flag_and_mode_matrix or test_buffer_search_paths "
         "or test_stochastic_baselines or test_linear_wait_rule or test_zone_by_zone or test_more_than_32_policy_tiles "
         "or test_mixed_timeline_classes or test_generation_slower or test_sorted_ticks_around "
         "or test_one_prompt_length or test_more_groups_than_fit or test_family_whose_first_tile")


def _run(args, **more):
    env = dict(os.environ, DISCO_CHECKED_BUILD="1", **more)
    return subprocess.run([sys.executable] + args, cwd=ROOT, env=env, capture_output=True, text=True, timeout=1500)


def test_parity_cases_pass_with_every_index_checked():
    r = _run(["-m", "pytest", "tests/test_gpu_parity.py", "tests/test_gpu_shards.py", "tests/test_zz_no_alloc.py",
              "-x", "-q", "-m", "gpu", "-k", CASES + " or shards or two_calls or limits"])
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout and "failed" not in r.stdout


def test_small_traces_run_by_run():
    # the grid kernels of large traces, which small ones do not reach: the same cases, and those made for runs, against the oracle
    r = _run(["-m", "pytest", "tests/test_gpu_parity.py", "tests/test_gpu_variants.py", "-x", "-q", "-m", "gpu", "-k",
              CASES + " or few_requests or eight_overheads or several_overheads or reduced_together or beside_the_slope or many_kinds"], DISCO_DEBUG_RUNS="1")
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout and "failed" not in r.stdout


def test_the_checks_are_live():
    code = (
        "import ctypes\n"
        "from paper_2502_11417_b200 import api, synth, Trace\n"
        "L = api.lib()\n"
        "assert api._build.LIB_CHECKED in [api._build.build(checked=True)]\n"
        "rc = L.disco_debug_selftest(None)\n"
        "msg = L.disco_last_error().decode()\n"
        "assert rc == -3 and 'checked build' in msg and 'self-test' in msg and 'index 34' in msg and 'bound 32' in msg, (rc, msg)\n"
        "assert L.disco_debug_selftest(None) == -3\n"              # the record is cleared and taken again
        "w = synth.make_workload(1, n=3000, n_budgets=5)\n"          # the context is still usable after a refusal
        "t = Trace.from_workload(w); t.eval_policies(w.policies, 1); s = t.reduce_stats()\n"
        "assert s[0].n_requests == 3000\n"
        "print('live')\n")
    r = _run(["-c", code])
    assert r.returncode == 0 and "live" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


WAITS = """
import os, sys
sys.path[:0] = [os.getcwd(), os.path.join(os.getcwd(), "tests")]
import numpy as np, torch
from paper_2502_11417_b200 import DiscoError, Trace, synth
from paper_2502_11417_b200.api import sort_ttft_ticks_noalloc
from parity import check_tables
from oracle import Oracle

def lost(call):
    try:
        call()
    except DiscoError as e:
        assert e.code == -3 and "lost each other" in str(e), str(e)
        return
    raise AssertionError("a wait ran out and nobody was told")

def load(t, w):
    return t.load_trace(w.prompt_len, w.output_len, w.server_ttft_s, w.server_profile, w.device_profile, w.servers, w.devices)

waits = os.environ["WAITS"].split()
large = synth.make_workload(4, n=40000, n_budgets=2)
small = {"once": lambda: synth.make_workload(4, n=9000, n_budgets=2),
         "groups": lambda: synth.tiny_workload(4, 9000, n_servers=4, n_devices=5, max_prompt=4096, policies=[synth.policy(0.3)])}[os.environ["TRACE"]]()
x = torch.from_numpy(large.server_ttft_s).cuda()
out = torch.full((large.n,), -7, dtype=torch.int32, device="cuda")
t, u = load(Trace(), large), load(Trace(), small)
cnt = np.stack([u.group_tables(g)[0] for g in range(u.n_groups)])
ticks = torch.cat([u.sorted_ticks_device(g) for g in range(u.n_groups)])
for wait in waits:
    os.environ["DISCO_DEBUG_ABSENT"] = wait
    lost(lambda: load(t, small))
    lost(lambda: sort_ttft_ticks_noalloc(x, out))
    assert bool((out == -7).all())
    lost(lambda: u.set_group_tables(cnt, ticks, cnt.sum(axis=1).astype(np.uint64)))
    del os.environ["DISCO_DEBUG_ABSENT"]
    for c in (t, u):
        try:
            c.eval_policies(small.policies, 1)
            raise AssertionError("evaluated a trace that was not loaded")
        except DiscoError as e:
            assert e.code == -1
        load(c, small)
        check_tables(c, Oracle.from_workload(small), "after wait " + wait)
assert (sort_ttft_ticks_noalloc(x, out).cpu().numpy() == np.sort(np.rint(large.server_ttft_s.astype(np.float64) * 1e6))).all()
print("waited")
"""


@pytest.mark.parametrize("trace", ["once", "groups"])
def test_blocks_leave_when_a_wait_runs_out(trace):
    # each of the ingestion kernels' waits in turn expects an arrival that nobody makes: the call fails, nothing has been placed or
    # sorted, and the context takes the next load.  Six groups are loaded, and their ticks imported, by k_load_once with its two
    # waits (4 is the first again, 3 the second), as are the ticks of the allocation-free sort; twenty groups by k_load (three
    # barriers, and the blocks' sums as 4).
    r = _run(["-c", WAITS], WAITS="1 2 3 4", TRACE=trace)
    assert r.returncode == 0 and "waited" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def test_large_traces_with_every_index_checked():
    # the kernels of large traces (with rows, whose requests' places are looked up, from device and page-locked memory), buckets that
    # are crowded or left to the radix sort, and a trace that k_load places in rounds
    r = _run(["-m", "pytest", "tests/test_gpu_variants.py", "-x", "-q", "-m", "gpu", "-k",
              "by_way_of_buckets and (3500000 or 3508193 or 4000003 or 16777) or coarse_clock and 4000003 and pairs"])
    assert r.returncode == 0 and " passed" in r.stdout, r.stdout[-3000:] + r.stderr[-2000:]


LATE = """
import os, sys
sys.path[:0] = [os.getcwd(), os.path.join(os.getcwd(), "tests")]
import numpy as np, torch
from paper_2502_11417_b200 import DiscoError, Trace, synth
for n, shape in ((5000, (1, 1)), (5000, (3, 2)), (40001, (1, 7)), (500009, (1, 1)), (1150000, (3, 2))):
    w = synth.tiny_workload(n, n, n_servers=shape[0], n_devices=shape[1], max_prompt=4096, max_out=60)
    w.output_len[n - 3] = 4000                      # (the longest output is the last block's)
    cols = [torch.from_numpy(getattr(w, f)).cuda() for f in ("prompt_len", "output_len", "server_ttft_s", "server_profile", "device_profile")]
    t = Trace()
    for _ in range(2):
        t.load_trace(*cols, w.servers, w.devices)
        t.eval_policies([synth.policy(0.4), synth.policy(0.0)], 1)
        for s in t.reduce_stats():
            assert s.tok_server + s.tok_device == w.output_len.sum(dtype=np.int64), (n, shape)
            assert s.n_intervals == w.output_len.sum(dtype=np.int64) - n and s.n_requests == n, (n, shape)
        try:                                        # 4,000 tokens at one a second would outlast 2^31 ticks, 60 would not
            t.eval_policies([synth.policy(0.4, r_c=1.0)], 1)
            raise AssertionError("the longest output was overlooked")
        except DiscoError as e:
            assert e.code == -1 and "outlast" in str(e)
    t.close()
print("late")
"""


def test_totals_of_a_block_that_is_late():
    # the last block of a load adds its output tokens and its longest output long behind the others
    r = _run(["-c", LATE], DISCO_DEBUG_ABSENT="5")
    assert r.returncode == 0 and "late" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


FEW = """
import numpy as np, torch
from paper_2502_11417_b200 import DiscoError
from paper_2502_11417_b200.api import sort_ttft_ticks_noalloc
rng = np.random.default_rng(3)
for n in (5000, 131072, 131073, 5000, 200001, 262144, 9000, 262143):
    for wide in (False, True):                      # (the second: left to the radix sort)
        x = (1000.0 + 100.0 * rng.random(n) if wide else np.exp(rng.normal(-0.5, 0.9, n))).astype(np.float32)
        out = torch.empty(n, dtype=torch.int32, device="cuda")
        got = sort_ttft_ticks_noalloc(torch.from_numpy(x).cuda(), out).cpu().numpy()
        assert (got == np.sort(np.rint(x.astype(np.float64) * 1e6))).all(), (n, wide)
    x[n // 2] = float("nan")
    try:
        sort_ttft_ticks_noalloc(torch.from_numpy(x).cuda(), out)
        raise AssertionError("a value out of range was taken")
    except DiscoError as e:
        assert e.code == -1
print("few")
"""


def test_allocation_free_sort_on_few_multiprocessors():
    # more than 8,192 values a multiprocessor: a kernel that reads them twice
    r = _run(["-c", FEW], DISCO_DEBUG_MULTIPROCESSORS="16")
    assert r.returncode == 0 and "few" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def test_the_ordinary_build_has_no_selftest():
    from paper_2502_11417_b200 import api
    if os.environ.get("DISCO_CHECKED_BUILD") == "1":
        pytest.skip("this process runs the checked build")
    L = api.lib()
    assert L.disco_debug_selftest(None) == -1 and b"not a checked build" in L.disco_last_error()
