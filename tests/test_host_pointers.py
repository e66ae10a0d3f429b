"""Which memory the library's host side reads where, against a CUDA runtime that runs nothing (no GPU needed).  Each case
is a process of its own, with tests/fake_cudart.cpp in front of the real runtime."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests")
CUDA_INCLUDE = "/usr/local/cuda/include"

PRELUDE = """
import ctypes as C, mmap, os, sys
sys.path.insert(0, os.getcwd())
import numpy as np
from paper_2502_11417_b200 import api, synth
L, fake = api.lib(), C.CDLL(os.environ["LD_PRELOAD"])
fake.fake_memory.argtypes = [C.c_void_p, C.c_size_t, C.c_int, C.c_int]
fake.fake_copied.restype = fake.fake_loads.restype = C.c_uint64
fake.fake_last_ticks.restype = fake.fake_last_stats.restype = C.c_void_p
HOST, DEVICE, MANAGED = 1, 2, 3                       # cudaMemoryType

libc = C.CDLL(None)
libc.mmap.restype = C.c_void_p
libc.mmap.argtypes = [C.c_void_p, C.c_size_t, C.c_int, C.c_int, C.c_int, C.c_long]

def unreadable(count, kind, device=0):
    # addresses the host cannot read, taken for memory of that kind
    p = libc.mmap(None, 4 * count, 0, mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS, -1, 0)
    fake.fake_memory(p, 4 * count, kind, device)
    return p

def load(ctx, n, columns, arrays_on_device=0):
    sv, dv = api.server_array([synth.server()]), api.device_array([synth.device(500.0, 20.0)])
    desc = api.TraceDesc(n, *columns, C.addressof(sv), 1, C.addressof(dv), 1, arrays_on_device, 0)
    return L.disco_load_trace(C.byref(ctx), C.byref(desc), None)

def host_columns(n):
    cols = [np.full(n, 7, np.int32), np.full(n, 5, np.int32), np.full(n, 0.5, np.float32), np.zeros(n, np.uint8), np.zeros(n, np.uint8)]
    return cols, [c.ctypes.data for c in cols]

def set_tables(ctx, n, ticks):
    cnt = np.zeros((1, 4097), np.int64)
    cnt[0, 7] = n
    sizes = np.array([n], np.uint64)
    return L.disco_set_group_tables(ctx, cnt.ctypes.data, ticks, sizes.ctypes.data, None)
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    if not os.path.exists(os.path.join(CUDA_INCLUDE, "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    lib = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CUDA_INCLUDE, "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2502_11417_b200", "csrc"), "-o", lib, os.path.join(HERE, "fake_cudart.cpp")])
    return lib


def _run(fake, code):
    env = {k: v for k, v in os.environ.items() if k != "DISCO_CHECKED_BUILD"}
    r = subprocess.run([sys.executable, "-c", PRELUDE + code + "\nprint('as it should')\n"], cwd=ROOT, env=dict(env, LD_PRELOAD=fake),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "as it should" in r.stdout, (r.returncode, r.stdout[-1000:], r.stderr[-2000:])


@pytest.mark.parametrize("kind,device,in_place", [("DEVICE", 0, True), ("DEVICE", 1, False), ("MANAGED", 0, True), ("MANAGED", 1, False)])
def test_ticks_of_another_gpu_are_copied(fake, kind, device, in_place):
    # a kernel may read this GPU's memory where it is; memory of another one may not be mapped here
    _run(fake, f"""
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
ticks = unreadable(9000, {kind}, {device})
loads = fake.fake_loads()
assert set_tables(ctx, 9000, ticks) == 0, L.disco_last_error()
assert fake.fake_loads() == loads + 1
assert (fake.fake_last_ticks() == ticks) == {in_place}
assert fake.fake_copied() == {0 if in_place else 4 * 9000}
""")


@pytest.mark.parametrize("column", range(5))
@pytest.mark.parametrize("others", ["pageable", "pinned"])
@pytest.mark.parametrize("device", [0, 1])
def test_device_memory_given_as_host_memory_is_refused(fake, column, others, device):
    # (ordinary host arrays are packed by the CPU, which must not touch device memory), whichever column it is
    _run(fake, f"""
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
if "{others}" == "pinned":
    for c in keep:
        fake.fake_memory(c.ctypes.data, c.nbytes, HOST, 0)
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
cols[{column}] = unreadable(5000, DEVICE, {device})
assert load(ctx, 5000, cols) == -1 and b"device memory" in L.disco_last_error()
assert load(ctx, 0, cols) == 0, L.disco_last_error()         # (of an empty trace nothing is read)
""")


@pytest.mark.parametrize("over", [-1, 0, 1, 2**20 - 1])
def test_more_ticks_than_the_kernels_can_count_are_refused(fake, over):
    # the kernels' 32-bit loops step by up to 2^20 ticks
    _run(fake, f"""
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
loads, total = fake.fake_loads(), 2**32 - 2**20 + {over}
rc = set_tables(ctx, total, unreadable(total, DEVICE))
assert (rc, fake.fake_loads() - loads) == {(0, 1) if over <= 0 else (-1, 0)}, (rc, L.disco_last_error())
""")


def test_host_memory_that_runs_out_is_an_error_code(fake):
    # nothing throws across the C boundary: 2^19 policies with 16 MB of address space left, then as much as there was
    _run(fake, """
import resource
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
pols = api.policy_array([synth.policy(0.5)] * (1 << 19))
before = resource.getrlimit(resource.RLIMIT_AS)
now = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (now + (16 << 20), before[1]))
rc = L.disco_eval_policies(ctx, pols, len(pols), 1, None, None)
resource.setrlimit(resource.RLIMIT_AS, before)
assert rc == -2 and b"memory" in L.disco_last_error(), (rc, L.disco_last_error())
assert L.disco_eval_policies(ctx, pols, 2, 1, None, None) == 0, L.disco_last_error()
""")


@pytest.mark.parametrize("lengths", ["pageable", "pinned", "managed"])
def test_host_arrays_that_the_stream_still_writes(fake, lengths):
    # what the CPU packs is read in the stream's order, as a copy would: page-locked columns (among pageable ones) may be the
    # target of a copy under way, managed ones of a kernel
    _run(fake, f"""
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
kind = dict(pageable=None, pinned=HOST, managed=MANAGED)["{lengths}"]
if kind:
    fake.fake_memory(C.c_void_p(cols[0]), C.c_size_t(keep[0].nbytes), kind, 0)
new = np.full(5000, 9, np.int32)
fake.fake_pending(C.c_void_p(cols[0]), C.c_void_p(new.ctypes.data), C.c_size_t(new.nbytes))
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
assert fake.fake_first_packed() == 9 | 5 << 16
""")


@pytest.mark.parametrize("offset", [0, 1, 2, 4, 12])
def test_ticks_off_their_alignment_are_copied(fake, offset):
    _run(fake, f"""
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
ticks = unreadable(9004, DEVICE) + {offset}
assert set_tables(ctx, 9000, ticks) == 0, L.disco_last_error()
assert (fake.fake_last_ticks() == ticks) == {offset % 4 == 0}
assert fake.fake_copied() == {0 if offset % 4 == 0 else 4 * 9000}
""")


@pytest.mark.parametrize("offset", [0, 4, 8, 3])
def test_statistics_off_their_alignment_are_copied(fake, offset):
    # from 64 policies on the kernel writes 8-byte words straight into a page-locked array
    _run(fake, f"""
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
pols = api.policy_array([synth.policy(k / 63) for k in range(64)])
assert L.disco_eval_policies(ctx, pols, 64, 1, None, None) == 0, L.disco_last_error()
room = np.zeros(64 * C.sizeof(api.PolicyStats) + 64, np.uint8)
stats = (room.ctypes.data + 15) // 16 * 16 + {offset}
fake.fake_memory(room.ctypes.data, room.nbytes, HOST, 0)
assert L.disco_reduce_stats(ctx, C.c_void_p(stats), None) == 0, L.disco_last_error()
assert (fake.fake_last_stats() == stats) == {offset % 8 == 0}
""")


@pytest.mark.parametrize("sms", [1, 16, 31, 32, 148])
def test_allocation_free_sort_whatever_the_multiprocessors(fake, sms):
    # the kernel whose threads keep their values takes 8,192 a multiprocessor; the other one takes the rest, and clears what it
    # needs alone
    _run(fake, f"""
fake.fake_multiprocessors({sms})
x, out = np.full(262144, 0.5, np.float32), np.zeros(262144, np.int32)
fits = 8192 * {sms}
clear = False
for n in (5000, 1, 5000, fits, fits + 1, 5000, 262144, 262144, 5000, 5000):
    n = min(n, 262144)
    loads = fake.fake_loads()
    rc = L.disco_sort_ttft_ticks_noalloc(C.c_void_p(x.ctypes.data), n, C.c_void_p(out.ctypes.data), None)
    assert rc == 0, (n, L.disco_last_error())
    assert fake.fake_loads() == loads + 1 and 1 <= fake.fake_last_blocks() <= {sms}
    if n <= fits:
        assert bool(fake.fake_last_zeroed()) == clear, n
    clear = n <= fits
""")


def test_a_load_behind_one_that_found_no_memory(fake):
    # a context remembers which of its words the last load has cleared for the next one: not when their memory was given back in
    # between, though the next buffer may lie in the same place
    _run(fake, """
fake.fake_device_left.argtypes = [C.c_uint64]
ctx = C.c_void_p(None)
keep, cols = host_columns(50000)
for known in (0, 1, 1):
    assert load(ctx, 50000, cols) == 0 and fake.fake_last_zeroed() == known, L.disco_last_error()
more, many = host_columns(100000)
fake.fake_device_left(1 << 20)
assert load(ctx, 100000, many) == -2 and b"device allocation" in L.disco_last_error()
assert load(ctx, 50000, cols) == 0 and fake.fake_last_zeroed() == 0, L.disco_last_error()
assert load(ctx, 50000, cols) == 0 and fake.fake_last_zeroed() == 1, L.disco_last_error()
""")


def test_evaluations_in_a_row_wait_for_their_own_stream_alone(fake):
    # the tables of 2,048 policies lie in page-locked memory until a kernel has read them; other streams may be busy for long
    _run(fake, """
fake.fake_device_waits.restype = C.c_uint64
ctx = C.c_void_p(None)
keep, cols = host_columns(5000)
assert load(ctx, 5000, cols) == 0, L.disco_last_error()
pols = api.policy_array([synth.policy(k / 2047) for k in range(2048)])
for turn in range(4):
    assert L.disco_eval_policies(ctx, pols, 2048, 1, None, None) == 0, L.disco_last_error()
    assert fake.fake_device_waits() == 0
""")


def test_a_large_load_without_room_for_its_buckets(fake):
    # 4 M requests: 28 bytes each and 16 more for the buckets, which k_load does without
    _run(fake, """
fake.fake_device_left.argtypes = [C.c_uint64]
L.disco_kernel_launch_count.restype = C.c_uint64
ctx = C.c_void_p(None)
n = 4_000_000
cols = [unreadable(n, DEVICE) for _ in range(5)]
fake.fake_device_left(n * 36)
for again in range(2):
    launches = L.disco_kernel_launch_count()
    assert load(ctx, n, cols, 1) == 0, L.disco_last_error()
    assert L.disco_kernel_launch_count() == launches + 1
fake.fake_device_left(n * 20)
c2 = C.c_void_p(None)
assert load(c2, n, cols, 1) == -2 and b"device allocation" in L.disco_last_error()
""")


@pytest.mark.parametrize("room", [9 << 20, 8_001_300, 6 << 20, 3 << 20])
def test_paces_without_room_for_all_records(fake, room):
    # five paces are played out into records of their own, of 1.6 MB here; with less room (or what follows without any) in
    # smaller waves
    _run(fake, f"""
fake.fake_device_left.argtypes = [C.c_uint64]
ctx = C.c_void_p(None)
keep, cols = host_columns(200000)
assert load(ctx, 200000, cols) == 0, L.disco_last_error()
pols = api.policy_array([synth.policy(0.5, r_c=r) for r in (2.0, 3.0, 4.0, 5.0, 6.0)])
fake.fake_device_left({room})
for again in range(2):
    assert L.disco_eval_policies(ctx, pols, 5, 1, None, None) == 0, L.disco_last_error()
""")


def test_allocation_free_sort_after_a_device_reset(fake):
    # a reset moves the library's array and takes the page away where the kernel reports
    _run(fake, """
x, out = np.full(9000, 0.5, np.float32), np.zeros(9000, np.int32)
for reset in (False, False, True, False, True):
    if reset:
        fake.fake_reset_device()
    rc = L.disco_sort_ttft_ticks_noalloc(C.c_void_p(x.ctypes.data), 9000, C.c_void_p(out.ctypes.data), None)
    assert rc == 0, L.disco_last_error()
    assert fake.fake_last_words_in_place() and fake.fake_last_report_locked()
""")


@pytest.mark.parametrize("n,policies,runs,joined", [
    (10_000, "grid(2)", 0, 1), (18_000, "grid(2)", 1, 0), (60_000, "grid(2)", 1, 0),     # budgets of 0 and 1 part no requests
    (24_000, "grid(2) * 4", 1, 0), (24_000, "grid(8)", 0, 1), (24_000, "grid(4)", 0, 1), (25_000, "grid(4)", 1, 0),
    (60_000, "grid(1)", 0, 1), (90_000, "grid(1)", 1, 0),             # one: a run a request
    (150_000, "grid(256, 4)", 0, 1), (500_000, "grid(256, 4)", 1, 0),
    # a wide grid and narrow ones beside it: each its own way, in the same launch where the ways are the same
    (150_000, "grid(256, 4) + grid(2, 4, 7) + grid(2, 4, 8)", 1, 1), (150_000, "grid(2, 4, 7) + grid(256, 4) + grid(2, 4, 8)", 1, 1),
    (10_000, "grid(2, 4, 7) + grid(256, 4) + grid(2, 4, 8)", 0, 1), (500_000, "grid(2, 4, 7) + grid(256, 4) + grid(2, 4, 8)", 1, 0)])
def test_grids_go_run_by_run_or_side_by_side(fake, n, policies, runs, joined):
    # k_grid<rows, windows, way>: ways 0 and 1 run by run, 2 side by side
    _run(fake, f"""
fake.fake_launched.restype = C.c_uint64
ctx = C.c_void_p(None)
keep, cols = host_columns({n})
assert load(ctx, {n}, cols) == 0, L.disco_last_error()
def grid(K, T=1, E=0):
    return [synth.policy(b, mig_threshold=1e-6 * k, expected_len=E) for k in range(T) for b in synth.budget_grid(K)]
pols = api.policy_array({policies})
assert L.disco_eval_policies(ctx, pols, len(pols), 1, None, None) == 0, L.disco_last_error()
rows = min(4, max(p.mig_threshold for p in pols) * 1e6 + 1)
ways = [fake.fake_launched(b"k_gridILi%dELb0ELi%dE" % (rows, way)) for way in range(3)]
assert (ways[0] + ways[1], ways[2]) == ({runs}, {joined}), ways
""")
